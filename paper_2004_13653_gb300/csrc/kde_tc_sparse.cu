// The block-sparse split-FP16 Gaussian contraction on 128 x 128 tiles, one CTA
// per tile and piece.
//
// The factorisation and the operands are those of kde_tc2.cu (A[i,p] =
// 2^(15-u^2), B[j,p] = (w_p/w_max) 2^(15-v^2), hi/lo FP16, three products).
// A point belongs to every tile within its reach, so smaller tiles compute
// fewer cells that the point does not touch: at a reach of 31 cells and 16-cell
// bins 206^2 cells per point instead of the 334^2 of 256 x 256 tiles, for 2.6 x
// 256 operand values instead of 1.7 x 512.  What a 128 x 128 MMA costs is its
// operand reads (128 bytes per clock for one with N = 128, all that shared
// memory gives), so the two products with A's hi part run as one MMA with
// N = 256 over B's hi and lo rows, which lie next to each other:
//   columns 0-127   += Ahi Bhi^T
//   columns 128-255 += Ahi Blo^T (the same MMA), += Alo Bhi^T (N = 128)
// 20 KB instead of 24 KB of operands per K step, and the small products have an
// accumulator of their own: the tensor core truncates its FP32 sums at the
// accumulator's magnitude, so only the four large steps of a 64-point stage
// lose anything.  Chunks of two stages keep the error at that of the dense
// contraction's or below.
//
// Roles, by warpgroup (setmaxnreg divides the registers):
//   WG0    warp 0: MMA issue (one thread); warps 1-3: point loaders, stages in
//          turn (a stage is a chain of dependent reads).  48 registers.
//   WG1    epilogue: each thread owns one TMEM lane (an x cell) and keeps its
//          128 columns' running sums in registers (200 registers).
//   WG2-5  operand producers: eight warps per stage, the two halves take the
//          stages in turn; four warps per operand, each thread a quarter of
//          four rows (56 registers).
#include <cuda_fp16.h>

#include <algorithm>

#include "kde_internal.cuh"
#include "tc_ptx.cuh"

namespace kde {
namespace {

using namespace tc;

constexpr int kT = 128;      // cells of a tile's side
constexpr int kKS = 64;      // points per stage
constexpr int kStages = 3;
constexpr int kPS = 8;       // point-parameter ring depth
constexpr int kRowBytes = 2 * kKS;
constexpr int kPart = kT * kRowBytes;  // 16 KB: one operand part of a stage
constexpr int kOffA = 0, kOffB = 2 * kPart, kStageBytes = 4 * kPart;

// parameter ring slot: A coordinates, B coordinates, B exponent offsets
// (-(15 + log2(|w|/w_max)), +inf for w = 0), B sign words of point pairs
constexpr int kPrmA = 0, kPrmB = kKS, kPrmN = 2 * kKS, kPrmS = 3 * kKS;
constexpr int kPrmFloats = 3 * kKS + kKS / 2;

constexpr int kWarps = 24, kThreads = 32 * kWarps;
constexpr int kLoaders = 3;              // warps 1..3
constexpr int kFirstEpiWarp = 4, kEpiWarps = 4;
constexpr int kFirstProducerWarp = 8, kGroupWarps = 8;  // two groups
constexpr int kRowsPerThread = kT / 32;
constexpr int kRegsLaunch = 80;  // 768 threads: at most 65536 / 768 = 85, allocated in 8s
constexpr int kRegsCtl = 48, kRegsEpi = 200, kRegsProd = 56;
static_assert(128 * kRegsCtl + 128 * kRegsEpi + 512 * kRegsProd <= kThreads * kRegsLaunch,
              "the warpgroups' register budgets exceed the block's pool");

constexpr int kOffParams = kStages * kStageBytes;
constexpr int kOffBars = kOffParams + kPS * kPrmFloats * 4;
constexpr int kNumBars = 2 * kStages + 2 * kPS + 2 + 2 + 1;
constexpr int kOffMisc = kOffBars + kNumBars * 8;
constexpr int kSmemBytes = kOffMisc + 64 + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");

enum Role : int { kRoleMma = 41, kRoleLoader = 42, kRoleEpilogue = 43, kRoleProducer = 44 };

struct Item {
  const TcInst* I;
  int tm, tn, nst;
  int64_t k_begin, vend;  // positions in the tile's runs
  int64_t slot;           // the piece's partial tile
};

// The work item at schedule position pos: full pieces first (tile by tile),
// then the tiles' short last pieces, longest first (kde_sparse.cu's list).
__device__ __forceinline__ Item sparse_item(const TcInst* __restrict__ tab, int ninst,
                                            const SparseCtl& sp, int pos) {
  const int n_full = (int)__ldg(sp.full_begin + sp.tiles_total);
  int t, p;
  if (pos < n_full) {
    int lo = 0, hi = sp.tiles_total - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if ((int)__ldg(sp.full_begin + mid) <= pos) lo = mid; else hi = mid - 1;
    }
    t = lo;
    p = pos - (int)__ldg(sp.full_begin + t);
  } else {
    t = (int)__ldg(sp.tail_tile + (pos - n_full));
    p = (int)(__ldg(sp.piece_begin + t + 1) - __ldg(sp.piece_begin + t)) - 1;
  }
  int a = 0, b = ninst - 1;
  while (a < b) {
    const int mid = (a + b + 1) >> 1;
    if (tab[mid].tile_begin <= t) a = mid; else b = mid - 1;
  }
  Item r;
  r.I = tab + a;
  const int local = t - r.I->tile_begin;
  r.tm = local % r.I->tiles_m;
  r.tn = local / r.I->tiles_m;
  r.k_begin = (int64_t)p * sp.piece_len;
  r.vend = min((int64_t)__ldg(sp.tile_total + t), r.k_begin + (int64_t)sp.piece_len);
  r.nst = r.vend > r.k_begin ? (int)((r.vend - r.k_begin + kKS - 1) / kKS) : 0;
  r.slot = (int64_t)__ldg(sp.piece_begin + t) + p;
  return r;
}

__global__ void __launch_bounds__(kThreads, 1)
    k_tc_sparse(const TcInst* __restrict__ tab, int ninst, const __grid_constant__ SparseCtl sp,
                CallScalars* __restrict__ scal) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  float* params = reinterpret_cast<float*>(smem + kOffParams);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOffBars);
  uint64_t* full = bars;                 // [kStages] producers -> MMA
  uint64_t* empty = bars + kStages;      // [kStages] MMA -> producers
  uint64_t* pfull = bars + 2 * kStages;  // [kPS] loader -> producers
  uint64_t* pempty = pfull + kPS;        // [kPS] producers -> loader
  uint64_t* accfull = pempty + kPS;      // [2] MMA -> epilogue
  uint64_t* accempty = accfull + 2;      // [2] epilogue -> MMA
  uint64_t* mmadone = accempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the work list was built on the device by the preceding launches; a list
  // longer than the partial buffer is an error and no piece of it is computed,
  // nor of one whose sort timed out (its bin starts are not trusted)
  const int listed = (int)__ldg(sp.piece_begin + sp.tiles_total);
  const bool sort_failed = *reinterpret_cast<const volatile int*>(&scal->err) & kErrSortTimeout;
  const int n_items = listed > sp.max_pieces || sort_failed ? 0 : listed;
  if (listed > sp.max_pieces && blockIdx.x == 0 && threadIdx.x == 0)
    atomicOr(&scal->err, kErrBadArg);
  // dealt in snake order: forward in even rounds, backward in odd ones
  auto item_at = [&](int r) -> int {
    const int nc = gridDim.x, c = blockIdx.x;
    const int it = r * nc + ((r & 1) ? nc - 1 - c : c);
    return it < n_items ? it : -1;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], kGroupWarps);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < kPS; ++s) {
      mbar_init(&pfull[s], 32);
      mbar_init(&pempty[s], kGroupWarps);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], kEpiWarps);
    }
    mbar_init(mmadone, 1);
    *abort_flag = 0;
    mbar_init_fence();
  }
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp < kFirstEpiWarp) {
    regs_dec<kRegsCtl>();
    if (warp == 0) {
      // ------------------------------------------------------------ MMA issue
      if (lane == 0) {
        constexpr uint32_t kIdescHi = idesc_f16_f32(kT, 2 * kT), kIdescLo = idesc_f16_f32(kT, kT);
        uint32_t g = 0, mc = 0;
        bool ok = true;
        const uint32_t sbase = smem_u32(smem);
        for (int rd = 0, it = item_at(0); ok && it >= 0; it = item_at(++rd)) {
          const Item itm = sparse_item(tab, ninst, sp, it);
          const int CS = itm.I->chunk_stages;
          uint32_t acc = tmem_base;
          for (int st = 0; ok && st < itm.nst; ++st, ++g) {
            const bool fresh = st % CS == 0;
            if (fresh) {  // the epilogue has taken this accumulator's last chunk
              const uint32_t b = mc & 1u;
              if (!(ok = mbar_wait(&accempty[b], ((mc >> 1) & 1u) ^ 1u, abort_flag, scal,
                                   kRoleMma)))
                break;
              tc_fence_after();
              acc = tmem_base + b * 256u;
            }
            const uint32_t s = g % kStages;
            if (!(ok = mbar_wait(&full[s], (g / kStages) & 1, abort_flag, scal, kRoleMma))) break;
            tc_fence_after();
            const uint32_t a0 = sbase + s * kStageBytes + kOffA, b0 = sbase + s * kStageBytes + kOffB;
            const uint64_t ahi = desc_swz(a0, 2u, 1024u), alo = desc_swz(a0 + kPart, 2u, 1024u);
            const uint64_t bb = desc_swz(b0, 2u, 1024u);  // hi rows, then lo rows
#pragma unroll
            for (int k = 0; k < kKS / 16; ++k) {
              const uint64_t dk = (uint64_t)(2 * k);
              mma_f16(acc, ahi + dk, bb + dk, kIdescHi, fresh && k == 0 ? 0u : 1u);
              mma_f16(acc + 128u, alo + dk, bb + dk, kIdescLo, 1u);
            }
            mma_commit(&empty[s]);
            if (st + 1 == itm.nst || (st + 1) % CS == 0) {
              mma_commit(&accfull[mc & 1u]);
              ++mc;
            }
          }
        }
        mma_commit(mmadone);
        mbar_wait(mmadone, 0, abort_flag, scal, kRoleMma, /*honour_abort=*/false);
      }
      __syncwarp();
    } else {
      // -------------------------------------------------------- point loaders
      const uint32_t mine = (uint32_t)warp - 1u;
      uint32_t g = 0;
      bool ok = true;
      for (int rd = 0, it = item_at(0); ok && it >= 0; it = item_at(++rd)) {
        const Item itm = sparse_item(tab, ninst, sp, it);
        const TcInst& I = *itm.I;
        const float wmax = __uint_as_float(I.scal->wmax_bits);
        const float inv_wmax = wmax > 0.f ? 1.0f / wmax : 1.0f;
        const float2 cx = I.gxt[min(itm.tm * kT + kT / 2, I.nx - 1)];
        const float2 cy = I.gyt[min(itm.tn * kT + kT / 2, I.ny - 1)];
        RunCursor cur;  // items exist only for tiles whose range holds points
        cur.init(I.start, I.bin_begin, I.nbx,
                 tile_bins(I.cs, I.range_reach, I.inv_binw, I.nbx, I.nby, itm.tm, itm.tn, kT));
        for (int st = 0; ok && st < itm.nst; ++st, ++g) {
          if (g % kLoaders != mine) continue;  // another loader's stage
          float4 P[2];
          float W[2];
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const int64_t v = itm.k_begin + (int64_t)st * kKS + lane + 32 * hh;
            if (v < itm.vend) {
              const int64_t p = cur.map(v);
              P[hh] = __ldg(I.pts + p);
              W[hh] = __ldg(I.wts + p);
            } else {  // past the piece: a zero-weight point (B = 0)
              P[hh] = make_float4(0.f, 0.f, 0.f, 0.f);
              W[hh] = 0.f;
            }
          }
          const uint32_t ps = g % kPS;
          if (!(ok = mbar_wait(&pempty[ps], ((g / kPS) & 1) ^ 1, abort_flag, scal, kRoleLoader)))
            break;
          float* prm = params + ps * kPrmFloats;
          uint32_t neg[2];
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const int e = lane + 32 * hh;
            const float4 q = P[hh];
            prm[kPrmA + e] = (q.x - cx.x) + (q.y - cx.y);
            prm[kPrmB + e] = (q.z - cy.x) + (q.w - cy.y);
            const float w = W[hh];
            neg[hh] = w < 0.f ? 1u : 0u;
            prm[kPrmN + e] = w != 0.f ? -(15.0f + log2f(fabsf(w) * inv_wmax)) : INFINITY;
          }
          // sign word of points (2 lane, 2 lane + 1): bit 15 and bit 31, the
          // sign bits of their packed FP16 halves
          const int src = (2 * lane) & 31;
          const uint32_t h = lane < 16 ? 0u : 1u;
          const uint32_t s_lo = __shfl_sync(0xffffffffu, neg[0], src) |
                                (__shfl_sync(0xffffffffu, neg[1], src) << 1);
          const uint32_t s_hi = __shfl_sync(0xffffffffu, neg[0], src + 1) |
                                (__shfl_sync(0xffffffffu, neg[1], src + 1) << 1);
          reinterpret_cast<uint32_t*>(prm + kPrmS)[lane] =
              (((s_lo >> h) & 1u) << 15) | (((s_hi >> h) & 1u) << 31);
          mbar_arrive(&pfull[ps]);
        }
      }
    }
  } else if (warp < kFirstProducerWarp) {
    // --------------------------------------------------------------- epilogue
    regs_inc<kRegsEpi>();
    const int q = warp & 3;  // TMEM lane quadrant
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    uint32_t dc = 0;
    bool ok = true;
    for (int rd = 0, it = item_at(0); ok && it >= 0; it = item_at(++rd)) {
      const Item itm = sparse_item(tab, ninst, sp, it);
      const int CS = itm.I->chunk_stages;
      float run[kT];
      const int nchunks = (itm.nst + CS - 1) / CS;
      for (int ch = 0; ok && ch < nchunks; ++ch, ++dc) {
        const uint32_t b = dc & 1u;
        if (!(ok = mbar_wait(&accfull[b], (dc >> 1) & 1u, abort_flag, scal, kRoleEpilogue))) break;
        tc_fence_after();
        const uint32_t acc = tmem_base + b * 256u + lane_off;
#pragma unroll
        for (int cb = 0; cb < kT / 16; ++cb) {
          uint32_t hi[16], lo[16];
          tmem_ld_async(acc + cb * 16, hi);
          tmem_ld_async(acc + 128u + cb * 16, lo);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 16; c += 2) {
            float x = __uint_as_float(hi[c]), y = __uint_as_float(hi[c + 1]);
            add2_rn(x, y, lo[c], lo[c + 1]);
            if (ch == 0) {
              run[cb * 16 + c] = x;
              run[cb * 16 + c + 1] = y;
            } else {
              add2_rn(run[cb * 16 + c], run[cb * 16 + c + 1], __float_as_uint(x),
                      __float_as_uint(y));
            }
          }
        }
        // the accumulator is read: the MMAs of chunk dc + 2 may overwrite it
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&accempty[b]);
      }
      if (!ok) break;
      // the piece's own 128 x 128 partial, [j_local][i_local]
      const float wmax = __uint_as_float(itm.I->scal->wmax_bits);
      const float scale = itm.I->base_scale * (wmax > 0.f ? wmax : 1.0f);
      float* piece = sp.part + itm.slot * (kT * kT) + q * 32 + lane;
      if (itm.nst == 0) {
        for (int c = 0; c < kT; ++c) piece[c * kT] = 0.f;
      } else {
#pragma unroll
        for (int c = 0; c < kT; ++c) piece[c * kT] = run[c] * scale;
      }
    }
  } else {
    // -------------------------------------------------------------- producers
    // Lane l of warp k of an operand's four writes rows l, l + 32, l + 64,
    // l + 96 in chunks 2k and 2k + 1, so that one broadcast load of a chunk's
    // point parameters serves four rows.
    regs_dec<kRegsProd>();
    const int pw = (warp - kFirstProducerWarp) & (kGroupWarps - 1);
    const uint32_t group = (uint32_t)(warp - kFirstProducerWarp) / kGroupWarps;
    const bool isA = pw < kGroupWarps / 2;  // warp-uniform
    const int c0 = 2 * (pw & 3);
    uint32_t g = 0;
    bool ok = true;
    for (int rd = 0, it = item_at(0); ok && it >= 0; it = item_at(++rd)) {
      const Item itm = sparse_item(tab, ninst, sp, it);
      const TcInst& I = *itm.I;
      const bool signs = !isA && I.scal->negw != 0;
      float ngv[kRowsPerThread];  // minus the rows' cell coordinates
      {
        const int base = (isA ? itm.tm : itm.tn) * kT;
        const float2* tab_g = isA ? I.gxt : I.gyt;
        const int n_g = isA ? I.nx : I.ny;
        const float2 c = tab_g[min(base + kT / 2, n_g - 1)];
#pragma unroll
        for (int k = 0; k < kRowsPerThread; ++k) {
          const float2 v = tab_g[min(base + k * 32 + lane, n_g - 1)];
          ngv[k] = -((v.x - c.x) + (v.y - c.y));
        }
      }
      const int nst = itm.nst;
      for (int st = 0; ok && st < nst; ++st, ++g) {
        if ((g & 1u) != group) continue;  // the other group's stage
        const uint32_t s = g % kStages, ps = g % kPS;
        if (!(ok = mbar_wait(&pfull[ps], (g / kPS) & 1, abort_flag, scal, kRoleProducer))) break;
        if (!(ok = mbar_wait(&empty[s], ((g / kStages) & 1) ^ 1, abort_flag, scal, kRoleProducer)))
          break;
        unsigned char* row0 = smem + s * kStageBytes + (isA ? kOffA : kOffB) + lane * kRowBytes;
        const float* prm = params + ps * kPrmFloats;
        const float4* crd = reinterpret_cast<const float4*>(prm + (isA ? kPrmA : kPrmB));
        const float4* nce = reinterpret_cast<const float4*>(prm + kPrmN);
        const uint4* sgn = reinterpret_cast<const uint4*>(prm + kPrmS);
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          const int c = c0 + cc;
          const float4 p0 = crd[2 * c], p1 = crd[2 * c + 1];
          float4 n0 = make_float4(-15.f, -15.f, -15.f, -15.f), n1 = n0;
          if (!isA) {
            n0 = nce[2 * c];
            n1 = nce[2 * c + 1];
          }
          uint4 sg = make_uint4(0u, 0u, 0u, 0u);
          if (signs) sg = sgn[c];
          const float2 P2[4] = {make_float2(p0.x, p0.y), make_float2(p0.z, p0.w),
                                make_float2(p1.x, p1.y), make_float2(p1.z, p1.w)};
          const float2 N2[4] = {make_float2(n0.x, n0.y), make_float2(n0.z, n0.w),
                                make_float2(n1.x, n1.y), make_float2(n1.z, n1.w)};
          // rows lane + 32 k share the swizzle phase lane & 7
          const int off = (c ^ (lane & 7)) << 4;
#pragma unroll
          for (int k = 0; k < kRowsPerThread; ++k) {
            const float2 ng2 = make_float2(ngv[k], ngv[k]);
            uint32_t hw[4], lw[4];
#pragma unroll
            for (int e2 = 0; e2 < 4; ++e2) {
              const float2 u = add2(P2[e2], ng2);   // point - cell, in units of h sqrt(2 ln 2)
              const float2 y = fma2(u, u, N2[e2]);  // u^2 - exponent offset
              const float v0 = ex2_neg(y.x), v1 = ex2_neg(y.y);
              // hi = v rounded to FP16, lo = v - hi (one instruction each; masking hi
              // out of v and subtracting it took three for two: 5.31 ms, now 5.21 for
              // 20M points x 4096^2)
              const __half2 hh = __floats2half2_rn(v0, v1);
              const __half2 ll = __floats2half2_rn(minus_half(v0, __low2half(hh)),
                                                   minus_half(v1, __high2half(hh)));
              hw[e2] = *reinterpret_cast<const uint32_t*>(&hh);
              lw[e2] = *reinterpret_cast<const uint32_t*>(&ll);
            }
            if (signs) {  // negative weights: flip the FP16 sign bits of those points
              hw[0] ^= sg.x; hw[1] ^= sg.y; hw[2] ^= sg.z; hw[3] ^= sg.w;
              lw[0] ^= sg.x; lw[1] ^= sg.y; lw[2] ^= sg.z; lw[3] ^= sg.w;
            }
            unsigned char* row = row0 + k * 32 * kRowBytes;
            *reinterpret_cast<uint4*>(row + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
            *reinterpret_cast<uint4*>(row + kPart + off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
          }
        }
        // order this warp's stores before the tensor core's reads of them
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&full[s]);
          mbar_arrive(&pempty[ps]);
        }
      }
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

cudaError_t launch_tc_sparse(const TcPlan& plan, const TcInst* tab, int ninst, const SparseCtl& sp,
                             CallScalars* err, cudaStream_t s) {
  if (ninst < 1 || !plan.split16 || sp.side != kT || sp.tiles_total < 1 || sp.piece_len < kKS ||
      sp.piece_len % kKS)
    return cudaErrorInvalidValue;
  // setmaxnreg draws on the registers the block was launched with: refuse a
  // build whose launch register count would not hold the warpgroups' budgets
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, k_tc_sparse);
  if (e != cudaSuccess) return e;
  if ((fa.numRegs + 7) / 8 * 8 < kRegsLaunch) return cudaErrorInvalidConfiguration;
  e = cudaFuncSetAttribute(k_tc_sparse, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e != cudaSuccess) return e;
  k_tc_sparse<<<std::max(1, plan.ctas), kThreads, kSmemBytes, s>>>(tab, ninst, sp, err);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace kde
