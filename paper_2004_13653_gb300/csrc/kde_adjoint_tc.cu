// Adjoint of the Gaussian density as two tcgen05 contractions (Eq. 7 with
// the Gaussian row of Table 1), the form for wide bandwidths.
//
// With A_ip = 2^(-u_ip^2), B_jp = 2^(-v_jp^2) (u, v: offsets of cell and
// point in units of h sqrt(2 ln 2)) and a cotangent G = dL/dF,
//   U_ip = sum_j G_ij B_jp   (contraction 1, over the y cells)
//   V_jp = sum_i G_ij A_ip   (contraction 2, over the x cells)
//   dL/dw_p = c sum_i A_ip U_ip
//   dL/dx_p = c w_p sqrt(2 ln 2)/h sum_i u_ip A_ip U_ip
//   dL/dy_p = c w_p sqrt(2 ln 2)/h sum_j v_jp B_jp V_jp
//   h-term  = c w_p (2 ln 2)/h [sum_i u^2 A U + sum_j v^2 B V]
// (c = 1/(2 pi N h^2)).  Each contraction is D[p, n] = sum_k E[p, k] T[n, k]
// with M = 128 points per tile (TMEM lanes), N = 256 cells of the
// accumulated axis per accumulator (TMEM columns) and K = the other axis, 64
// cells per stage:
//   - E (the generated operand, rows = points): 2^(15 - (g_k - y_p)^2) for
//     contraction 1 (2^(15 - (g_k - x_p)^2) for 2), made by producer warps
//     in shared memory as FP16 hi/lo, as the forward makes its operands;
//   - T (rows = cells of the accumulated axis): the cotangent, scaled by a
//     power of two so its largest entry is near 2^14, split into FP16 hi/lo
//     and laid out beforehand in global memory exactly as a stage wants it in
//     shared memory (128-byte swizzled K-major rows), so two bulk copies (async
//     proxy, completing on an mbarrier) move each stage's rows, hi and lo;
//   - three FP16 MMAs per K step (hi*hi, hi*lo, lo*hi), FP32 accumulation in
//     TMEM; two accumulators alternate between consecutive N tiles, so the
//     MMAs never wait for the epilogue;
//   - the epilogue regenerates the factor of the accumulated axis for each of
//     its cells and folds U (or V) into three per-point sums, so neither U
//     nor V ever leaves the SM.
// The points come in bin order (kde_cutoff.cu's sort), so the 128 points of a
// tile lie close together, and a tile takes only the cells within +-8
// bandwidths of some point of it: columns i0..i1 of the accumulated axis, cut
// into equal accumulators of at most 256, and the 16-cell steps of the
// contracted axis that hold j0..j1.  Beyond 7.6 bandwidths E is exactly zero in
// FP16; the accumulated axis' factor there is below 2^-46.  Without room for
// the sort the points stay in the caller's order and every tile takes the
// whole grid.  500,000 points x 1024^2, h = 16.4 cells: 3.09 ms for the two
// contractions over the whole grid, 0.57 now.
#include <cuda_fp16.h>

#include <algorithm>

#include "kde_internal.cuh"
#include "kernel_factors.cuh"
#include "tc_ptx.cuh"

namespace kde {
namespace {

using namespace tc;

constexpr int kM = 128;       // points per tile (TMEM lanes)
constexpr int kN = 256;       // cells of the accumulated axis per accumulator
constexpr int kK = 64;        // cells of the contracted axis per stage
constexpr int kStages = 2;
constexpr int kRowBytes = 2 * kK;                         // 64 FP16 per operand row
constexpr int kEBytes = kM * kRowBytes;                   // 16 KB per part
constexpr int kTBytes = kN * kRowBytes;                   // 32 KB per part
constexpr int kStageBytes = 2 * (kEBytes + kTBytes);      // hi and lo: 96 KB
constexpr int kWarps = 14;    // 0 MMA, 1 bulk loader, 2-9 epilogue, 10-13 producers
constexpr int kThreads = 32 * kWarps;
constexpr int kFirstEpiWarp = 2, kEpiWarps = 8, kFirstProducerWarp = 10;
constexpr int kOffBars = kStages * kStageBytes;
constexpr int kNumBars = 3 * kStages + 4 + 1;
constexpr int kOffComb = kOffBars + kNumBars * 8;         // [4][32][3] float2
constexpr int kOffMisc = kOffComb + 4 * 32 * 3 * 8;
constexpr int kSmemBytes = kOffMisc + 64 + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
constexpr int kBarEpi = 1;    // named barrier of the epilogue warps

enum Role : int { kRoleMma = 21, kRoleLoader = 22, kRoleEpilogue = 23, kRoleProducer = 24 };

struct AdjTcArgs {
  const float4* pts;        // prepared points (Gaussian units), n_pad entries
  const float* wts;
  const uint32_t* vals;     // the caller's index of each, null: its own
  const CallScalars* sort_err;  // with vals: where the sort records a timeout
  const int4* ranges;       // each tile's cells i0, i1, j0, j1 (empty: i0 > i1); null: all
  int64_t n;
  const unsigned char* tiles;  // [n_stages][part][rows][128 B]
  const float2* acc_tab;    // cell centres of the accumulated axis (hi, lo)
  const float2* k_tab;      // cell centres of the contracted axis
  int acc_cells, k_cells, rows;  // rows: acc_cells rounded up to 256
  float inv_cs;
  float cs;                 // cell side in prepared units
  int axis;                 // 0: x accumulated (dL/dw, dL/dx, h), 1: y (dL/dy, h)
  const CallScalars* gscal; // wmax_bits: max |G|
  double c;                 // 1/(2 pi N h^2)
  double k_xy, k_h;         // sqrt(2 ln 2)/h and 2 ln 2/h
  float* grad_xy;
  float* grad_w;
  double* hterm;
  double* lterm;
};

// The power of two the cotangent is scaled by before the FP16 split.
__host__ __device__ inline int g_exponent(unsigned gmax_bits) {
  if (gmax_bits == 0u || gmax_bits >= 0x7f800000u) return 0;
  const int e = (int)((gmax_bits >> 23) & 0xff) - 127;  // floor(log2 max|G|)
  return max(-100, min(100, 13 - e));
}

// max |G| into gscal->wmax_bits (non-negative floats order as unsigned ints).
__global__ void k_abs_max(const float* __restrict__ G, int64_t cells, CallScalars* gscal) {
  unsigned m = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < cells; q += stride) {
    const float v = fabsf(G[q]);
    if (v == v) m = max(m, __float_as_uint(v));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned*)&gscal->wmax_bits)
    atomicMax(&gscal->wmax_bits, m);
}

// The cotangent as the contraction's T operand: stage ks holds rows n
// (accumulated axis, padded to `rows`) and columns k = ks kK + e (contracted
// axis) of G scaled by 2^s, hi (11 significant bits, exact in FP16) and lo =
// the rest, each part `rows` rows of 128 bytes with the 16-byte chunks of row r
// at chunk ^ (r & 7) (the tensor core's 128-byte swizzle), so that any eight
// rows from a multiple of eight on are as shared memory wants them.  Cells
// outside the grid are zero.  One thread per (stage, row, chunk).
__global__ void k_tile_cotangent(const float* __restrict__ G, int nx, int ny, int axis,
                                 int rows, int n_stages, const CallScalars* __restrict__ gscal,
                                 unsigned char* __restrict__ tiles) {
  const int64_t total = (int64_t)rows * n_stages * 8;
  const float scale = ldexpf(1.0f, g_exponent(gscal->wmax_bits));
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += stride) {
    const int chunk = (int)(q & 7);
    const int row = (int)((q >> 3) % rows);
    const int ks = (int)((q >> 3) / rows);
    uint32_t hw[4], lw[4];
#pragma unroll
    for (int e2 = 0; e2 < 4; ++e2) {
      float v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int col = ks * kK + chunk * 8 + 2 * e2 + h;
        // axis 0: rows are x cells i, columns y cells j; axis 1 the reverse
        const int i = axis == 0 ? row : col, j = axis == 0 ? col : row;
        v[h] = (i < nx && j < ny) ? G[(int64_t)j * nx + i] * scale : 0.0f;
      }
      const float h0 = __uint_as_float(__float_as_uint(v[0]) & 0xFFFFE000u);
      const float h1 = __uint_as_float(__float_as_uint(v[1]) & 0xFFFFE000u);
      const __half2 hh = __floats2half2_rn(h0, h1);
      const __half2 ll = __floats2half2_rn(v[0] - h0, v[1] - h1);
      hw[e2] = *reinterpret_cast<const uint32_t*>(&hh);
      lw[e2] = *reinterpret_cast<const uint32_t*>(&ll);
    }
    const int64_t part = (int64_t)rows * kRowBytes;
    unsigned char* base =
        tiles + ks * 2 * part + (int64_t)row * kRowBytes + ((chunk ^ (row & 7)) << 4);
    *reinterpret_cast<uint4*>(base) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    *reinterpret_cast<uint4*>(base + part) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
  }
}

// One warp per tile of 128 points: the cells within `reach` of its points, those
// of them that can reach the grid at all (the others' sums are zero whatever
// the cells).
__global__ void k_adj_ranges(const float4* __restrict__ pts, int64_t n, int items, float cs,
                             float reach, int nx, int ny, int4* __restrict__ ranges) {
  const int it = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (it >= items) return;
  float x0 = INFINITY, x1 = -INFINITY, y0 = INFINITY, y1 = -INFINITY;
  const float ex = nx * cs + reach, ey = ny * cs + reach;
  for (int u = 0; u < kM / 32; ++u) {
    const int64_t p = (int64_t)it * kM + u * 32 + lane;
    if (p >= n) continue;
    const float4 P = pts[p];
    const float x = P.x + P.y, y = P.z + P.w;
    if (x >= -reach && y >= -reach && x <= ex && y <= ey) {
      x0 = fminf(x0, x);
      x1 = fmaxf(x1, x);
      y0 = fminf(y0, y);
      y1 = fmaxf(y1, y);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
    x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
    y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
    y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
  }
  if (lane) return;
  int4 r = make_int4(0, -1, 0, -1);
  if (x0 <= x1) {
    // cells to spare on either side for the FP32 rounding (four units of 2^-24
    // of the grid's extent)
    const float inv = 1.0f / cs;
    const int sx = 1 + (nx >> 21), sy = 1 + (ny >> 21);
    r.x = max(0, (int)floorf((x0 - reach) * inv) - sx);
    r.y = (int)fminf((float)nx, floorf((x1 + reach) * inv) + sx);
    r.z = max(0, (int)floorf((y0 - reach) * inv) - sy);
    r.w = (int)fminf((float)ny, floorf((y1 + reach) * inv) + sy);
    r.y = min(nx - 1, r.y);
    r.w = min(ny - 1, r.w);
    if (r.x > r.y || r.z > r.w) r = make_int4(0, -1, 0, -1);
  }
  ranges[it] = r;
}

// The cell of the axis nearest the point at ph + pl (prepared units).
__device__ __forceinline__ int near_cell(float ph, float pl, float inv_cs, int cells) {
  const float c = floorf((ph + pl) * inv_cs);
  return (int)fminf(fmaxf(c, 0.f), (float)(cells - 1));
}

// What a tile contracts: n_tiles accumulators of `width` cells (a multiple of
// 32, at most kN) from cell `first` (a multiple of 8) on, and the stages
// ks0..ks1 of the contracted axis, of which the 16-cell steps k16_0..k16_1
// count.  Every role derives the same from the tile's range.
struct TileWork {
  int first, width, n_tiles, ks0, ks1, k16_0, k16_1;
};
__device__ __forceinline__ TileWork tile_work(const AdjTcArgs& a, int it) {
  int4 r = a.ranges ? __ldg(a.ranges + it)
                    : (a.axis == 0 ? make_int4(0, a.acc_cells - 1, 0, a.k_cells - 1)
                                   : make_int4(0, a.k_cells - 1, 0, a.acc_cells - 1));
  if (a.axis) r = make_int4(r.z, r.w, r.x, r.y);
  TileWork w = {};
  if (r.x > r.y || r.z > r.w) return w;  // nothing in reach: n_tiles = 0
  w.first = r.x & ~7;
  const int cells = r.y - w.first + 1;
  w.n_tiles = (cells + kN - 1) / kN;
  w.width = ((cells + w.n_tiles - 1) / w.n_tiles + 31) & ~31;
  // the last accumulator's rows end inside the padded rows
  w.first = max(0, min(w.first, a.rows - w.n_tiles * w.width));
  w.ks0 = r.z / kK;
  w.ks1 = r.w / kK;
  w.k16_0 = r.z / 16;
  w.k16_1 = r.w / 16;
  return w;
}

// One persistent CTA per SM; work item = a tile of 128 points, which the CTA
// takes through every accumulator of its range and, for each, every stage of
// the contracted axis.  Roles: warp 0 issues the MMAs (one thread), warp 1 the
// stage bulk copies, warps 2-9 drain the accumulators into per-point sums (two
// warps per TMEM lane quadrant, half of the columns each), warps 10-13 generate
// the points' operand rows.
__global__ void __launch_bounds__(kThreads, 1)
    k_adjoint_tc(const __grid_constant__ AdjTcArgs a, CallScalars* __restrict__ scal) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOffBars);
  uint64_t* full_e = bars;                // [kStages] producers -> MMA
  uint64_t* full_t = bars + kStages;      // [kStages] bulk copy -> MMA (transaction bytes)
  uint64_t* empty = bars + 2 * kStages;   // [kStages] MMA -> producers and loader
  uint64_t* accfull = bars + 3 * kStages; // [2] MMA -> epilogue
  uint64_t* accempty = accfull + 2;       // [2] epilogue -> MMA
  uint64_t* mmadone = accempty + 2;
  float2* comb = reinterpret_cast<float2*>(smem + kOffComb);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_items = (int)((a.n + kM - 1) / kM);
  // after a timed-out sort the indices are not trusted: compute nothing (the
  // call reports the timeout); every thread reads the same value
  if (a.vals && (*reinterpret_cast<const volatile int*>(&a.sort_err->err) & kErrSortTimeout)) return;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full_e[s], 4);
      mbar_init(&full_t[s], 1);
      mbar_init(&empty[s], 1);
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

  if (warp == 0) {
    // -------------------------------------------------------------- MMA issue
    if (lane == 0) {
      uint32_t g = 0, mc = 0;
      bool ok = true;
      const uint32_t sbase = smem_u32(smem);
      for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
        const TileWork w = tile_work(a, it);
        const uint32_t idesc = idesc_f16_f32(kM, w.width);
        for (int nt = 0; ok && nt < w.n_tiles; ++nt, ++mc) {
          const uint32_t b = mc & 1u;
          if (!(ok = mbar_wait(&accempty[b], ((mc >> 1) & 1u) ^ 1u, abort_flag, scal, kRoleMma)))
            break;
          tc_fence_after();
          const uint32_t acc = tmem_base + b * 256u;
          for (int ks = w.ks0; ks <= w.ks1; ++ks, ++g) {
            const uint32_t s = g % kStages, ph = (g / kStages) & 1u;
            if (!(ok = mbar_wait(&full_e[s], ph, abort_flag, scal, kRoleMma))) break;
            if (!(ok = mbar_wait(&full_t[s], ph, abort_flag, scal, kRoleMma))) break;
            tc_fence_after();
            const uint32_t st = sbase + s * kStageBytes;
            const uint64_t ehi = desc_swz(st, 2u, 1024u), elo = desc_swz(st + kEBytes, 2u, 1024u);
            const uint64_t thi = desc_swz(st + 2 * kEBytes, 2u, 1024u);
            const uint64_t tlo = desc_swz(st + 2 * kEBytes + kTBytes, 2u, 1024u);
            const int first = max(0, w.k16_0 - 4 * ks), last = min(3, w.k16_1 - 4 * ks);
            // the small products first: a step's truncation is relative to the
            // accumulator, which they leave nearly empty in the first stage
            for (int k = first; k <= last; ++k) {
              const uint64_t dk = (uint64_t)(2 * k);
              mma_f16(acc, ehi + dk, tlo + dk, idesc, ks == w.ks0 && k == first ? 0u : 1u);
              mma_f16(acc, elo + dk, thi + dk, idesc, 1u);
            }
            for (int k = first; k <= last; ++k) {
              const uint64_t dk = (uint64_t)(2 * k);
              mma_f16(acc, ehi + dk, thi + dk, idesc, 1u);
            }
            mma_commit(&empty[s]);
          }
          if (!ok) break;
          mma_commit(&accfull[b]);
        }
      }
      mma_commit(mmadone);
      mbar_wait(mmadone, 0, abort_flag, scal, kRoleMma, /*honour_abort=*/false);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------- stage bulk copies of T
    if (lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
        const TileWork w = tile_work(a, it);
        const int64_t part = (int64_t)a.rows * kRowBytes;
        const uint32_t bytes = (uint32_t)w.width * kRowBytes;
        for (int nt = 0; ok && nt < w.n_tiles; ++nt)
          for (int ks = w.ks0; ks <= w.ks1; ++ks, ++g) {
            const uint32_t s = g % kStages;
            if (!(ok = mbar_wait(&empty[s], ((g / kStages) & 1u) ^ 1u, abort_flag, scal,
                                 kRoleLoader)))
              break;
            // rows first + nt width .. of stage ks, hi then lo
            const unsigned char* src =
                a.tiles + ks * 2 * part + (int64_t)(w.first + nt * w.width) * kRowBytes;
            unsigned char* dst = smem + s * kStageBytes + 2 * kEBytes;
            mbar_arrive_expect_tx(&full_t[s], 2 * bytes);
            bulk_g2s(dst, src, bytes, &full_t[s]);
            bulk_g2s(dst + kTBytes, src + part, bytes, &full_t[s]);
          }
      }
    }
    __syncwarp();
  } else if (warp < kFirstProducerWarp) {
    // --------------------------------------------------------------- epilogue
    const int q = warp & 3, colh = (warp - kFirstEpiWarp) >> 2;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    // The eight warps meet at a named barrier once per item, so none of them
    // leaves the item loop early: after a failed wait they skip the work.
    uint32_t dc = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
      const int64_t p = (int64_t)it * kM + q * 32 + lane;
      const float4 P = a.pts[p];  // n_pad is a multiple of 512: in bounds
      // the point's coordinate along the accumulated axis (hi, lo)
      const float ph = a.axis == 0 ? P.x : P.z, pl = a.axis == 0 ? P.y : P.w;
      const TileWork w = tile_work(a, it);
      // The cell the point lies in, and the point's offset r from its centre:
      // the offset of cell c is then (c - near) cs - r, exact but for one
      // rounding however far the accumulator's first cell is.
      const int near = near_cell(ph, pl, a.inv_cs, a.acc_cells);
      const float2 gn = a.acc_tab[near];
      const float r = (ph - gn.x) + (pl - gn.y);
      const int half = w.width >> 1;  // columns of this thread: a multiple of 16
      float2 s0 = make_float2(0.f, 0.f), s1 = s0, s2 = s0;  // hi + lo
      for (int nt = 0; nt < w.n_tiles; ++nt, ++dc) {
        const uint32_t b = dc & 1u;
        if (ok) ok = mbar_wait(&accfull[b], (dc >> 1) & 1u, abort_flag, scal, kRoleEpilogue);
        if (!ok) continue;
        tc_fence_after();
        float c = (float)(w.first + nt * w.width + colh * half - near);
        float t0 = 0.f, t1 = 0.f, t2 = 0.f;
        const uint32_t acc = tmem_base + b * 256u + lane_off + colh * half;
        auto fold = [&](uint32_t bits, float e) {
          const float u = fmaf(c + e, a.cs, -r);
          const float f = ex2_neg(u * u) * __uint_as_float(bits);
          t0 += f;
          t1 = fmaf(u, f, t1);
          t2 = fmaf(u * u, f, t2);
        };
#pragma unroll 1
        for (int cb = 0; cb < half; cb += 16, c += 16.f) {
          uint32_t d[16];
          tmem_ld_async(acc + cb, d);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) fold(d[e], (float)e);
        }
        // every column is read: release the accumulator
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&accempty[b]);
        two_sum_acc(s0, t0);
        two_sum_acc(s1, t1);
        two_sum_acc(s2, t2);
      }
      // the two column halves of each point, added in a fixed order
      if (colh == 1) {
        float2* o = comb + (q * 32 + lane) * 3;
        o[0] = s0;
        o[1] = s1;
        o[2] = s2;
      }
      named_sync(kBarEpi, 32 * kEpiWarps);
      if (ok && colh == 0 && p < a.n) {
        const float2* o = comb + (q * 32 + lane) * 3;
        auto both = [](float2 x, float2 y) {
          return ((double)x.x + (double)y.x) + (double)(x.y + y.y);
        };
        const double d0 = both(s0, o[0]), d1 = both(s1, o[1]), d2 = both(s2, o[2]);
        // D carries 2^15 (the generated operand) and 2^s (the cotangent)
        const double k = a.c * ldexp(1.0, -15 - g_exponent(a.gscal->wmax_bits));
        const double wt = a.wts[p];
        const int64_t to = a.vals ? (int64_t)a.vals[p] : p;  // the caller's index
        if (a.axis == 0) {
          const double gw = k * d0;
          if (a.grad_w) a.grad_w[to] = (float)gw;
          a.grad_xy[2 * to] = (float)(k * wt * a.k_xy * d1);
          a.hterm[p] = k * wt * a.k_h * d2;
          a.lterm[p] = wt * gw;
        } else {
          a.grad_xy[2 * to + 1] = (float)(k * wt * a.k_xy * d1);
          a.hterm[p] += k * wt * a.k_h * d2;
        }
      }
      named_sync(kBarEpi, 32 * kEpiWarps);  // comb is free for the next item
    }
    if (!ok && lane == 0) *abort_flag = 1;
  } else {
    // -------------------------------------------------- point operand rows
    const int t = threadIdx.x - kFirstProducerWarp * 32;  // row = point of the tile
    uint32_t g = 0;
    bool ok = true;
    for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
      const float4 P = a.pts[(int64_t)it * kM + t];
      // coordinate along the contracted axis (hi, lo)
      const float ph = a.axis == 0 ? P.z : P.x, pl = a.axis == 0 ? P.w : P.y;
      const TileWork w = tile_work(a, it);
      // offsets from the cell the point lies in, as in the epilogue
      const int near = near_cell(ph, pl, a.inv_cs, a.k_cells);
      const float2 gn = a.k_tab[near];
      const float r = (ph - gn.x) + (pl - gn.y);
      const int stages = w.n_tiles * (w.ks1 - w.ks0 + 1);
      int ks = w.ks0;
      for (int q = 0; ok && q < stages; ++q, ++g) {
        const uint32_t s = g % kStages;
        if (!(ok = mbar_wait(&empty[s], ((g / kStages) & 1u) ^ 1u, abort_flag, scal,
                             kRoleProducer)))
          break;
        const float k0 = (float)(ks * kK - near);  // first cell of the stage
        const int first = max(0, w.k16_0 - 4 * ks), last = min(3, w.k16_1 - 4 * ks);
        ks = ks == w.ks1 ? w.ks0 : ks + 1;
        unsigned char* row = smem + s * kStageBytes + t * kRowBytes;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          if (c < 2 * first || c > 2 * last + 1) continue;  // steps the MMAs skip
          uint32_t hw[4], lw[4];
#pragma unroll
          for (int e2 = 0; e2 < 4; ++e2) {
            const float v0 = fmaf(k0 + (float)(c * 8 + 2 * e2), a.cs, -r);
            const float v1 = fmaf(k0 + (float)(c * 8 + 2 * e2 + 1), a.cs, -r);
            const float2 y = fma2(make_float2(v0, v1), make_float2(v0, v1),
                                  make_float2(-15.f, -15.f));
            const float x0 = ex2_neg(y.x), x1 = ex2_neg(y.y);
            const __half2 hh = __floats2half2_rn(x0, x1);
            const __half2 ll = __floats2half2_rn(minus_half(x0, __low2half(hh)),
                                                 minus_half(x1, __high2half(hh)));
            hw[e2] = *reinterpret_cast<const uint32_t*>(&hh);
            lw[e2] = *reinterpret_cast<const uint32_t*>(&ll);
          }
          const int off = (c ^ (t & 7)) << 4;
          *reinterpret_cast<uint4*>(row + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
          *reinterpret_cast<uint4*>(row + kEBytes + off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full_e[s]);
      }
    }
    if (!ok && lane == 0) *abort_flag = 1;
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

int blocks_for_tc(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

}  // namespace

size_t adjoint_tc_workspace(int nx, int ny) {
  const size_t tx = (size_t)((nx + kN - 1) / kN) * ((ny + kK - 1) / kK);  // contraction 1
  const size_t ty = (size_t)((ny + kN - 1) / kN) * ((nx + kK - 1) / kK);  // contraction 2
  return 256 + (tx + ty) * 2 * kTBytes;
}

size_t adjoint_tc_ranges_bytes(int64_t n) { return sizeof(int4) * (size_t)((n + kM - 1) / kM); }

cudaError_t launch_adjoint_gauss_tc(const float4* pts, const float* wts, const uint32_t* vals,
                                    int4* ranges, const CallScalars* sort_err, int64_t n,
                                    const float* G, const float2* gxt, const float2* gyt, int nx,
                                    int ny, double cell, double h, float* grad_xy, float* grad_w,
                                    double* hterm, double* lterm, void* ws, int max_ctas,
                                    cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_adjoint_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSmemBytes);
  if (e != cudaSuccess) return e;
  CallScalars* gscal = static_cast<CallScalars*>(ws);
  unsigned char* tiles1 = static_cast<unsigned char*>(ws) + 256;
  const int rows1 = (nx + kN - 1) / kN * kN, ns1 = (ny + kK - 1) / kK;
  const int rows2 = (ny + kN - 1) / kN * kN, ns2 = (nx + kK - 1) / kK;
  unsigned char* tiles2 = tiles1 + (size_t)rows1 * ns1 * 2 * kRowBytes;
  const int64_t cells = (int64_t)nx * ny;
  if ((e = cudaMemsetAsync(gscal, 0, sizeof(CallScalars), s)) != cudaSuccess) return e;
  k_abs_max<<<std::min(blocks_for_tc(cells), 152 * 4), 256, 0, s>>>(G, cells, gscal);
  k_tile_cotangent<<<blocks_for_tc((int64_t)rows1 * ns1 * 8), 256, 0, s>>>(G, nx, ny, 0, rows1, ns1,
                                                                           gscal, tiles1);
  k_tile_cotangent<<<blocks_for_tc((int64_t)rows2 * ns2 * 8), 256, 0, s>>>(G, nx, ny, 1, rows2, ns2,
                                                                           gscal, tiles2);
  note_launches(3);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const double sigma = 1.0 / (h * 1.17741002251547469101);  // Gaussian prepared units
  const int items = (int)((n + kM - 1) / kM);
  AdjTcArgs a = {};
  a.pts = pts;
  a.wts = wts;
  a.vals = vals;
  a.ranges = ranges;
  a.sort_err = sort_err;
  a.n = n;
  a.cs = (float)(cell * sigma);
  a.inv_cs = (float)(1.0 / (cell * sigma));
  a.gscal = gscal;
  a.c = 1.0 / (2.0 * 3.14159265358979323846 * (double)n * h * h);
  a.k_xy = 1.17741002251547469101 / h;  // sqrt(2 ln 2) / h
  a.k_h = 1.38629436111989061883 / h;   // 2 ln 2 / h
  a.grad_xy = grad_xy;
  a.grad_w = grad_w;
  a.hterm = hterm;
  a.lterm = lterm;
  if (ranges) {
    k_adj_ranges<<<(items + 7) / 8, 256, 0, s>>>(pts, n, items, a.cs, (float)kAdjTcReach, nx, ny,
                                                 ranges);
    note_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const int grid = std::max(1, std::min(items, max_ctas));
  for (int axis = 0; axis < 2; ++axis) {
    a.axis = axis;
    a.tiles = axis == 0 ? tiles1 : tiles2;
    a.acc_tab = axis == 0 ? gxt : gyt;
    a.k_tab = axis == 0 ? gyt : gxt;
    a.acc_cells = axis == 0 ? nx : ny;
    a.k_cells = axis == 0 ? ny : nx;
    a.rows = axis == 0 ? rows1 : rows2;
    k_adjoint_tc<<<grid, kThreads, kSmemBytes, s>>>(a, gscal);
    note_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace kde
