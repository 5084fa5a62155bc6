// Path (a): FP32 direct sum on the CUDA cores, any Table 1 kernel.
//
// Every Table 1 kernel is a product f(s,t) = k(s) k(t) (Sec. III-C).  A CTA
// owns 128 x 64 cells; for each batch of 32 points it first tabulates the
// 128 x-factors and 64 (weighted) y-factors of every point in shared memory,
// each evaluated once, then every thread accumulates the outer products of its
// 8 x 8 cells (columns 4t..4t+3 and 64+4t..64+4t+3, eight consecutive rows):
// per point two 16-byte reads of each table and 64 FMAs.  The tables are
// double-buffered, so one barrier per batch separates a batch's tabulation
// from its use, and the next batch's points are loaded into registers
// while the current batch is accumulated.  Points arrive in tiles of 256;
// each thread sums one tile in registers and adds that partial into a
// (hi, lo) running sum with an error-free two-sum, so the result does not
// degrade with the number of points a cell sees.  The running sums of a CTA's
// 8192 cells, 64 KB, live in tensor memory, which this path has no other use
// for: four CTAs take all of an SM's.
#include "kde_internal.cuh"
#include "kernel_factors.cuh"
#include "tc_ptx.cuh"

namespace kde {
namespace {

constexpr int kThreads = 128;  // 16 (x) x 8 (y) threads, 8 x 8 cells each
constexpr int kTileX = 128;    // cells along x per CTA
constexpr int kTileY = 64;     // cells along y per CTA
constexpr int kPtsTile = 256;  // points per register partial (two-sum cadence)
constexpr int kBatch = 32;     // points per factor table
constexpr uint32_t kRunCols = 128;  // tensor memory columns of a CTA's running sums
// a table row, a point's x and y factors, is four floats longer than these, so
// that eight lanes' 16-byte stores, a row each, take all the banks
constexpr int kRow = kTileX + kTileY + 4;
constexpr int kTable = kBatch * kRow;  // floats per table buffer

struct TableRow {
  float4 xa, xb, ya, yb;
};

__device__ __forceinline__ TableRow table_row(const float* KX, const float* KY, int q, int tx,
                                              int ty) {
  // columns 4tx.. and 64+4tx..: a half-warp reads 256 contiguous bytes
  TableRow r;
  r.xa = *reinterpret_cast<const float4*>(KX + q * kRow + tx * 4);
  r.xb = *reinterpret_cast<const float4*>(KX + q * kRow + 64 + tx * 4);
  r.ya = *reinterpret_cast<const float4*>(KY + q * kRow + ty * 8);
  r.yb = *reinterpret_cast<const float4*>(KY + q * kRow + ty * 8 + 4);
  return r;
}

// f32x2 arithmetic as the scalar instructions round it (denormals kept).
__device__ __forceinline__ float2 p_add(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) {
  return p_add(a, make_float2(-b.x, -b.y));
}
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// Bound by the FMA pipe (a packed FMA is two of its cycles) and shared memory's
// 128 bytes per clock to the registers.  1M points x 512^2: 11.9 ms with the
// running sums in global memory, a table stage of a cell per lane and scalar
// FMAs; 11.5 with points per lane and packed FMAs; 9.6 with the sums in tensor
// memory; 9.3 = 28 Tpair/s with twice the splits (choose_simt_splits).
template <int KID>
__global__ void __launch_bounds__(kThreads, kSimtCtasPerSm)
    k_simt(const float4* __restrict__ pts, const float* __restrict__ wts, int64_t n_pad,
           int64_t per_split, const float2* __restrict__ gxt, const float2* __restrict__ gyt,
           int nx, int ny, float cs_hi, float cs_lo, float scale, float* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* tables = reinterpret_cast<float*>(smem);                        // [2][kTable]
  const int tid = threadIdx.x, lane = tid & 31;
  const int tx = tid & 15, ty = tid >> 4;
  const int cx0 = blockIdx.x * kTileX, cy0 = blockIdx.y * kTileY;
  float* dst = part + (int64_t)blockIdx.z * nx * ny;
  auto cell = [&](int b, int a, int& x, int& y) {
    y = cy0 + ty * 8 + b;
    x = cx0 + (a < 4 ? tx * 4 + a : 64 + tx * 4 + a - 4);
  };

  const int64_t p_begin = (int64_t)blockIdx.z * per_split;
  int64_t p_end = p_begin + per_split;
  if (p_end > n_pad) p_end = n_pad;
  if (p_begin >= p_end) {  // no points in this split: a zero partial
#pragma unroll
    for (int b = 0; b < 8; ++b)
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        int x, y;
        cell(b, a, x, y);
        if (x < nx && y < ny) dst[(int64_t)y * nx + x] = 0.f;
      }
    return;
  }
  __shared__ uint32_t tmem_slot;
  if (tid < 32) tc::tmem_alloc(&tmem_slot, kRunCols);
  __syncthreads();
  // this warp's lanes; row b's eight hi parts at column 16 b, its lo parts after
  const uint32_t run = tmem_slot + ((uint32_t)(tid >> 5) << 21);
  {
    const float zero[16] = {};
#pragma unroll
    for (int b = 0; b < 8; ++b) tc::tmem_st16(run + 16 * b, zero);
    tc::tmem_wait_st();
  }

  // factor roles: warp w makes columns 32 w.. and rows 16 w.. of every point,
  // a point per lane
  static_assert(kThreads == kTileX && kThreads == 2 * kTileY, "factor roles");
  static_assert(kPtsTile % kBatch == 0 && kBatch == 32, "one point per lane per batch");
  const int warp = tid >> 5;
  const float2 gx0 = gxt[cx0], gy0 = gyt[cy0];

  // Every warp holds the points of the next batch in registers, one per
  // lane, loaded while the current batch is accumulated (the global-memory
  // latency hides behind a whole batch), and makes their factors lane by lane:
  // the offset from cell j is that from the tile's first cell plus j times the
  // cell's side (pair_offset).  A cell per lane, with the points broadcast by shuffles, took three
  // times as much of shared memory's bandwidth.
  float4 nP;
  float nW;
  auto fetch = [&](int64_t first) {
    const int64_t p = first + lane;
    const bool in = p < p_end;
    nP = in ? pts[p] : make_float4(0.f, 0.f, 0.f, 0.f);
    nW = in ? wts[p] : 0.f;
  };
  fetch(p_begin);

  int buf = 0;
  for (int64_t base = p_begin; base < p_end; base += kPtsTile) {
    float2 acc[8][4];
#pragma unroll
    for (int b = 0; b < 8; ++b)
#pragma unroll
      for (int a = 0; a < 4; ++a) acc[b][a] = make_float2(0.f, 0.f);

    for (int bb = 0; bb < kPtsTile; bb += kBatch, buf ^= 1) {
      float* KX = tables + buf * kTable;  // [kBatch][kRow]
      float* KY = KX + kTileX;            // the same rows' y factors
      const float4 P = nP;
      const float W = nW;
      // This buffer was last read two batches ago, before the barrier of the
      // previous batch, which every thread has passed.
      auto factors = [&](float2 d0, int j0, int count, float w, float* row) {
#pragma unroll 8
        for (int q = 0; q < count; q += 4) {
          float v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float j = (float)(j0 + q + e);
            v[e] = w * kfactor<KID>(fmaf(j, cs_hi, d0.x) + fmaf(j, cs_lo, d0.y));
          }
          *reinterpret_cast<float4*>(row + j0 + q) = make_float4(v[0], v[1], v[2], v[3]);
        }
      };
      factors(pair_offset(gx0, make_float2(P.x, P.y)), 32 * warp, 32, 1.0f, KX + lane * kRow);
      factors(pair_offset(gy0, make_float2(P.z, P.w)), 16 * warp, 16, W, KY + lane * kRow);
      __syncthreads();
      fetch(base + bb + kBatch);
#pragma unroll 2
      for (int q = 0; q < kBatch; ++q) {
        const TableRow cur = table_row(KX, KY, q, tx, ty);
        const float2 kx[4] = {make_float2(cur.xa.x, cur.xa.y), make_float2(cur.xa.z, cur.xa.w),
                              make_float2(cur.xb.x, cur.xb.y), make_float2(cur.xb.z, cur.xb.w)};
        const float ky[8] = {cur.ya.x, cur.ya.y, cur.ya.z, cur.ya.w,
                             cur.yb.x, cur.yb.y, cur.yb.z, cur.yb.w};
#pragma unroll
        for (int b = 0; b < 8; ++b)
#pragma unroll
          for (int a = 0; a < 4; ++a)
            acc[b][a] = p_fma(kx[a], make_float2(ky[b], ky[b]), acc[b][a]);
      }
    }
    // this tile's partials into the running sums, a row at a time
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      uint32_t in[16];
      tc::tmem_ld_async(run + 16 * b, in);
      tc::tmem_wait_ld();
      float out[16];
#pragma unroll
      for (int a = 0; a < 8; a += 2) {
        const float2 r = make_float2(__uint_as_float(in[a]), __uint_as_float(in[a + 1]));
        const float2 v = acc[b][a / 2], hi = p_add(r, v), t = p_sub(hi, r);
        const float2 lo = p_add(make_float2(__uint_as_float(in[8 + a]), __uint_as_float(in[9 + a])),
                                p_add(p_sub(r, p_sub(hi, t)), p_sub(v, t)));
        out[a] = hi.x;
        out[a + 1] = hi.y;
        out[8 + a] = lo.x;
        out[9 + a] = lo.y;
      }
      tc::tmem_st16(run + 16 * b, out);
    }
    tc::tmem_wait_st();
  }
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    uint32_t in[16];
    tc::tmem_ld_async(run + 16 * b, in);
    tc::tmem_wait_ld();
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      int x, y;
      cell(b, a, x, y);
      if (x < nx && y < ny)
        dst[(int64_t)y * nx + x] = (__uint_as_float(in[a]) + __uint_as_float(in[8 + a])) * scale;
    }
  }
  __syncthreads();
  if (tid < 32) tc::tmem_dealloc(tmem_slot, kRunCols);
}

template <int KID>
cudaError_t launch_kid(const float4* pts, const float* wts, int64_t n_pad, const float2* gxt,
                       const float2* gyt, int nx, int ny, double cs, int splits, float scale,
                       float* part, cudaStream_t s) {
  constexpr size_t smem = 2 * kTable * sizeof(float);
  // per-device attribute; cheap, so set on every launch
  cudaError_t e = cudaFuncSetAttribute(k_simt<KID>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  int64_t per = (n_pad + splits - 1) / splits;
  per = (per + kPtsTile - 1) / kPtsTile * kPtsTile;
  if (per < kPtsTile) per = kPtsTile;
  float cs_hi, cs_lo;
  split_side(cs, &cs_hi, &cs_lo);
  dim3 grid((nx + kTileX - 1) / kTileX, (ny + kTileY - 1) / kTileY, splits);
  k_simt<KID><<<grid, kThreads, smem, s>>>(pts, wts, n_pad, per, gxt, gyt, nx, ny, cs_hi,
                                           cs_lo, scale, part);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_simt(int kid, const float4* pts, const float* wts, int64_t n_pad,
                        const float2* gxt, const float2* gyt, int nx, int ny, double cs, int splits,
                        float scale, float* part, cudaStream_t s) {
  switch (kid) {
#define KDE_CASE(K)                                                                          \
  case K:                                                                                    \
    return launch_kid<K>(pts, wts, n_pad, gxt, gyt, nx, ny, cs, splits, scale, part, s);
    KDE_CASE(KDE_UNIFORM)
    KDE_CASE(KDE_TRIANGULAR)
    KDE_CASE(KDE_EPANECHNIKOV)
    KDE_CASE(KDE_QUARTIC)
    KDE_CASE(KDE_TRIWEIGHT)
    KDE_CASE(KDE_TRICUBE)
    KDE_CASE(KDE_GAUSSIAN)
    KDE_CASE(KDE_COSINE)
#undef KDE_CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace kde
