// The window form of the Gaussian adjoint (kde_adjoint.cu) for points in bin
// order: groups of points of one bin share their window.
//
// A point's window of +-8 bandwidths costs 2601 cells and three FMAs per cell
// at h = 3 cells, one warp per point, each cell read again for every point.
// Here the points are sorted into bins of 8 x 8 cells; a CTA takes up to 64
// points of a bin and the W x W cells that hold all their windows
// (W = 8 + 2 R rounded up), and forms two small matrix products in FP32
//   U[p, j] = sum_i A[p, i] G[j, i]     V[p, i] = sum_j B[p, j] G[j, i]
// from the points' factors A, B and the cotangent tile, all in shared memory:
// two FMAs per cell and point instead of three, eight points by W / 8 cells per
// thread, so that each shared-memory read feeds 8 FMAs.  Then
//   dL/dw ~ sum_j B U,  dL/dy ~ sum_j t B U,  dL/dx ~ sum_i s A V,
//   h-term ~ sum_j t^2 B U + sum_i s^2 A V.
// Terms beyond a point's own +-8 bandwidths but inside the shared window are
// added where the other form leaves them out (they are below e^-32, for a finite
// cotangent: a group whose window holds an infinity or a NaN, which makes all its
// sums infinities or NaN, sums each point over its own window instead, so that only
// the points that reach that cell see it).
// The chains over i and j run from the window's ends towards its middle, the small
// terms first, so that each of the W additions rounds a sum no larger than it has
// to be: against FP64, rms over 200,000 points of the mixture x 512^2, from one end
// to the other 0.97 to 1.06 times the one-point form's error for the random
// cotangent and the LSCV loss's at h = 0.8 to 2.2 cells and 1.1 to 1.4 times for a smooth
// one whose dL/dx nearly cancels; so 0.86 to 1.03 and 1.1 to 1.24.
// Bound by FP32 FMA issue.  1.47M points x 1024^2, h = 3.07 cells: 3.33 ms one
// warp per point, 0.79 ms in groups (0.9 with the sort), 0.75 with the inner loops
// ended at the window's 58 cells instead of the 64 of the tables.
#include <algorithm>

#include "kde_internal.cuh"
#include "kernel_factors.cuh"

namespace kde {
namespace {

constexpr float kLog2e = 1.44269504088896340736f;
__device__ __forceinline__ float gauss(float s) { return ex2_approx(-0.5f * kLog2e * s * s); }

constexpr int kP = kAdjGroup;  // points per group
constexpr uint32_t kFar = 1024;  // points per item beyond every cell's reach
constexpr int kThreads = 128;  // two warps form U, two form V
constexpr int kPP = kP + 4;    // row of the y-factor table: 16-byte aligned, spread over the banks

// Lists the groups of every bin (first point and count; the order is whatever
// the atomics give and decides only which CTA takes a group), and those of the
// points beyond every cell's reach, which only get zeros.  Fewer than kAdjFew points
// left over in a bin are listed one by one instead, for the one-point form: a
// group costs its tile however few its points are, as much as about 9 to 17 of them
// one at a time (points spread evenly, 1M x 4096^2, 4 a bin, h = 3 cells: 6.0 ms
// in groups, 2.3 one by one; a mixture of lanes, ports and even ones 2.7 and 1.2).  After a timed-out sort the bin starts need not rise,
// and the differences of two that fall would list groups past the end of the list:
// nothing is listed then.
__device__ __forceinline__ uint32_t take_slots(uint32_t mine, uint32_t* count) {
  const int lane = threadIdx.x & 31;
  uint32_t incl = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  uint32_t base = 0;
  if (lane == 31 && incl) base = atomicAdd(count, incl);
  return __shfl_sync(0xffffffffu, base, 31) + incl - mine;
}
__global__ void __launch_bounds__(256)
    k_adj_groups(const uint32_t* __restrict__ start, int nbins, int64_t m,
                 int4* __restrict__ list, uint32_t* __restrict__ singles,
                 uint32_t* __restrict__ count, const CallScalars* __restrict__ err) {
  if (*reinterpret_cast<const volatile int*>(&err->err) & kErrSortTimeout) return;
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t a = 0, n = 0;
  if (b <= nbins) {
    a = start[b];
    n = (b < nbins ? start[b + 1] : (uint32_t)m) - a;
  }
  uint32_t rest = n % kP;
  if (b == nbins || rest >= (uint32_t)kAdjFew) rest = 0;
  n -= rest;
  const uint32_t most = b < nbins ? kP : kFar, g = (n + most - 1) / most;
  const uint32_t base = take_slots(g, count);
  for (uint32_t k = 0; k < g; ++k)
    list[base + k] = make_int4(b, (int)(a + k * most), (int)min(most, n - k * most), 0);
  const uint32_t first = take_slots(rest, count + 2);
  for (uint32_t k = 0; k < rest; ++k) singles[first + k] = a + n + k;
}

template <int RT>
struct GroupCfg {
  static constexpr int W = 8 * RT;    // cells of the window's side
  static constexpr int WP = W + 4;    // its rows in shared memory (WP / 4 odd: no bank conflicts)
  static constexpr int kG = 0, kA = kG + W * WP, kB = kA + kP * WP, kGx = kB + W * kPP;
  static constexpr int kGy = kGx + 2 * W, kPt = kGy + 2 * W, kW = kPt + 4 * kP;
  static constexpr int kSum = kW + 2 * kP, kFloats = kSum + 5 * kP;
  static constexpr size_t kSmem = sizeof(float) * kFloats;
};

// The sums of a group's points over their own windows, +-reach cells from the
// point's cell as in the one-point form, one warp per point, lanes over the columns.
template <int RT>
__device__ __noinline__ void own_windows(const float* sm, int np, int ib, int jb, int nx, int ny,
                                         int reach, double cell_s, float* sum) {
  using C = GroupCfg<RT>;
  const float2* sgx = reinterpret_cast<const float2*>(sm + C::kGx);
  const float2* sgy = reinterpret_cast<const float2*>(sm + C::kGy);
  const int lane = threadIdx.x & 31;
  for (int p = threadIdx.x >> 5; p < np; p += kThreads / 32) {
    const float4 P = reinterpret_cast<const float4*>(sm + C::kPt)[p];
    const int ic = (int)floor(((double)P.x + (double)P.y) / cell_s);
    const int jc = (int)floor(((double)P.z + (double)P.w) / cell_s);
    const int i0 = max(max(ic - reach, 0), ib), i1 = min(min(ic + reach, nx - 1), ib + C::W - 1);
    const int j0 = max(max(jc - reach, 0), jb), j1 = min(min(jc + reach, ny - 1), jb + C::W - 1);
    float aw = 0.f, ax = 0.f, ay = 0.f, ah = 0.f;
    for (int j = j0; j <= j1; ++j) {
      const float2 gy = sgy[j - jb];
      const float t = (gy.x - P.z) + (gy.y - P.w), B = gauss(t);
      float u = 0.f, v = 0.f, x = 0.f;
      for (int i = i0 + lane; i <= i1; i += 32) {
        const float2 gx = sgx[i - ib];
        const float S = (gx.x - P.x) + (gx.y - P.y), A = gauss(S);
        const float g = sm[C::kG + (j - jb) * C::WP + (i - ib)];
        u = fmaf(g, A, u);
        v = fmaf(g, S * A, v);
        x = fmaf(g, S * (S * A), x);
      }
      const float Bu = B * u;
      aw += Bu;
      ax = fmaf(B, v, ax);
      ay = fmaf(t, Bu, ay);
      ah = fmaf(B, x, fmaf(t * t, Bu, ah));
    }
    for (int o = 16; o > 0; o >>= 1) {
      aw += __shfl_xor_sync(0xffffffffu, aw, o);
      ax += __shfl_xor_sync(0xffffffffu, ax, o);
      ay += __shfl_xor_sync(0xffffffffu, ay, o);
      ah += __shfl_xor_sync(0xffffffffu, ah, o);
    }
    if (lane == 0) {
      sum[5 * p] = aw;
      sum[5 * p + 1] = ay;
      sum[5 * p + 2] = ah;
      sum[5 * p + 3] = ax;
      sum[5 * p + 4] = 0.f;
    }
  }
}

template <int RT>
__global__ void __launch_bounds__(kThreads)
    k_adj_group(const float4* __restrict__ pts, const float* __restrict__ wts,
                const uint32_t* __restrict__ vals, int64_t n, const int4* __restrict__ list,
                const uint32_t* __restrict__ count, uint32_t* __restrict__ next,
                const float* __restrict__ G, const float2* __restrict__ gxt,
                const float2* __restrict__ gyt, int nx, int ny, int nbx, int nbins, int R, int reach,
                double cell_s, float c, float inv_h, float* __restrict__ grad_xy,
                float* __restrict__ grad_w, double* __restrict__ hterm,
                double* __restrict__ lterm, const CallScalars* __restrict__ err) {
  using C = GroupCfg<RT>;
  constexpr int W = C::W, WP = C::WP;
  extern __shared__ __align__(16) float sm[];
  float* sG = sm + C::kG;  // [W][WP], row j
  float* sA = sm + C::kA;  // [kP][WP], point p, column i
  float* sB = sm + C::kB;  // [W][kPP], row j, point p
  float2* sgx = reinterpret_cast<float2*>(sm + C::kGx);
  float2* sgy = reinterpret_cast<float2*>(sm + C::kGy);
  float4* sP = reinterpret_cast<float4*>(sm + C::kPt);
  float* sW = sm + C::kW;
  uint32_t* sIdx = reinterpret_cast<uint32_t*>(sW + kP);
  float* sum = sm + C::kSum;  // [kP][5]: w, y, y h-term, x, x h-term
  __shared__ uint32_t s_item;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // after a timed-out sort the bin starts are not trusted: compute nothing
  if (*reinterpret_cast<const volatile int*>(&err->err) & kErrSortTimeout) return;
  const int wu = kAdjBin + 2 * R;  // the window's cells, of the W (a multiple of 32) computed
  const uint32_t n_items = *count;
  for (;;) {
    __syncthreads();
    if (tid == 0) s_item = atomicAdd(next, 1u);
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= n_items) return;
    const int4 it = list[item];
    const int np = it.z;
    if (it.x >= nbins) {  // out of every cell's reach
      for (int t = tid; t < np; t += kThreads) {
        const uint32_t p = (uint32_t)it.y + t;
        const uint32_t o = vals[p];
        if (o < n) {
          if (grad_w) grad_w[o] = 0.f;
          grad_xy[2 * (int64_t)o] = 0.f;
          grad_xy[2 * (int64_t)o + 1] = 0.f;
          hterm[p] = 0.0;
          lterm[p] = 0.0;
        }
      }
      continue;
    }
    const int ib = (it.x % nbx) * kAdjBin - R, jb = (it.x / nbx) * kAdjBin - R;
    if (tid < kP) {
      float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
      float w = 0.f;
      uint32_t o = 0xffffffffu;
      if (tid < np) {
        P = pts[it.y + tid];
        w = wts[it.y + tid];
        o = vals[it.y + tid];
      }
      sP[tid] = P;
      sW[tid] = w;
      sIdx[tid] = o;
    }
    for (int x = tid; x < W; x += kThreads) {
      sgx[x] = gxt[min(max(ib + x, 0), nx - 1)];
      sgy[x] = gyt[min(max(jb + x, 0), ny - 1)];
    }
    // the cotangent tile, zero outside the grid
    for (int r = warp; r < W; r += kThreads / 32) {
      const int j = jb + r;
      const float* row = G + (int64_t)j * nx + ib;
#pragma unroll
      for (int x0 = 0; x0 < W; x0 += 32) {
        const int x = x0 + lane, i = ib + x;
        sG[r * WP + x] = j >= 0 && j < ny && i >= 0 && i < nx ? __ldg(row + x) : 0.f;
      }
    }
    __syncthreads();
    // the factor tables, lanes along a row of each
    const int np8 = (np + 7) & ~7;
    for (int p = warp; p < np8; p += kThreads / 32) {
      const float4 P = sP[p];
      const bool in = p < np;
#pragma unroll
      for (int x0 = 0; x0 < W; x0 += 32) {
        const float2 g = sgx[x0 + lane];
        sA[p * WP + x0 + lane] = in ? gauss((g.x - P.x) + (g.y - P.y)) : 0.f;
      }
    }
#pragma unroll
    for (int h = 0; h < kP / 32; ++h) {
      const int p = 32 * h + lane;
      if (32 * h >= np8) break;
      const float4 P = sP[p];
      const bool in = p < np;
      for (int r = warp; r < W; r += kThreads / 32) {
        const float2 g = sgy[r];
        sB[r * kPP + p] = in ? gauss((g.x - P.z) + (g.y - P.w)) : 0.f;
      }
    }
    __syncthreads();
    const int blk = lane & 7;  // block of cells
    const int steps = (wu + 3) / 4;  // of four columns, from either end in turn
    bool odd = false;  // a sum that is not finite: every point's is when a cell is not
    if (warp < 2) {
      // U: points p = 8 s + pb, rows j = 8 r + blk; four columns per step
      const int pb = (warp << 2) | (lane >> 3);
      if (pb < np) {
        float acc[8][RT];
#pragma unroll
        for (int s = 0; s < 8; ++s)
#pragma unroll
          for (int r = 0; r < RT; ++r) acc[s][r] = 0.f;
        const float* a0 = sA + pb * WP;
        const float* g0 = sG + blk * WP;
#pragma unroll 1
        for (int q = 0; q < steps; ++q) {
          const int i = 4 * (q & 1 ? steps - 1 - (q >> 1) : q >> 1);
          float4 a[8];
#pragma unroll
          for (int s = 0; s < 8; ++s)
            a[s] = *reinterpret_cast<const float4*>(a0 + 8 * s * WP + i);
#pragma unroll
          for (int r = 0; r < RT; ++r) {
            const float4 g = *reinterpret_cast<const float4*>(g0 + 8 * r * WP + i);
#pragma unroll
            for (int s = 0; s < 8; ++s) {
              acc[s][r] = fmaf(a[s].x, g.x, acc[s][r]);
              acc[s][r] = fmaf(a[s].y, g.y, acc[s][r]);
              acc[s][r] = fmaf(a[s].z, g.z, acc[s][r]);
              acc[s][r] = fmaf(a[s].w, g.w, acc[s][r]);
            }
          }
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const int p = 8 * s + pb;
          const float4 P = sP[p];
          float w4[4], y4[4], h4[4];  // four chains, added in pairs: less rounding
#pragma unroll
          for (int r = 0; r < RT; ++r) {
            const int j = 8 * r + blk;
            const float2 g = sgy[j];
            const float t = (g.x - P.z) + (g.y - P.w);
            const float Bu = (p < np8 ? sB[j * kPP + p] : 0.f) * acc[s][r];
            w4[r & 3] = r < 4 ? Bu : w4[r & 3] + Bu;
            y4[r & 3] = r < 4 ? t * Bu : fmaf(t, Bu, y4[r & 3]);
            h4[r & 3] = r < 4 ? t * t * Bu : fmaf(t * t, Bu, h4[r & 3]);
          }
          float aw = (w4[0] + w4[1]) + (w4[2] + w4[3]);
          float ay = (y4[0] + y4[1]) + (y4[2] + y4[3]);
          float ah = (h4[0] + h4[1]) + (h4[2] + h4[3]);
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) {
            const unsigned m = 0xffu << (lane & 24);
            aw += __shfl_xor_sync(m, aw, o);
            ay += __shfl_xor_sync(m, ay, o);
            ah += __shfl_xor_sync(m, ah, o);
          }
          if (blk == 0 && p < np) {
            sum[5 * p] = aw;
            sum[5 * p + 1] = ay;
            sum[5 * p + 2] = ah;
            odd |= !(fabsf(aw) + fabsf(ay) + fabsf(ah) < INFINITY);
          }
        }
      }
    } else {
      // V: points p = 8 pb + s, columns i = 32 g + 4 blk + c; one row per step
      const int pb = ((warp - 2) << 2) | (lane >> 3);
      if (8 * pb < np) {
        float acc[8][RT];
#pragma unroll
        for (int s = 0; s < 8; ++s)
#pragma unroll
          for (int r = 0; r < RT; ++r) acc[s][r] = 0.f;
        const float* b0 = sB + 8 * pb;
        const float* g0 = sG + 4 * blk;
#pragma unroll 2
        for (int q = 0; q < wu; ++q) {  // wu is even
          const int j = q & 1 ? wu - 1 - (q >> 1) : q >> 1;
          const float4 b1 = *reinterpret_cast<const float4*>(b0 + j * kPP);
          const float4 b2 = *reinterpret_cast<const float4*>(b0 + j * kPP + 4);
          const float b[8] = {b1.x, b1.y, b1.z, b1.w, b2.x, b2.y, b2.z, b2.w};
#pragma unroll
          for (int g = 0; g < RT / 4; ++g) {
            const float4 v = *reinterpret_cast<const float4*>(g0 + j * WP + 32 * g);
#pragma unroll
            for (int s = 0; s < 8; ++s) {
              acc[s][4 * g] = fmaf(b[s], v.x, acc[s][4 * g]);
              acc[s][4 * g + 1] = fmaf(b[s], v.y, acc[s][4 * g + 1]);
              acc[s][4 * g + 2] = fmaf(b[s], v.z, acc[s][4 * g + 2]);
              acc[s][4 * g + 3] = fmaf(b[s], v.w, acc[s][4 * g + 3]);
            }
          }
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const int p = 8 * pb + s;
          const float4 P = sP[p];
          float x4[4], h4[4];
#pragma unroll
          for (int r = 0; r < RT; ++r) {
            const int i = 32 * (r >> 2) + 4 * blk + (r & 3);
            const float2 g = sgx[i];
            const float sx = (g.x - P.x) + (g.y - P.y);
            const float f = sA[p * WP + i] * acc[s][r];
            x4[r & 3] = r < 4 ? sx * f : fmaf(sx, f, x4[r & 3]);
            h4[r & 3] = r < 4 ? sx * sx * f : fmaf(sx * sx, f, h4[r & 3]);
          }
          float ax = (x4[0] + x4[1]) + (x4[2] + x4[3]);
          float ah = (h4[0] + h4[1]) + (h4[2] + h4[3]);
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) {
            const unsigned m = 0xffu << (lane & 24);
            ax += __shfl_xor_sync(m, ax, o);
            ah += __shfl_xor_sync(m, ah, o);
          }
          if (blk == 0 && p < np) {
            sum[5 * p + 3] = ax;
            sum[5 * p + 4] = ah;
            odd |= !(fabsf(ax) + fabsf(ah) < INFINITY);
          }
        }
      }
    }
    if (__syncthreads_or(odd)) {
      own_windows<RT>(sm, np, ib, jb, nx, ny, reach, cell_s, sum);
      __syncthreads();
    }
    if (tid < np) {
      const uint32_t o = sIdx[tid];
      if (o < n) {  // the caller's order
        const float w = sW[tid];
        const float* r = sum + 5 * tid;
        const float gw = c * r[0];
        if (grad_w) grad_w[o] = gw;
        grad_xy[2 * (int64_t)o] = c * w * inv_h * r[3];
        grad_xy[2 * (int64_t)o + 1] = c * w * inv_h * r[1];
        // only summed: kept in bin order
        hterm[it.y + tid] = (double)c * w * inv_h * (r[2] + r[4]);
        lterm[it.y + tid] = (double)w * gw;
      }
    }
  }
}

template <int RT>
cudaError_t launch_rt(const AdjGroupArgs& a, cudaStream_t s) {
  using C = GroupCfg<RT>;
  cudaError_t e = cudaFuncSetAttribute(k_adj_group<RT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adj_group<RT>, kThreads, C::kSmem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorLaunchOutOfResources;
  const int64_t most = a.m / kP + a.nbins + 2;
  const int grid = (int)std::min<int64_t>((int64_t)per_sm * a.sms, most);
  k_adj_group<RT><<<grid, kThreads, C::kSmem, s>>>(
      a.pts, a.wts, a.vals, a.n, a.list, a.counters, a.counters + 1, a.G, a.gxt, a.gyt, a.nx, a.ny,
      a.nbx, a.nbins, a.R, a.reach, a.cell_s, a.c, a.inv_h, a.grad_xy, a.grad_w, a.hterm, a.lterm,
      a.err);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

// The points' bins come from FP32 keys, off by up to 3 units of 2^-24 of the
// coordinate, and the window hangs on the bin: one cell to spare for keys of up to
// 2^21 cells, one more for every further 2^21 along the longer axis.
int adj_group_radius(double cell, double h, int nx, int ny) {
  return (int)ceil(std::min(8.0 * h / cell, 1e6)) + 1 + (std::max(nx, ny) >> 21);
}
// 12 cells per thread at most: 96 x 96 cells and the tables of 64 points take 88 KB
bool adj_group_fits(int R) { return kAdjBin + 2 * R <= 96; }

cudaError_t launch_adjoint_list(const AdjGroupArgs& a, cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(a.counters, 0, 3 * sizeof(uint32_t), s);
  if (e != cudaSuccess) return e;
  k_adj_groups<<<(a.nbins + 1 + 255) / 256, 256, 0, s>>>(a.start, a.nbins, a.m, a.list, a.singles,
                                                         a.counters, a.err);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_group(const AdjGroupArgs& a, double cell, double h, cudaStream_t s) {
  cudaError_t e = launch_adjoint_list(a, s);
  if (e != cudaSuccess) return e;
  const int W = kAdjBin + 2 * a.R;
  e = W <= 32 ? launch_rt<4>(a, s) : W <= 64 ? launch_rt<8>(a, s) : launch_rt<12>(a, s);
  return e == cudaSuccess ? launch_adjoint_listed(a, cell, h, s) : e;
}

}  // namespace kde
