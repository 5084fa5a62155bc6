// Adjoint of the Gaussian density and the grid LSCV loss.
//
// Density (Sec. III-C, Eq. 7 read as a direct sum, Gaussian row of Table 1):
//   F_ij = c sum_p w_p A_ip B_jp,  A_ip = exp(-s_ip^2/2), B_jp = exp(-t_jp^2/2),
//   s_ip = (gx_i - x_p)/h, t_jp = (gy_j - y_p)/h, c = 1/(2 pi N h^2).
// For a cotangent G = dL/dF:
//   dL/dw_p = c sum_ij G_ij A_ip B_jp
//   dL/dx_p = c w_p / h sum_ij G_ij s_ip A_ip B_jp     (dA/dx_p = A s / h)
//   dL/dy_p = c w_p / h sum_ij G_ij t_jp A_ip B_jp
//   dL/dh   = -(2/h) sum_ij G_ij F_ij + c/h sum_p w_p sum_ij G_ij (s^2 + t^2) A B
// and sum_ij G_ij F_ij = sum_p w_p dL/dw_p, so F itself is not needed.
//
// One warp per point in turn, over batches of 32 points: lanes take the
// columns of the point's window (for a window of at most 16 columns, groups
// of lanes take alternate rows), the rows are walked in order, and the four
// sums are reduced across the warp in a fixed order (reproducible).  The sum
// over a window is separable: per row, three FMAs per cell form sum G A,
// sum G s A and sum G s^2 A, which the row's B and t then weight.  The window
// itself (FP64) is found once per point, by the lane that later writes the
// point's results; the batch's points, windows and sums pass between the
// lanes through shared memory.  The window spans +-8 bandwidths (clamped to
// the grid): beyond it every term is below exp(-32) of the largest, far under
// the accuracy of the FP32 sums.
#include "kde_internal.cuh"
#include "kernel_factors.cuh"

namespace kde {
namespace {

constexpr float kLog2e = 1.44269504088896340736f;

__device__ __forceinline__ float gauss(float s) { return ex2_approx(-0.5f * kLog2e * s * s); }

// COLS: window columns a lane keeps in registers per block of 32 * COLS
// columns (the host picks the smallest power of two that covers the window).
// A window of at most 16 columns takes 2^sub_log2 >= its width lanes per row
// and 32 / 2^sub_log2 rows at a time (sub_log2 = 5 otherwise).  The launch
// bounds are the blocks per SM each COLS fits without spilling registers.
// LIST: the points are those at the sorted positions list[0 .. *list_count), what
// the groups of kde_adjoint_group.cu leave over.  Their count is known here only:
// where they are few, a warp takes as few at a time as keep `busy` warps, those
// that fit the GPU, at work.
template <int COLS, bool LIST>
__global__ void __launch_bounds__(256, COLS == 1 ? 5 : (COLS == 2 ? 4 : (COLS == 4 ? 3 : 1)))
    k_adjoint_gauss(const float4* __restrict__ pts, const float* __restrict__ wts, int64_t n,
                    const uint32_t* __restrict__ list, const uint32_t* __restrict__ list_count,
                    int busy, const uint32_t* __restrict__ vals, const float* __restrict__ G, const float2* __restrict__ gxt,
                    const float2* __restrict__ gyt, int nx, int ny, double cell_s, int R,
                    int sub_log2, float c, float inv_h, float* __restrict__ grad_xy,
                    float* __restrict__ grad_w, double* __restrict__ hterm,
                    double* __restrict__ lterm) {
  // per warp: the batch's points, windows and reduced sums (one slot per point)
  __shared__ float4 sP[8][32];
  __shared__ int4 sWin[8][32];
  __shared__ float4 sSum[8][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  // lanes in groups of 2^sub_log2 over the columns; group g takes rows g, g + ng, ...
  const int ci = lane & ((1 << sub_log2) - 1), rg = lane >> sub_log2, ng = 32 >> sub_log2;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  // batches, and points of a batch: the list's are taken `batches` apart, so that the
  // warps that run at a time, not the points of one, are neighbours
  const int64_t count = LIST ? (int64_t)*list_count : n;
  const int per = LIST ? (int)min((int64_t)32, (count + busy - 1) / busy) : 32;
  const int64_t batches = count ? (count + per - 1) / per : 0;
  for (int64_t batch = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; batch < batches;
       batch += warps) {
    // Lane l prepares point pb + l: its window of cells within R of its cell
    // (X, Y in bandwidths).  This is the FP64 part, so it runs once per point
    // instead of once per lane of the warp.
    auto point = [&](int64_t& pl) {  // the lane's point, if it has one
      const int64_t at = LIST ? batch + lane * batches : batch * 32 + lane;
      if (lane >= per || at >= count) return false;
      pl = LIST ? (int64_t)list[at] : at;
      return true;
    };
    int64_t pl;
    if (point(pl)) {
      const float4 P = pts[pl];
      const double X = (double)P.x + (double)P.y, Y = (double)P.z + (double)P.w;
      const int ic = (int)floor(X / cell_s), jc = (int)floor(Y / cell_s);
      sP[wib][lane] = P;
      sWin[wib][lane] = make_int4(max(ic - R, 0), min(ic + R, nx - 1), max(jc - R, 0),
                                  min(jc + R, ny - 1));
    }
    __syncwarp();
    const int cnt = (int)min((int64_t)per, LIST ? (count - batch + batches - 1) / batches
                                                : count - batch * 32);
    for (int q = 0; q < cnt; ++q) {
      const float4 P = sP[wib][q];
      const int4 win = sWin[wib][q];
      const int i0 = win.x, i1 = win.y, j0 = win.z, j1 = win.w;
      float aw = 0.f, ax = 0.f, ay = 0.f, ah = 0.f;
      if (i0 <= i1 && j0 <= j1) {
        for (int ib = i0; ib <= i1; ib += 32 * COLS) {
          // per column: A, s A and s^2 A (zero outside the window)
          float A[COLS], SA[COLS], S2A[COLS];
          int col[COLS];
#pragma unroll
          for (int k = 0; k < COLS; ++k) {
            const int i = ib + ci + 32 * k;
            col[k] = i <= i1 ? i : -1;
            const float2 g = gxt[min(i, nx - 1)];
            const float S = (g.x - P.x) + (g.y - P.y);
            A[k] = col[k] >= 0 ? gauss(S) : 0.f;
            SA[k] = S * A[k];
            S2A[k] = S * SA[k];
          }
          // Rows in order, four per iteration so their loads are in flight
          // together.  The window sum is separable: with the lane's row sums
          // u = sum G A, v = sum G s A, x = sum G s^2 A,
          //   w += B u,  x_p += B v,  y_p += t B u,  h += B x + t^2 B u.
#pragma unroll 4
          for (int j = j0 + rg; j <= j1; j += ng) {
            const float2 g = gyt[j];
            const float t = (g.x - P.z) + (g.y - P.w);
            const float B = gauss(t);
            const float* Grow = G + (int64_t)j * nx;
            float u = 0.f, v = 0.f, x = 0.f;
#pragma unroll
            for (int k = 0; k < COLS; ++k) {
              const float Gv = col[k] >= 0 ? __ldg(Grow + col[k]) : 0.f;
              u = fmaf(Gv, A[k], u);
              v = fmaf(Gv, SA[k], v);
              x = fmaf(Gv, S2A[k], x);
            }
            const float Bu = B * u;
            aw += Bu;
            ax = fmaf(B, v, ax);
            ay = fmaf(t, Bu, ay);
            ah = fmaf(B, x, fmaf(t * t, Bu, ah));
          }
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        aw += __shfl_xor_sync(0xffffffffu, aw, o);
        ax += __shfl_xor_sync(0xffffffffu, ax, o);
        ay += __shfl_xor_sync(0xffffffffu, ay, o);
        ah += __shfl_xor_sync(0xffffffffu, ah, o);
      }
      if (lane == 0) sSum[wib][q] = make_float4(aw, ax, ay, ah);
    }
    __syncwarp();
    if (point(pl)) {
      const float w = wts[pl];
      const float4 r = sSum[wib][lane];
      const float gw = c * r.x;
      const int64_t to = LIST ? (int64_t)vals[pl] : pl;  // the caller's order
      if (grad_w) grad_w[to] = gw;
      grad_xy[2 * to] = c * w * inv_h * r.y;
      grad_xy[2 * to + 1] = c * w * inv_h * r.z;
      hterm[pl] = (double)c * w * inv_h * r.w;
      lterm[pl] = (double)w * gw;
    }
    __syncwarp();
  }
}

// Fixed-order sums of up to kMaxSums double arrays in two launches: the first
// sums slices of kSumSlice numbers (block x: slice, y: array), the second the
// slices' sums.
constexpr int kMaxSums = 3, kSumThreads = 1024;
constexpr int64_t kSumSlice = 8192;  // one round of kSumThreads x 8 numbers
struct SumSet {
  SumJob job[kMaxSums];
};
template <int THREADS>
__device__ __forceinline__ double block_sum(const double* __restrict__ v, int64_t b0, int64_t b1) {
  __shared__ double sh[THREADS / 32];
  double acc = 0.0;
  constexpr int kAhead = 8;
  for (int64_t i = b0 + threadIdx.x; i < b1; i += (int64_t)kAhead * THREADS) {
    double x[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) x[u] = i + u * THREADS < b1 ? v[i + u * THREADS] : 0.0;
#pragma unroll
    for (int u = 0; u < kAhead; ++u) acc += x[u];
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < THREADS / 32; ++w) r += sh[w];
  return r;
}
__global__ void __launch_bounds__(kSumThreads) k_sum_slices(const __grid_constant__ SumSet s) {
  const SumJob& j = s.job[blockIdx.y];
  const int64_t b0 = (int64_t)blockIdx.x * kSumSlice;
  if (b0 >= j.n && blockIdx.x > 0) return;
  const double r = block_sum<kSumThreads>(j.v, b0, min(b0 + kSumSlice, j.n));
  if (threadIdx.x == 0) j.partial[blockIdx.x] = r;
}
__global__ void __launch_bounds__(256) k_sum_totals(const __grid_constant__ SumSet s) {
  const SumJob& j = s.job[blockIdx.x];
  const int64_t slices = j.n > 0 ? (j.n + kSumSlice - 1) / kSumSlice : 1;
  const double r = block_sum<256>(j.partial, 0, slices);
  if (threadIdx.x == 0) *j.result = r;
}

// ----------------------------------------------------------------- LSCV

// Gd = 2 cell^2 F; per-block partial sums of F^2 (FP64).
__global__ void k_lscv_grid(const float* __restrict__ F, int64_t cells, double two_cell2,
                            double* __restrict__ G, double* __restrict__ sq_part) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < cells;
       q += (int64_t)gridDim.x * blockDim.x) {
    const float f = F[q];
    if (G) G[q] = two_cell2 * f;
    acc += (double)f * f;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) sq_part[blockIdx.x] = sh[0];
}

// exp(-c^2 t^2 / 2) for 0 <= t <= 1, c the cell in bandwidths: a polynomial in
// t^2 (the series of exp, cut where its terms fall below 2^-56), with the
// coefficients set on the host; for narrow bandwidths (many terms) the exp()
// of the library.
constexpr int kMaxTerms = 14;
struct CellGauss {
  double c[kMaxTerms];  // (-c^2/2)^k / k!
  double a;             // -c^2/2
  int terms;            // 0: use exp()
};
__device__ __forceinline__ double cell_gauss(double t, const CellGauss& g) {
  const double z = t * t;
  if (g.terms == 0) return exp(g.a * z);
  double r = g.c[g.terms - 1];
  for (int k = g.terms - 2; k >= 0; --k) r = fma(r, z, g.c[k]);
  return r;
}

// One axis of a point's own term at its two neighbouring cell centres (offsets
// -t and 1 - t cells; k0, k1: 1 where that cell is in the grid): with weights
// 1 - t and t, factors e and offsets d in bandwidths,
//   p = sum w e,  q = sum w e d^2,  dp = d p / d x (in bandwidths: weights' and
//   factors' slopes, sum (+-e / c + w e d)).
struct AxisTerm {
  double p, q, dp;
};
__device__ __forceinline__ AxisTerm axis_term(double t, double k0, double k1, double c, double inv_c,
                                              const CellGauss& g) {
  const double u = 1.0 - t;
  const double e0 = k0 * cell_gauss(t, g), e1 = k1 * cell_gauss(u, g);
  const double d0 = -c * t, d1 = c * u;
  const double a0 = u * e0, a1 = t * e1;
  const double b0 = a0 * d0, b1 = a1 * d1;
  AxisTerm r;
  r.p = a0 + a1;
  r.q = fma(b0, d0, b1 * d1);
  r.dp = fma(e1 - e0, inv_c, b0 + b1);
  return r;
}

// Per point: the leave-one-out term w_p bilerp(F - F_p, x_p) (the bilinear
// sample of F between cell centres, zero outside, minus the same sample of
// the point's own term F_p = w_p S, S = exp(-r^2/2h^2)/(2 pi N h^2)), the
// loss's direct partials (through the bilinear weights, w_p and F_p), and the
// scatter of -(2/N) w_p beta into the FP64 cotangent (atomic adds; in FP64
// their order does not show in the FP32 result).  FP64 throughout, which
// bounds it (16 SM cycles per warp instruction): S and the bilinear weights
// are products over the axes, so the sums over the four cells are products of
// two-cell sums, and the four exponentials are values of one polynomial.
// 1.47M points: 655 us with the four cells one by one, 368 now.
__global__ void __launch_bounds__(256)
    k_lscv_points(const float4* __restrict__ pts, const float* __restrict__ wts, int64_t n,
                  const float* __restrict__ F, int nx, int ny, double cells_per_h, double cell_h,
                  double inv_cell, double inv_h, double inv_N, double self_term,
                  const __grid_constant__ CellGauss cg, double* __restrict__ G,
                  float* __restrict__ gw_direct, float* __restrict__ gxy_direct,
                  double* __restrict__ loo, double* __restrict__ hdir) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
    const float4 P = pts[p];
    const double w = wts[p];
    const double fx = fma((double)P.x + (double)P.y, cells_per_h, -0.5);  // in cells
    const double fy = fma((double)P.z + (double)P.w, cells_per_h, -0.5);
    const double fi = floor(fx), fj = floor(fy);
    const double ax = fx - fi, ay = fy - fj;
    // the cell in 32 bits: far outside either way gives cells outside the grid
    const int i = (int)fmin(fmax(fi, -2.0), (double)nx);
    const int j = (int)fmin(fmax(fj, -2.0), (double)ny);
    const bool x0 = i >= 0 && i < nx, x1 = i >= -1 && i < nx - 1;
    const bool y0 = j >= 0 && j < ny, y1 = j >= -1 && j < ny - 1;
    const int64_t q = (int64_t)j * nx + i;
    const double f00 = x0 && y0 ? F[q] : 0.f, f10 = x1 && y0 ? F[q + 1] : 0.f;
    const double f01 = x0 && y1 ? F[q + nx] : 0.f, f11 = x1 && y1 ? F[q + nx + 1] : 0.f;
    const double g0 = f10 - f00, g1 = f11 - f01;
    const double r0 = fma(ax, g0, f00), r1 = fma(ax, g1, f01);
    const double v = fma(ay, r1 - r0, r0);
    const double dvx = fma(ay, g1 - g0, g0), dvy = r1 - r0;  // times 1 / cell
    const AxisTerm X = axis_term(ax, x0 ? 1.0 : 0.0, x1 ? 1.0 : 0.0, cell_h, cells_per_h, cg);
    const AxisTerm Y = axis_term(ay, y0 ? 1.0 : 0.0, y1 ? 1.0 : 0.0, cell_h, cells_per_h, cg);
    const double sv = self_term * X.p * Y.p;
    if (G) {
      const double k = -2.0 * inv_N * w;
      const double k0 = k * (1.0 - ay), k1 = k * ay;
      if (x0 && y0) atomicAdd(&G[q], k0 * (1.0 - ax));
      if (x1 && y0) atomicAdd(&G[q + 1], k0 * ax);
      if (x0 && y1) atomicAdd(&G[q + nx], k1 * (1.0 - ax));
      if (x1 && y1) atomicAdd(&G[q + nx + 1], k1 * ax);
    }
    if (gw_direct) gw_direct[p] = (float)(-2.0 * inv_N * (v - 2.0 * w * sv));
    if (gxy_direct) {
      const double ws = w * self_term * inv_h;
      gxy_direct[2 * p] = (float)(-2.0 * inv_N * w * fma(-ws * X.dp, Y.p, dvx * inv_cell));
      gxy_direct[2 * p + 1] = (float)(-2.0 * inv_N * w * fma(-ws * Y.dp, X.p, dvy * inv_cell));
    }
    loo[p] = w * (v - w * sv);
    hdir[p] = w * w * inv_h * self_term * (fma(X.q, Y.p, X.p * Y.q) - 2.0 * X.p * Y.p);
  }
}

__global__ void k_to_float(const double* __restrict__ src, int64_t n, float* __restrict__ dst) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride)
    dst[q] = (float)src[q];
}

int grid_blocks(int64_t n, int threads, int cap) {
  const int64_t b = (n + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, cap));
}

}  // namespace

size_t sum_partials(int64_t n) { return (size_t)((n + kSumSlice - 1) / kSumSlice) + 1; }

cudaError_t launch_sums(const SumJob* jobs, int count, cudaStream_t s) {
  if (count < 1 || count > kMaxSums) return cudaErrorInvalidValue;
  SumSet set = {};
  int64_t most = 1;
  for (int k = 0; k < count; ++k) {
    set.job[k] = jobs[k];
    most = std::max<int64_t>(most, (jobs[k].n + kSumSlice - 1) / kSumSlice);
  }
  k_sum_slices<<<dim3((unsigned)most, count), kSumThreads, 0, s>>>(set);
  k_sum_totals<<<count, 256, 0, s>>>(set);
  note_launches(2);
  return cudaGetLastError();
}

namespace {

struct AdjWindow {  // what the one-point kernel's launches share
  int R, cols, sub_log2;
  float c, inv_h;
};
AdjWindow adj_window(int64_t n, double cell, double h) {
  AdjWindow w = {};
  w.R = (int)ceil(8.0 * h / cell) + 1;
  const int width = 2 * w.R + 1;
  w.cols = width <= 32 ? 1 : width <= 64 ? 2 : width <= 128 ? 4 : 8;
  while ((1 << w.sub_log2) < width && w.sub_log2 < 5) ++w.sub_log2;
  if (w.cols > 1) w.sub_log2 = 5;
  w.c = (float)(1.0 / (2.0 * 3.14159265358979323846 * (double)n * h * h));
  w.inv_h = (float)(1.0 / h);
  return w;
}

}  // namespace

cudaError_t launch_adjoint_gauss(const float4* pts, const float* wts, int64_t n, const float* G,
                                 const float2* gxt, const float2* gyt, int nx, int ny,
                                 double cell, double h, float* grad_xy, float* grad_w,
                                 double* hterm, double* lterm, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const AdjWindow w = adj_window(n, cell, h);
  const int blocks = grid_blocks((n + 31) / 32 * 32, 256, 152 * 64);  // a warp per 32 points
#define KDE_ADJ(C)                                                                             \
  k_adjoint_gauss<C, false><<<blocks, 256, 0, s>>>(pts, wts, n, nullptr, nullptr, 1, nullptr,   \
                                                   G, gxt, gyt, nx, ny, cell / h, w.R,          \
                                                   w.sub_log2, w.c, w.inv_h, grad_xy, grad_w,  \
                                                   hterm, lterm)
  if (w.cols == 1) KDE_ADJ(1);
  else if (w.cols == 2) KDE_ADJ(2);
  else if (w.cols == 4) KDE_ADJ(4);
  else KDE_ADJ(8);
#undef KDE_ADJ
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_listed(const AdjGroupArgs& a, double cell, double h, cudaStream_t s) {
  const AdjWindow w = adj_window(a.n, cell, h);
  // the groups' windows end at 44 cells to either side, so no 8 columns per lane
  if (w.cols > 4) return cudaErrorInvalidValue;
  const int resident = (w.cols == 1 ? 5 : w.cols == 2 ? 4 : 3) * a.sms;  // launch bounds
  const int blocks = std::max(resident, grid_blocks((a.n + 31) / 32 * 32, 256, 152 * 64));
#define KDE_ADJ(C)                                                                             \
  k_adjoint_gauss<C, true><<<blocks, 256, 0, s>>>(a.pts, a.wts, a.n, a.singles, a.counters + 2, \
                                                  8 * resident, a.vals, a.G, a.gxt, a.gyt, a.nx, a.ny,       \
                                                  cell / h, w.R, w.sub_log2, w.c, w.inv_h,     \
                                                  a.grad_xy, a.grad_w, a.hterm, a.lterm)
  if (w.cols == 1) KDE_ADJ(1);
  else if (w.cols == 2) KDE_ADJ(2);
  else KDE_ADJ(4);
#undef KDE_ADJ
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_lscv(const float4* pts, const float* wts, int64_t n, const float* F, int nx,
                        int ny, double cell, double h, double* Gd, float* G, float* gw_direct,
                        float* gxy_direct, double* sq_part, int sq_blocks, double* loo,
                        double* hdir, cudaStream_t s) {
  const int64_t cells = (int64_t)nx * ny;
  k_lscv_grid<<<sq_blocks, 256, 0, s>>>(F, cells, 2.0 * cell * cell, Gd, sq_part);
  note_launches(1);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (n > 0) {
    const double self = 1.0 / (2.0 * 3.14159265358979323846) / ((double)n * h * h);
    CellGauss cg = {};
    cg.a = -0.5 * (cell / h) * (cell / h);
    double term = 1.0;
    int k = 0;
    for (; k < kMaxTerms && fabs(term) >= 0x1p-56; ++k) {
      cg.c[k] = term;
      term *= cg.a / (k + 1);
    }
    cg.terms = fabs(term) < 0x1p-56 ? k : 0;
    k_lscv_points<<<grid_blocks(n, 256, 152 * 16), 256, 0, s>>>(
        pts, wts, n, F, nx, ny, h / cell, cell / h, 1.0 / cell, 1.0 / h, 1.0 / (double)n, self,
        cg, Gd, gw_direct, gxy_direct, loo, hdir);
    note_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (G) {
    k_to_float<<<grid_blocks(cells, 256, 152 * 16), 256, 0, s>>>(Gd, cells, G);
    note_launches(1);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace kde
