// Small Gaussian densities in one launch.
//
// A few thousand fixes on a small grid take a microsecond or two of arithmetic;
// the general path spends four launches on them (tables, centring, contraction,
// reduction).  Here a cluster of up to eight CTAs owns 16 x 16 cells; its warps
// take the points 32 at a time, one per lane: each lane centres its point (the
// arithmetic of the prepare kernel, from the caller's points), the warp
// tabulates the 16 x- and 16 y-factors of its points in shared memory and adds
// the outer products, eight cells per lane, into (hi, lo) sums.  The sums of
// the CTA's eight warps and of the cluster's CTAs are added in a fixed order,
// through distributed shared memory, so there is nothing to reduce afterwards
// and results are reproducible bit for bit.  FP32 factors and sums, as the SIMT
// path.  2000 points x 64^2: four launches, 18 us of GPU time and 30 us per
// call on the general path, 6 and 20 us (the host's part) in this form.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "kde_internal.cuh"
#include "kernel_factors.cuh"
#include "prep_device.cuh"

namespace kde {
namespace {

namespace cg = cooperative_groups;

constexpr int kTile = 16;   // cells of a tile's side
constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;

struct WarpTables {
  float kx[32][kTile];
  float ky[32][kTile];
};

__global__ void __launch_bounds__(kThreads)
    k_small_gauss(const __grid_constant__ PrepInst I, float scale, float post, int tiles_x,
                  float* __restrict__ out, CallScalars* __restrict__ scal) {
  __shared__ __align__(16) WarpTables tables[kWarps];
  __shared__ float2 part[kWarps][8][32];
  __shared__ float2 total[kTile * kTile];
  __shared__ float2 centre[2 * kTile];
  cg::cluster_group cluster = cg::this_cluster();
  const int ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tile = blockIdx.x / ranks;
  const int x0 = (tile % tiles_x) * kTile, y0 = (tile / tiles_x) * kTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WarpTables& T = tables[warp];
  // the lane's table column: cell ej of the tile along either axis
  const int ej = lane & (kTile - 1), half = lane >> 4;
  // cell centres, x then y: FP64, so one warp finds them
  if (warp == 0) {
    const int c = half ? min(y0 + ej, I.ny - 1) : min(x0 + ej, I.nx - 1);
    centre[lane] = split_double(((double)c + 0.5) * I.cell_sigma);
  }
  __syncthreads();
  const float2 gx = centre[ej], gy = centre[kTile + ej];
  const int cx = 2 * (lane & 7), cy = 4 * (lane >> 3);  // the lane's 2 x 4 cells
  float2 run[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) run[r] = make_float2(0.f, 0.f);
  for (int64_t b = (int64_t)(rank * kWarps + warp) * 32; b < I.n;
       b += (int64_t)ranks * kWarps * 32) {
    const int64_t p = b + lane;
    float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
    float w = 0.f;
    if (p < I.n) {
      const double2 v = reinterpret_cast<const double2*>(I.xy)[p];
      // the density's scale goes into the weights, but for a power of two that
      // leaves what goes in below 2^-14: no weight and no sum overflows then
      // (n <= 2^14), only a result that does
      const float wv = I.w ? I.w[p] : 1.0f;
      w = wv * scale;
      if (!(I.usual && prepare_usual(v, I, P))) P = prepare_any(v, I);
      if (P.x != P.x || !isfinite(wv)) {
        P = make_float4(0.f, 0.f, 0.f, 0.f);
        w = 0.f;
        if (scal) atomicOr(&scal->err, kErrNonFinite);
      }
    }
    __syncwarp();  // the last batch's tables are read
    // the half-warps take alternate points: rows of 16 floats, no bank conflicts
#pragma unroll 8
    for (int k = 0; k < 16; ++k) {
      const int c = 2 * k + half;
      const float px = __shfl_sync(0xffffffffu, P.x, c), pxl = __shfl_sync(0xffffffffu, P.y, c);
      const float py = __shfl_sync(0xffffffffu, P.z, c), pyl = __shfl_sync(0xffffffffu, P.w, c);
      const float pw = __shfl_sync(0xffffffffu, w, c);
      T.kx[c][ej] = kfactor<KDE_GAUSSIAN>((gx.x - px) + (gx.y - pxl));
      T.ky[c][ej] = pw * kfactor<KDE_GAUSSIAN>((gy.x - py) + (gy.y - pyl));
    }
    __syncwarp();
    float acc[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = 0.f;
#pragma unroll 8
    for (int c = 0; c < 32; ++c) {
      const float2 kx = *reinterpret_cast<const float2*>(&T.kx[c][cx]);
      const float4 ky = *reinterpret_cast<const float4*>(&T.ky[c][cy]);
      const float y[4] = {ky.x, ky.y, ky.z, ky.w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        acc[2 * r] = fmaf(kx.x, y[r], acc[2 * r]);
        acc[2 * r + 1] = fmaf(kx.y, y[r], acc[2 * r + 1]);
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) two_sum_acc(run[r], acc[r]);
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) part[warp][r][lane] = run[r];
  __syncthreads();
  // warp r adds cell r of every lane's eight over the warps
  float2 sum = part[0][warp][lane];
#pragma unroll
  for (int h = 1; h < kWarps; ++h) {
    const float2 o = part[h][warp][lane];
    two_sum_acc(sum, o.x);
    sum.y += o.y;
  }
  if (ranks > 1) {
    total[threadIdx.x] = sum;
    cluster.sync();
    if (rank == 0)
      for (int h = 1; h < ranks; ++h) {
        const float2 o = cluster.map_shared_rank(total, h)[threadIdx.x];
        two_sum_acc(sum, o.x);
        sum.y += o.y;
      }
    cluster.sync();  // no CTA leaves while its sums are read
  }
  if (rank == 0) {
    const int x = x0 + cx + (warp & 1), y = y0 + cy + (warp >> 1);
    if (x < I.nx && y < I.ny) out[(int64_t)y * I.nx + x] = (sum.x + sum.y) * post;
  }
}

}  // namespace

// GPU time, small against general form: 500 points x 128^2 4.8 / 17.8 us,
// 2000 x 200^2 (8e7 pairs) 17.7 / 19.5, 8000 x 128^2 (1.3e8) 22.7 / 21.6, 16000 x
// 64^2 (6.6e7) 22.1 / 24.7, 32000 x 64^2 40 / 31: the line lies where the two
// meet.  What the kernel computes are whole 16 x 16 tiles, so thin grids have a
// line of their own, by the tiles' pairs (1 x 3600: 1.2e8 of them 17.5 / 22.4, 2.3e8
// 31.5 / 28.2, 9.4e8 113 / 67), and so have grids of few points, by the tiles, each
// of which costs a CTA's start (1 point x 1024^2, 4096 tiles 17.7 / 20.9, x 1500^2
// 36 / 25, x 2048^2 64 / 21).
bool small_gauss_fits(int64_t n, int nx, int ny) {
  const double tiles = (double)((nx + kTile - 1) / kTile) * ((ny + kTile - 1) / kTile);
  return n >= 1 && n <= 16384 && (double)n * nx * ny <= 6e7 && tiles <= 4096.0 &&
         (double)n * tiles * (kTile * kTile) <= 1.5e8;
}

cudaError_t launch_small_gauss(const PrepInst& q, double scale, float* out, CallScalars* scal,
                               int sms, cudaStream_t s) {
  int e2 = 0;
  frexp(scale, &e2);  // scale < 2^e2
  const int post2 = std::max(0, std::min(e2 + 14, 127));
  const int tx = (q.nx + kTile - 1) / kTile, ty = (q.ny + kTile - 1) / kTile;
  const int64_t tiles = (int64_t)tx * ty;
  // clusters as large as leave every warp a batch, up to eight CTAs
  int ranks = 1;
  while (ranks < 8 && (int64_t)ranks * kWarps * 32 < q.n && 2 * ranks * tiles <= 4 * (int64_t)sms)
    ranks *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * ranks));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ranks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_small_gauss, q, (float)ldexp(scale, -post2),
                                           ldexpf(1.0f, post2), tx, out, scal);
  note_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace kde
