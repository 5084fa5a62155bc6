// Steps before the density sum: the Mercator projection (Sec. III-A, Eq. 1-4)
// and the centring of the points and cell centres against the grid origin
// (the x - x_min of Eq. 5-6), both in FP64, followed by the split of each
// centred, scaled coordinate into two FP32 numbers hi + lo.  These are the
// only FP64 steps of the library: the projected coordinates are ~1e7 m and
// their differences must be resolved to millimetres.
#include <string.h>

#include <algorithm>
#include <mutex>

#include "kde_internal.cuh"
#include "prep_device.cuh"

namespace kde {
namespace {

constexpr double kWgs84A = 6378137.0;
constexpr double kWgs84E2 = 0.00669437999014;

__global__ void k_mercator(const double* __restrict__ lonlat, int64_t n,
                           const __grid_constant__ MercParams m, double* __restrict__ xy) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride)
    reinterpret_cast<double2*>(xy)[p] =
        mercator_xy(reinterpret_cast<const double2*>(lonlat)[p], m);
}

// Truncated power series in d (order kOrd) on the host.
constexpr int kOrd = 8;
struct Series {
  double a[kOrd + 1];
};
Series series_mul(const Series& x, const Series& y) {
  Series r = {};
  for (int i = 0; i <= kOrd; ++i)
    for (int j = 0; i + j <= kOrd; ++j) r.a[i + j] += x.a[i] * y.a[j];
  return r;
}
Series series_recip(const Series& x) {  // x.a[0] != 0
  Series r = {};
  r.a[0] = 1.0 / x.a[0];
  for (int k = 1; k <= kOrd; ++k) {
    double s = 0.0;
    for (int j = 1; j <= k; ++j) s += x.a[j] * r.a[k - j];
    r.a[k] = -s / x.a[0];
  }
  return r;
}

// Taylor coefficients of q(phi0 + d) - q(phi0) from
// q'(phi) = (1 - e^2) / ((1 - e^2 sin^2 phi) cos phi), integrated term by term.
MercParams mercator_series(double phi0, double r0, double e2) {
  Series sd = {}, cd = {};  // sin d, cos d
  double f = 1.0;
  for (int k = 0; k <= kOrd; ++k) {
    if (k > 0) f /= k;
    const double v = f * ((k / 2) % 2 ? -1.0 : 1.0);
    if (k % 2) sd.a[k] = v; else cd.a[k] = v;
  }
  Series sn = {}, cs = {};  // sin(phi0 + d), cos(phi0 + d)
  for (int k = 0; k <= kOrd; ++k) {
    sn.a[k] = sin(phi0) * cd.a[k] + cos(phi0) * sd.a[k];
    cs.a[k] = cos(phi0) * cd.a[k] - sin(phi0) * sd.a[k];
  }
  Series den = series_mul(sn, sn);
  for (int k = 0; k <= kOrd; ++k) den.a[k] = (k == 0 ? 1.0 : 0.0) - e2 * den.a[k];
  den = series_mul(den, cs);
  const Series qp = series_recip(den);  // q'/(1 - e^2)
  MercParams m;
  const double e = sqrt(e2);
  const double s0 = sin(phi0);
  m.r0 = r0;
  m.kx = r0 * (kPi / 180.0);
  m.phi0 = phi0;
  m.y0 = r0 * (log(tan(0.25 * kPi + 0.5 * phi0)) + 0.5 * e * log((1.0 - e * s0) / (1.0 + e * s0)));
  m.c1 = r0 * (1.0 - e2) * qp.a[0];
  m.c2 = r0 * (1.0 - e2) * qp.a[1] / 2.0;
  for (int k = 3; k <= 7; ++k) m.c[k - 3] = (float)(r0 * (1.0 - e2) * qp.a[k - 1] / k);
  // range: the FP32 rounding of the order-3 term plus the first omitted term
  // stay below 2e-7 m (at most 0.01 rad, ~64 km of latitude)
  const double c3 = fabs(r0 * (1.0 - e2) * qp.a[2] / 3), c8 = fabs(r0 * (1.0 - e2) * qp.a[7] / 8);
  m.range = 0.01;
  while (m.range > 1e-4 && c3 * pow(m.range, 3) * 1.2e-7 + c8 * pow(m.range, 8) > 2e-7)
    m.range *= 0.9;
  m.e = e;
  return m;
}

// Instance of flattened index p: the last entry whose begin <= p.
template <class T>
__device__ __forceinline__ int find_instance(const T* tab, int ninst, int64_t p) {
  int lo = 0, hi = ninst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].begin <= p) lo = mid; else hi = mid - 1;
  }
  return lo;
}

constexpr int kPerWarp = 64;  // divides every instance's n_pad

// Centre, scale, split; weights copied (unit when w == NULL); padding zeroed;
// max |w| reduced per instance for the tensor path's operand scaling.  Every
// instance's n_pad is a multiple of 512, so a warp's points never straddle two.  The
// blocks from table_block on fill the cell-centre tables (one launch for
// both).  1M points: 29.6 us with every step in FP64, 13 now (HBM: 6 us);
// 20M (lon, lat) points: 0.897 -> 0.160 ms (HBM: 0.12 ms).  A warp keeps its
// maximum over all its points and skips the atomic when it would not change
// anything.
__global__ void __launch_bounds__(256)
    k_prepare(const PrepInst* __restrict__ tab, int ninst, int64_t total, int table_block,
              int blocks_per_side) {
  if ((int)blockIdx.x >= table_block) {
    const int b = (int)blockIdx.x - table_block;
    const PrepInst& I = tab[b / blocks_per_side];
    const int64_t stride = (int64_t)blocks_per_side * blockDim.x;
    for (int64_t t = (int64_t)(b % blocks_per_side) * blockDim.x + threadIdx.x;
         t < max(I.nx, I.ny); t += stride) {
      const float2 c = split_hi_lo(((double)t + 0.5) * I.cell_sigma);
      if (t < I.nx) I.gxt[t] = c;
      if (t < I.ny) I.gyt[t] = c;
    }
    return;
  }
  // A warp takes kPerWarp consecutive points at a time, all of one instance,
  // and has their loads in flight together.
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)table_block * (blockDim.x >> 5);
  unsigned wmax = 0;
  bool bad = false, neg = false;
  const PrepInst* cur = nullptr;
  auto flush = [&]() {
    const unsigned top = __reduce_max_sync(0xffffffffu, wmax);
    const unsigned anybad = __any_sync(0xffffffffu, bad), anyneg = __any_sync(0xffffffffu, neg);
    if (lane == 0) {
      if (top > *(volatile unsigned*)&cur->scal->wmax_bits) atomicMax(&cur->scal->wmax_bits, top);
      if (anybad) atomicOr(&cur->scal->err, kErrNonFinite);
      if (anyneg) atomicOr(&cur->scal->negw, 1);
    }
    wmax = 0;
    bad = neg = false;
  };
  for (int64_t g0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kPerWarp;
       g0 < total; g0 += warps * kPerWarp) {
    const PrepInst* ip = tab + (ninst > 1 ? find_instance(tab, ninst, g0) : 0);
    if (ip != cur) {
      if (cur) flush();
      cur = ip;
    }
    const PrepInst& I = *ip;
    const int64_t p0 = g0 - I.begin + lane;
    double2 v[kPerWarp / 32];
    float w[kPerWarp / 32];
#pragma unroll
    for (int u = 0; u < kPerWarp / 32; ++u) {
      const int64_t p = p0 + 32 * u;
      v[u] = p < I.n ? reinterpret_cast<const double2*>(I.xy)[p] : make_double2(0.0, 0.0);
      w[u] = p < I.n ? (I.w ? I.w[p] : 1.0f) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kPerWarp / 32; ++u) {
      const int64_t p = p0 + 32 * u;
      float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
      if (p < I.n) {
        if (!(I.usual && prepare_usual(v[u], I, r))) r = prepare_any(v[u], I);
        if (!(r.x != r.x) && isfinite(w[u])) {
          wmax = max(wmax, __float_as_uint(fabsf(w[u])));
        } else {
          bad = true;
          r = make_float4(0.f, 0.f, 0.f, 0.f);
          w[u] = 0.f;
        }
      }
      I.pts[p] = r;
      I.wts[p] = w[u];
      neg |= w[u] < 0.f;
    }
  }
  if (cur) flush();
}

// Table bytes carried by a launch's parameters; the small form keeps the
// parameters of the usual call (one instance) short.
constexpr int kBlobBytes = 31 * 1024, kSmallBlobBytes = 2 * 1024;
template <int BYTES>
struct __align__(16) Blob {
  unsigned char bytes[BYTES];
};

template <int BYTES>
__global__ void k_upload(const __grid_constant__ Blob<BYTES> blob, int nwords, uint4* dst) {
  for (int i = threadIdx.x; i < nwords; i += blockDim.x)
    dst[i] = reinterpret_cast<const uint4*>(blob.bytes)[i];
}

template <int BYTES>
cudaError_t upload_chunk(const unsigned char* src, size_t len, unsigned char* dst,
                         cudaStream_t s) {
  static Blob<BYTES> blob;  // staging for the launch parameters (copied at launch)
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  memcpy(blob.bytes, src, len);
  k_upload<BYTES><<<1, 256, 0, s>>>(blob, (int)(len / 16), reinterpret_cast<uint4*>(dst));
  note_launches(1);
  return cudaGetLastError();
}

int blocks_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 152 * 32) b = 152 * 32;
  return (int)b;
}

}  // namespace

MercParams mercator_params(double lat0_deg) {
  const double phi0 = lat0_deg * (kPi / 180.0);
  const double r0 = kWgs84A * cos(phi0) / sqrt(1.0 - kWgs84E2 * sin(phi0) * sin(phi0));
  return mercator_series(phi0, r0, kWgs84E2);
}

cudaError_t launch_mercator(const double* lonlat, int64_t n, double lat0_deg, double* xy,
                            cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const MercParams m = mercator_params(lat0_deg);
  k_mercator<<<blocks_for(n, 256), 256, 0, s>>>(lonlat, n, m, xy);
  note_launches(1);
  return cudaGetLastError();
}

namespace {
float2 pair_of(double v) {
  const float hi = (float)v;
  return make_float2(hi, (float)(v - (double)hi));
}
}  // namespace

void set_scale(PrepInst& q, int nx, int ny, double sigma, double cell, const MercParams* m) {
  q.nx = nx;
  q.ny = ny;
  q.sigma = sigma;
  q.cell_sigma = cell * sigma;
  // a scale outside the plain range sends every point to prepare_any: up to 2^27 the
  // product with a coordinate of the plain range (below 2^100) is an FP32 number.
  // The pairs' 2^-46 of a position is 2^-30 units or less over a grid of up to
  // 2^16 of them, far below the 2^-25 that FP32 leaves of an offset of one.  Beyond,
  // FP64 and its 2^-49 (3e7 cells at h = 0.3 cells, Epanechnikov: 2.7e-6 off with pairs, below 1.1e-6 now).
  const bool plain = sigma >= 0x1p-60 && sigma <= 0x1p27 &&
                     (double)std::max(nx, ny) * cell * sigma <= 0x1p16;
  q.usual = plain ? 1 : 0;
  q.sigma2 = plain ? pair_of(sigma) : make_float2(0.f, 0.f);
  q.lonlat = m ? 1 : 0;
  if (!m) return;
  q.merc = *m;
  q.lon_scale = m->kx * sigma;
  q.lon_off = -q.ox * sigma;
  q.lat_scale = m->c1 * sigma;
  q.lat_off = (m->y0 - q.oy) * sigma;
  q.lat_q = pair_of(m->c2 * sigma);
  q.range_f = (float)m->range;
}

cudaError_t launch_prepare(const PrepInst* tab, int ninst, int64_t total_pad, int max_side,
                           cudaStream_t s) {
  if (ninst <= 0) return cudaSuccess;
  // as many table blocks as fill the GPU, at least one an instance: a block for every
  // 256 cells of the longest side in every instance can be 2^31 of them
  const int per_side = std::max(1, std::min(blocks_for(max_side, 256), 152 * 32 / ninst));
  const int points = total_pad > 0 ? blocks_for(total_pad, 8 * kPerWarp) : 0;
  k_prepare<<<points + ninst * per_side, 256, 0, s>>>(tab, ninst, total_pad, points, per_side);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_upload(const void* bytes, size_t nbytes, void* dst, cudaStream_t s) {
  const unsigned char* src = static_cast<const unsigned char*>(bytes);
  unsigned char* to = static_cast<unsigned char*>(dst);
  if (nbytes % 16) return cudaErrorInvalidValue;
  for (size_t off = 0; off < nbytes; off += kBlobBytes) {
    const size_t len = std::min<size_t>(kBlobBytes, nbytes - off);
    const cudaError_t e = len <= kSmallBlobBytes
                              ? upload_chunk<kSmallBlobBytes>(src + off, len, to + off, s)
                              : upload_chunk<kBlobBytes>(src + off, len, to + off, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace kde
