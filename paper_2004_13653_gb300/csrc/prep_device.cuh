// A point's projection, centring, scaling and split into two FP32 numbers per
// coordinate (device side), shared by the kernels that prepare points.
#pragma once
#include "kde_internal.cuh"

namespace kde {

constexpr double kPi = 3.14159265358979323846;

// Eq. 1-4: x = lambda r0, y = q r0 with the isometric latitude q.  Near the
// standard latitude phi0 (|phi - phi0| <= m.range) y comes from the
// Taylor series of q about phi0: the constant, linear and quadratic terms in
// FP64, the terms of order 3..7 (a few metres at most) in FP32.  Elsewhere the
// closed form is evaluated in FP64.  GB300's FP64 rate makes the closed form
// (two logarithms, a tangent and a sine per point) the slow part.
// MercParams: kx = r0 pi/180; y0 = r0 q(phi0); c_k = r0 q^(k)(phi0)/k!
// (c[] holds c3 .. c7); range: |phi - phi0| up to which the series is used.

__device__ __forceinline__ double2 mercator_xy(double2 ll, const MercParams& m) {
  const double phi = ll.y * (kPi / 180.0);
  const double d = phi - m.phi0;
  double y;
  if (fabs(d) <= m.range) {
    const float df = (float)d;
    float t = m.c[4];
    t = fmaf(t, df, m.c[3]);
    t = fmaf(t, df, m.c[2]);
    t = fmaf(t, df, m.c[1]);
    t = fmaf(t, df, m.c[0]);
    y = fma(m.c2, d * d, fma(m.c1, d, m.y0)) + (double)(t * (df * df * df));
  } else {
    const double es = m.e * sin(phi);
    const double q = log(tan(0.25 * kPi + 0.5 * phi)) + 0.5 * m.e * log((1.0 - es) / (1.0 + es));
    y = q * m.r0;
  }
  return make_double2(ll.x * m.kx, y);
}

__device__ __forceinline__ float2 split_hi_lo(double v) {
  const float hi = __double2float_rn(v);
  const float lo = __double2float_rn(v - (double)hi);
  return make_float2(hi, lo);
}

__device__ __forceinline__ bool finite_bits(double v) {
  return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}
// v is zero or between 2^-60 and 2^100: split_bits and products with a scale
// of 2^-60 .. 2^27 then neither overflow nor lose bits to underflow
__device__ __forceinline__ bool plain_range(double v) {
  const unsigned h = (unsigned)__double2hiint(v) & 0x7fffffffu;
  return (h >> 20) - 963u < 160u || (h | (unsigned)__double2loint(v)) == 0u;
}

// (x, y) + (z, w), both sums of two FP32 numbers, within a few 2^-47 of the
// larger
__device__ __forceinline__ float2 add_pairs(float2 a, float2 b) {
  const float s = a.x + b.x, bb = s - a.x;
  const float e = ((a.x - (s - bb)) + (b.x - bb)) + (a.y + b.y);
  const float hi = s + e;
  return make_float2(hi, e - (hi - s));
}
// the product, within 2^-46 of it
__device__ __forceinline__ float2 mul_pairs(float2 a, float2 b) {
  const float p = a.x * b.x;
  const float e = fmaf(a.x, b.x, -p) + fmaf(a.x, b.y, a.y * b.x);
  const float hi = p + e;
  return make_float2(hi, e - (hi - p));
}

// Any point, in FP64 but for the split; a NaN in x: not finite.
static __device__ __noinline__ float4 prepare_any(double2 v, const PrepInst& I) {
  const double2 m = I.lonlat ? mercator_xy(v, I.merc) : v;
  const double x = (m.x - I.ox) * I.sigma, y = (m.y - I.oy) * I.sigma;
  const float2 X = split_hi_lo(x), Y = split_hi_lo(y);
  return make_float4(finite_bits(x) && finite_bits(y) ? X.x : __uint_as_float(0x7fffffffu), X.y,
                     Y.x, Y.y);
}

// The usual points: metres, and (lon, lat) near the standard latitude.  The
// FP64 pipe takes 16 cycles of an SM per warp instruction, so what needs
// FP64's 53 bits (the differences of projected coordinates, and the constant
// and linear terms of the projection with the centring and scaling in them)
// stays there, two or three operations a point, and the rest runs on pairs of
// FP32 numbers, whose 2^-46 is far below the 2^-24 of every use of the result on
// the grids that set_scale lets in.
// False: prepare_any decides.
__device__ __forceinline__ bool prepare_usual(double2 v, const PrepInst& I, float4& r) {
  float2 X, Y;
  if (!I.lonlat) {
    const double x = v.x - I.ox, y = v.y - I.oy;
    if (!(plain_range(x) && plain_range(y))) return false;
    X = mul_pairs(split_bits(x), I.sigma2);
    Y = mul_pairs(split_bits(y), I.sigma2);
  } else {
    // Eq. 1-4 as in mercator_xy: the quadratic term is a few hundred metres,
    // the terms beyond it a few
    const MercParams& m = I.merc;
    const double dd = fma(v.y, kPi / 180.0, -m.phi0);
    const double x = fma(v.x, I.lon_scale, I.lon_off), y = fma(dd, I.lat_scale, I.lat_off);
    if (!(plain_range(dd) && plain_range(x) && plain_range(y))) return false;
    const float2 d = split_bits(dd);
    if (!(fabsf(d.x) <= I.range_f)) return false;
    X = split_bits(x);
    float t = m.c[4];
    t = fmaf(t, d.x, m.c[3]);
    t = fmaf(t, d.x, m.c[2]);
    t = fmaf(t, d.x, m.c[1]);
    t = fmaf(t, d.x, m.c[0]);
    const float sq = d.x * d.x;
    const float sq_lo = fmaf(d.x, d.x, -sq) + 2.f * d.x * d.y;
    float2 q = mul_pairs(make_float2(sq, sq_lo), I.lat_q);
    q.y = fmaf(t * I.sigma2.x, d.x * sq, q.y);
    Y = add_pairs(split_bits(y), q);
  }
  r = make_float4(X.x, X.y, Y.x, Y.y);
  return true;
}

}  // namespace kde
