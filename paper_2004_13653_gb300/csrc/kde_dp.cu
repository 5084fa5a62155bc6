// Douglas-Peucker compression of the trajectories (Sec. III-B), in the
// level-synchronous form of Sec. IV-A: every curve segment of every
// trajectory is processed in the same iteration, so the recursion of the
// textbook algorithm becomes a loop over tree levels.
//
// Each point carries the two ends (s, e) of the segment it lies in, which
// plays the part of the paper's label set Lp, and each segment's length
// |e - s| is kept at its start index.  Eq. 9's VED is |cross| / length, and for
// one segment the correctly rounded quotient never decreases when the cross
// product grows, so the steps work on the cross product and divide only where
// the result could depend on it.  One iteration:
//   1. ved   : the cross product of every open point with its segment; its
//              maximum per segment by a segmented max over each warp's lanes
//              and one 64-bit atomicMax per run (non-negative doubles order
//              like their bit patterns);
//   2. arg   : the segment's largest VED is the maximum cross product divided
//              by the length; the points whose cross product is within 1e-15
//              of the maximum (no other can tie after rounding) compute their
//              VED exactly, and the first one equal to that largest VED, if it
//              exceeds eps, is the split (atomicMin) -- the tie rule of the
//              sequential algorithm;
//   3. split : that point is kept and records the lengths of the two segments
//              it starts and ends; the others move their s or e to it (the
//              label update of Eq. 11); segments with nothing above eps are
//              closed.  The per-segment slots of the next iteration
//              (double-buffered) are cleared here.
// The loop ends when an iteration keeps no point.  All iterations run in one
// cooperative launch: the three steps are phases of a persistent kernel
// separated by grid-wide barriers, and the count of points kept in an
// iteration is read on the device, so no level costs a host round trip.
// Trajectories that fit in shared memory (the usual case) skip all of that:
// k_dp_local gives each a CTA, which runs the same levels on it alone (see the
// kernel).
// The VED is evaluated with
// explicitly rounded FP64 operations in the order of Eq. 9, so every
// comparison -- and therefore the kept set -- is identical to a sequential
// FP64 evaluation.  The kept points are then compacted: counts per block of
// points, the Sec. IV-A exclusive scan over the blocks, and each point's place
// in its block from ballots.
#include <cooperative_groups.h>
#include <float.h>

#include "kde_internal.cuh"

namespace kde {
namespace {

namespace cg = cooperative_groups;

constexpr uint8_t kKept = 1, kDone = 2;
constexpr uint32_t kNoArg = 0xffffffffu;

// |e - s|, rounded as Eq. 9 is evaluated
__device__ __forceinline__ double seg_len(double2 a, double2 b) {
  const double dx = __dsub_rn(b.x, a.x), dy = __dsub_rn(b.y, a.y);
  return __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
}
// The numerator of Eq. 9, |(p - s) x (e - s)| -- or, for a segment of zero
// length, the distance |p - s| itself (the VED then).
__device__ __forceinline__ double ved_num(double2 q, double2 a, double2 b, double len) {
  const double vx = __dsub_rn(q.x, a.x), vy = __dsub_rn(q.y, a.y);
  if (len == 0.0) return __dsqrt_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)));
  const double dx = __dsub_rn(b.x, a.x), dy = __dsub_rn(b.y, a.y);
  return fabs(__dsub_rn(__dmul_rn(vx, dy), __dmul_rn(vy, dx)));
}
// The VED from its numerator.
__device__ __forceinline__ double ved_of(double num, double len) {
  return len == 0.0 ? num : __ddiv_rn(num, len);
}

// Trajectory bounds of point p: the last k with off[k] <= p; bounds clamped to
// [0, n] so that malformed offsets cannot index outside the points.
__device__ __forceinline__ void traj_bounds(const int64_t* __restrict__ off, int64_t ntraj,
                                            int64_t n, int64_t p, int64_t& a, int64_t& b) {
  if (!off) {
    a = 0;
    b = n;
    return;
  }
  int64_t lo = 0, hi = ntraj - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= p) lo = mid; else hi = mid - 1;
  }
  a = min(max(off[lo], (int64_t)0), n);
  b = min(max(off[lo + 1], a), n);
}

// What the planning kernel decides; lives in the workspace, zeroed per call.
struct DpCtl {
  uint32_t n_local[2];  // trajectories on the work lists of k_dp_local: short, long ones
  uint32_t next[2];     // the next of them to take
  uint32_t n_long;      // trajectories left to the level kernel
  uint32_t irregular;   // the offsets do not rise: every point goes to the level kernel
};

// One thread per trajectory: those of 3..short_max points go on the first work
// list (two points or fewer have nothing to split), those of up to local_max
// on the second, filled from its end; longer ones are counted.  Trajectories
// of one or two points are finished here.
__global__ void k_dp_plan(const double2* __restrict__ xy, const int64_t* __restrict__ off,
                          int64_t ntraj, int64_t n, uint8_t* __restrict__ flag,
                          CallScalars* __restrict__ scal, int short_max, int local_max, DpCtl* __restrict__ ctl,
                          uint32_t* __restrict__ list,
                          uint32_t list_cap, int* __restrict__ iterations) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0) atomicMax(iterations, 1);
  int64_t a = 0, b = 0;
  if (k < ntraj) {
    a = off ? off[k] : 0;
    b = off ? off[k + 1] : n;
    if (a < 0 || b < a || b > n || (k == 0 && a != 0) || (k == ntraj - 1 && b != n))
      atomicOr(&ctl->irregular, 1u);
  }
  const int64_t len = b - a;
  if ((len == 1 || len == 2) && a >= 0 && b <= n)
    for (int64_t p = a; p < b; ++p) {
      const double2 q = xy[p];
      flag[p] = kKept;
      if (!(isfinite(q.x) && isfinite(q.y))) atomicOr(&scal->err, kErrNonFinite);
    }
  if (len > local_max) atomicAdd(&ctl->n_long, 1u);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const bool mine = len >= 3 && len <= local_max && (len > short_max) == (c == 1);
    const unsigned m = __ballot_sync(0xffffffffu, mine);
    uint32_t at = 0;
    if (lane == 0 && m) at = atomicAdd(&ctl->n_local[c], (uint32_t)__popc(m));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (mine && at < list_cap) list[c ? list_cap - 1 - at : at] = (uint32_t)k;
  }
}

// The level kernel's per-point and per-segment state, for the points it will
// process, and every point's flag; nothing to do when that kernel has no
// trajectory (k_dp_plan and k_dp_local then cover every point).
__global__ void k_dp_init(const double2* __restrict__ xy, int64_t n,
                          const int64_t* __restrict__ off, int64_t ntraj, int32_t* __restrict__ s,
                          int32_t* __restrict__ e, uint8_t* __restrict__ flag,
                          unsigned long long* __restrict__ segmax, uint32_t* __restrict__ segarg,
                          double* __restrict__ seglen, int local_max,
                          const DpCtl* __restrict__ ctl, CallScalars* __restrict__ scal) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const bool all = __ldg(&ctl->irregular) != 0u;
  if (!all && __ldg(&ctl->n_long) == 0u) return;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
    int64_t a, b;
    traj_bounds(off, ntraj, n, p, a, b);
    const double2 q = xy[p];
    bool bad = !(isfinite(q.x) && isfinite(q.y));
    if (!(a <= p && p < b)) {  // offsets do not cover p: a trajectory of its own
      bad = true;
      a = p;
      b = p + 1;
    }
    flag[p] = (p == a || p == b - 1 || bad) ? kKept : 0;
    if (bad) atomicOr(&scal->err, kErrNonFinite);
    if (!all && b - a <= local_max) continue;
    s[p] = (int32_t)a;
    e[p] = (int32_t)(b - 1);
    if (p == a) seglen[p] = seg_len(q, xy[b - 1]);
    segmax[p] = 0ull;
    segmax[n + p] = 0ull;
    segarg[p] = kNoArg;
    segarg[n + p] = kNoArg;
  }
  if (off && blockIdx.x == 0 && threadIdx.x == 0 && (off[0] != 0 || off[ntraj] != n))
    atomicOr(&scal->err, kErrBadArg);
}

// ------------------------------------------- whole trajectories in one CTA
//
// A trajectory in shared memory: its segments are worked off level by level,
// each by one warp (no grid-wide barriers, and a trajectory that is finished
// costs nothing while others go on); short trajectories have a CTA of one
// warp, so not even CTA-wide ones.  GB300 does 2
// FP64 operations per SM and clock, so the cross product of every open point
// at every level would still take most of the time; it is bracketed in FP32
// instead.  On coordinates relative to the trajectory's first point, as sums
// of two FP32 numbers (within u^2 R of the exact ones, |x| <= R, u = 2^-24),
// each difference is within 2 u |v| + 6 u^2 R of the exact one, and
// c = |vx dy - vy dx| within
//   E = 6 u (|vx dy| + |vy dx|) + 6 u^2 R (|vx| + |vy| + |dx| + |dy|) + 36 u^4 R^2
// of the FP64 evaluation (whose own roundings are far smaller); a third is
// added for the rounding of E itself and 1e-37 for underflow.  Only the points
// whose upper bound c + E reaches the segment's largest lower bound
// c - E, and eps times a lower bound of the segment's length, can be the split
// or tie with it.  Where that leaves one point and its lower bound exceeds eps
// times an upper bound of the length, it is the split; otherwise (about one
// segment in a hundred) the points left are evaluated in FP64, from the
// original coordinates and by the same steps as in the level kernel.  Either
// way the split is the one that kernel finds.
//
// Segments of at most kSmall points leave the levels: one thread finishes each
// (dp_finish), a warp's 32 at a time.
// Bound by instruction issue (per point and level about 50 instructions).
// 4000 tracks of 500 fixes at 10 m: 3.51 ms in the level kernel; here 2.08 ms
// with FP64 for every point left by the brackets, 0.38 ms with FP64 for the
// undecided segments only but a thread per point and CTA-wide phases, 0.20 ms
// with a warp per segment.
__device__ __forceinline__ float sqrt_approx(float v) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
constexpr int kSmall = 16;       // interior points of a segment that one thread finishes
constexpr int kLocalMax = 9728;  // points of a trajectory: 21.5 bytes each, 209 KB
// Shared memory for trajectories of up to m points (m a multiple of 128): the
// coordinates, two lists of at most m / 16 longer segments (each has more than
// kSmall interior points of its own), one of at most m / 2 small ones, the
// points' levels and states.
constexpr size_t dp_local_smem(int m) { return (size_t)m * 21 + (size_t)m / 2; }

// The FP32 bracket of a point's cross product with its segment, and of the
// segment's length.
struct DpBracket {
  float lo, hi;          // of c; lo = 0, hi = inf: to be evaluated in FP64
  float len_lo, len_hi;
};
// v0, A, B: (x hi, y hi, x lo, y lo); uR = 8 u^2 R
__device__ __forceinline__ DpBracket dp_bracket(float4 v0, float4 A, float4 B, float uR,
                                                float tiny) {
  constexpr float u = 0x1p-24f;
  const float vx = (v0.x - A.x) + (v0.z - A.z), vy = (v0.y - A.y) + (v0.w - A.w);
  const float dx = (B.x - A.x) + (B.z - A.z), dy = (B.y - A.y) + (B.w - A.w);
  const float t0 = vx * dy, t1 = vy * dx;
  const float c = fabsf(t0 - t1);
  const float E = fmaf(uR, (fabsf(vx) + fabsf(vy)) + (fabsf(dx) + fabsf(dy)),
                       fmaf(8.f * u, fabsf(t0) + fabsf(t1), tiny));
  DpBracket r;
  const float len = sqrt_approx(fmaf(dx, dx, dy * dy));
  r.len_lo = fmaf(len, 1.f - 1e-6f, -6.f * uR);
  r.len_hi = fmaf(len, 1.f + 1e-6f, fmaf(6.f, uR, 1e-18f));
  r.hi = (c + E) * (1.f + 1e-6f);
  // a segment that may have zero length is measured by distances, not by cross
  // products: all its points are evaluated, as where the bounds overflow
  const bool exact = !(r.len_lo > 0.f) || !(r.hi < FLT_MAX);
  r.lo = exact || !(c > E) ? 0.f : (c - E) * (1.f - 1e-6f);
  if (exact) r.hi = INFINITY;  // below no bound, an overflown one included
  return r;
}

// The split of segment (s, e) by FP64 alone, by one thread; -1: nothing above
// eps.
__device__ __noinline__ int dp_split_exact(const double2* __restrict__ P, int s, int e,
                                           double eps) {
  const double2 A = P[s], B = P[e];
  const double len = seg_len(A, B);
  double cmax = 0.0;
  for (int i = s + 1; i < e; ++i) {
    const double c = ved_num(P[i], A, B, len);
    if (c > cmax) cmax = c;
  }
  const double dmax = cmax == 0.0 ? 0.0 : ved_of(cmax, len);
  if (!(dmax > eps)) return -1;
  for (int i = s + 1; i < e; ++i) {
    const double c = ved_num(P[i], A, B, len);
    if (c >= __dmul_rn(cmax, 1.0 - 1e-15) && (c == cmax || ved_of(c, len) == dmax)) return i;
  }
  return -1;
}

// Finishes the segment (s0, e0) by one thread: from left to right, splitting
// the leftmost open segment until nothing in it is above eps.  lvl[k] is one
// more than the level at which point k was kept; a segment's level is the
// larger one of its ends'.  Returns the largest level + 2 of a split (what the
// level loop would have counted).
__device__ __forceinline__ int dp_finish(const double2* __restrict__ P,
                                         const float4* __restrict__ q, uint8_t* st, uint16_t* lvl,
                                         int s0, int e0, float uR, float tiny, float eps_lo,
                                         float eps_hi, double eps) {
  int s = s0, e = e0, most = 0;
  while (s < e0) {
    const float4 A = q[s], B = q[e];
    float best_lo = 0.f, top = -1.f, second = -1.f, len_lo = 0.f, len_hi = 0.f;
    int at = -1;
    for (int i = s + 1; i < e; ++i) {
      const DpBracket b = dp_bracket(q[i], A, B, uR, tiny);
      best_lo = fmaxf(best_lo, b.lo);
      if (b.hi > top) {
        second = top;
        top = b.hi;
        at = i;
      } else {
        second = fmaxf(second, b.hi);
      }
      len_lo = b.len_lo;
      len_hi = b.len_hi;
    }
    int k = -1;
    if (at >= 0 && !(top < eps_lo * len_lo))
      k = second < best_lo && best_lo > eps_hi * len_hi ? at : dp_split_exact(P, s, e, eps);
    if (k >= 0) {
      const int level = max((int)lvl[s], (int)lvl[e]);
      st[k] = kKept;
      lvl[k] = (uint16_t)(level + 1);
      most = max(most, level + 2);
      e = k;
    } else {
      for (int i = s + 1; i < e; ++i) st[i] = kDone;
      s = e;
      if (s < e0) {
        ++e;
        while (e < e0 && st[e] != kKept) ++e;
      }
    }
  }
  return most;
}

// A lane's points begin, begin + step, ... of segment (s, e) whose upper bound
// reaches `low`, in FP64: the largest numerator and the first point that has it.
// tie: another one comes so close below it that the quotients may be equal.
struct DpBest {
  double c;
  int at;
  bool tie;
};
__device__ __forceinline__ DpBest dp_best(const double2* __restrict__ P,
                                          const float4* __restrict__ q, int begin, int step, int e,
                                          float4 A, float4 B, double2 Ad, double2 Bd, double len,
                                          float low, float uR, float tiny) {
  constexpr double near = 1.0 - 2e-15;
  DpBest r = {0.0, -1, false};
  for (int i = begin; i < e; i += step)
    if (dp_bracket(q[i], A, B, uR, tiny).hi >= low) {
      const double c = ved_num(P[i], Ad, Bd, len);
      if (c > r.c) {
        r.tie = r.tie || (r.at >= 0 && r.c >= __dmul_rn(c, near));
        r.c = c;
        r.at = i;
      } else if (c != r.c && c >= __dmul_rn(r.c, near)) {
        r.tie = true;
      }
    }
  return r;
}
// The first of the lane's points whose VED is the segment's largest: its best one,
// or, with ties about, by another look at all of them.
__device__ __forceinline__ uint32_t dp_first(const double2* __restrict__ P,
                                             const float4* __restrict__ q, int begin, int step,
                                             int e, float4 A, float4 B, double2 Ad, double2 Bd,
                                             double len, float low, float uR, float tiny,
                                             const DpBest& mine, bool ties, double cmax,
                                             double dmax) {
  const double from = __dmul_rn(cmax, 1.0 - 1e-15);
  auto is_it = [&](double c) { return c >= from && (c == cmax || ved_of(c, len) == dmax); };
  if (!ties) return mine.at >= 0 && is_it(mine.c) ? (uint32_t)mine.at : kNoArg;
  for (int i = begin; i < e; i += step)
    if (dp_bracket(q[i], A, B, uR, tiny).hi >= low && is_it(ved_num(P[i], Ad, Bd, len)))
      return (uint32_t)i;
  return kNoArg;
}

// The split of segment (s, e) by one warp, every lane alike; -1: nothing in it
// is above eps.
__device__ __forceinline__ int dp_split_warp(const double2* __restrict__ P,
                                             const float4* __restrict__ q, int s, int e, float uR,
                                             float tiny, float eps_lo, float eps_hi, double eps) {
  const int lane = threadIdx.x & 31;
  const float4 A = q[s], B = q[e];
  float best_lo = 0.f, top = 0.f, second = 0.f;
  int at = -1;
  DpBracket b = dp_bracket(A, A, B, uR, tiny);  // the length's bounds
  for (int i = s + 1 + lane; i < e; i += 32) {
    const DpBracket c = dp_bracket(q[i], A, B, uR, tiny);
    best_lo = fmaxf(best_lo, c.lo);
    if (c.hi > top) {
      second = top;
      top = c.hi;
      at = i;
    } else {
      second = fmaxf(second, c.hi);
    }
  }
  const float low = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(best_lo)));
  const float high = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(top)));
  if (high < eps_lo * b.len_lo) return -1;
  // the points whose upper bound reaches the largest lower bound
  const unsigned one = __ballot_sync(0xffffffffu, at >= 0 && top >= low);
  const unsigned more = __ballot_sync(0xffffffffu, at >= 0 && second >= low && second > 0.f);
  if (!more && __popc(one) == 1 && low > eps_hi * b.len_hi)
    return __shfl_sync(0xffffffffu, at, __ffs(one) - 1);
  // undecided: those points in FP64 (every point of a segment whose bounds say
  // nothing: low is 0 there)
  const double2 Ad = P[s], Bd = P[e];
  const double len = seg_len(Ad, Bd);
  const DpBest mine = dp_best(P, q, s + 1 + lane, 32, e, A, B, Ad, Bd, len, low, uR, tiny);
  double cmax = mine.c;
  for (int o = 16; o > 0; o >>= 1) {
    const double c = __shfl_xor_sync(0xffffffffu, cmax, o);
    if (c > cmax) cmax = c;
  }
  const double dmax = cmax == 0.0 ? 0.0 : ved_of(cmax, len);
  if (!(dmax > eps)) return -1;
  const bool ties = __any_sync(0xffffffffu, mine.tie);
  const uint32_t first = dp_first(P, q, s + 1 + lane, 32, e, A, B, Ad, Bd, len, low, uR, tiny, mine,
                                  ties, cmax, dmax);
  return (int)__reduce_min_sync(0xffffffffu, first);  // kNoArg = -1
}

// The split of segment (s, e) by a team of `size` warps, this one its `rank`-th (the
// same warps of the CTA for all of a team, first its first warp); -1: nothing in it
// is above eps.  The same decisions as dp_split_warp's, the maxima and the points
// left taken over the team through shared memory.  Every warp of the CTA calls it
// alike (warps without a segment: none), for its barriers.
struct TeamShared {
  double c[16];
  float low[16], high[16];
  int at[16], left[16];
  uint32_t first[16];
};
__device__ __forceinline__ int dp_split_team(const double2* __restrict__ P,
                                             const float4* __restrict__ q, int s, int e, bool none,
                                             int first_warp, int rank, int size, float uR,
                                             float tiny, float eps_lo, float eps_hi, double eps,
                                             TeamShared& S) {
  const int lane = threadIdx.x & 31, warp = first_warp + rank;
  const float4 A = q[s], B = q[e];
  const int begin = s + 1 + 32 * rank + lane, step = 32 * size;
  const DpBracket b = dp_bracket(A, A, B, uR, tiny);  // the length's bounds
  float best_lo = 0.f, top = 0.f, second = 0.f;
  int at = -1;
  if (!none)
    for (int i = begin; i < e; i += step) {
      const DpBracket c = dp_bracket(q[i], A, B, uR, tiny);
      best_lo = fmaxf(best_lo, c.lo);
      if (c.hi > top) {
        second = top;
        top = c.hi;
        at = i;
      } else {
        second = fmaxf(second, c.hi);
      }
    }
  float low = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(best_lo)));
  float high = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(top)));
  if (lane == 0) {
    S.low[warp] = low;
    S.high[warp] = high;
  }
  __syncthreads();
  if (!none)
    for (int w = first_warp; w < first_warp + size; ++w) {
      low = fmaxf(low, S.low[w]);
      high = fmaxf(high, S.high[w]);
    }
  const bool closed = none || high < eps_lo * b.len_lo;
  // the points whose upper bound reaches the largest lower bound
  const unsigned one = __ballot_sync(0xffffffffu, at >= 0 && top >= low);
  const unsigned more = __ballot_sync(0xffffffffu, at >= 0 && second >= low && second > 0.f);
  const int mine = one ? __shfl_sync(0xffffffffu, at, __ffs(one) - 1) : -1;
  if (lane == 0) {
    S.left[warp] = more ? 2 : __popc(one);
    S.at[warp] = mine;
  }
  __syncthreads();
  int left = 0, split = -1;
  if (!closed)
    for (int w = first_warp; w < first_warp + size; ++w) {
      left += S.left[w];
      if (S.left[w]) split = S.at[w];
    }
  const bool exact = !closed && !(left == 1 && low > eps_hi * b.len_hi);
  if (closed) split = -1;
  if (!__syncthreads_or(exact)) return split;
  // undecided somewhere: the points left in FP64
  const double2 Ad = P[s], Bd = P[e];
  const double len = seg_len(Ad, Bd);
  DpBest mine_d = {0.0, -1, false};
  if (exact) mine_d = dp_best(P, q, begin, step, e, A, B, Ad, Bd, len, low, uR, tiny);
  double cmax = mine_d.c;
  for (int o = 16; o > 0; o >>= 1) {
    const double c = __shfl_xor_sync(0xffffffffu, cmax, o);
    if (c > cmax) cmax = c;
  }
  bool ties = __any_sync(0xffffffffu, mine_d.tie);
  if (lane == 0) {
    S.c[warp] = cmax;
    S.left[warp] = ties;
  }
  __syncthreads();
  if (exact)
    for (int w = first_warp; w < first_warp + size; ++w) {
      if (S.c[w] > cmax) cmax = S.c[w];
      ties |= S.left[w] != 0;
    }
  const double dmax = cmax == 0.0 ? 0.0 : ved_of(cmax, len);
  uint32_t first = kNoArg;
  if (exact && dmax > eps)
    first = dp_first(P, q, begin, step, e, A, B, Ad, Bd, len, low, uR, tiny, mine_d, ties, cmax,
                     dmax);
  first = __reduce_min_sync(0xffffffffu, first);
  if (lane == 0) S.first[warp] = first;
  __syncthreads();
  if (!exact) return split;
  for (int w = first_warp; w < first_warp + size; ++w) first = min(first, S.first[w]);
  return (int)first;  // kNoArg = -1
}

// list: the trajectories of class cls (0: from the list's start, 1: from its
// end), each of at most m points.  While a level has fewer segments than half the
// CTA's warps and one of them is long, the warps share them in teams (one
// warp a segment left fifteen of sixteen idle at the top of a long track: one of
// 9000 points on a parabola 264 us per call, 172 so, 181 in the level kernel).
constexpr int kTeamPoints = 512;
__global__ void __launch_bounds__(512)
    k_dp_local(const double2* __restrict__ xy, const int64_t* __restrict__ off, int64_t n,
               double eps, int m, int cls, DpCtl* __restrict__ ctl,
               const uint32_t* __restrict__ list, uint32_t list_cap, uint8_t* __restrict__ flag,
               CallScalars* __restrict__ scal, int* __restrict__ iterations) {
  extern __shared__ __align__(16) unsigned char smem[];
  float4* q = reinterpret_cast<float4*>(smem);
  uint32_t* longs = reinterpret_cast<uint32_t*>(q + m);  // [2][m / 16]: start | end << 16
  uint32_t* small = longs + 2 * (m / 16);                // [m / 2]
  uint16_t* lvl = reinterpret_cast<uint16_t*>(small + m / 2);  // kept points: level + 1
  uint8_t* st = reinterpret_cast<uint8_t*>(lvl + m);
  __shared__ uint32_t s_item, s_r, s_small, s_count[2], s_team[2];
  __shared__ TeamShared team;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int warp = tid >> 5, warps = nt >> 5;
  if (__ldg(&ctl->irregular)) return;
  const uint32_t n_local = __ldg(&ctl->n_local[cls]);
  constexpr float u = 0x1p-24f;
  const float eps_lo = (float)(eps * (1.0 - 1e-6)), eps_hi = (float)(eps * (1.0 + 1e-6));
  int most = 1;
  bool worked = false;
  auto list_segment = [&](int s, int e, int which) {
    const uint32_t w = (uint32_t)s | ((uint32_t)e << 16);
    if (e - s < 2) return;
    if (e - s - 1 <= kSmall) {
      small[atomicAdd(&s_small, 1u)] = w;
    } else {
      longs[which * (m / 16) + atomicAdd(&s_count[which], 1u)] = w;
      if (e - s >= kTeamPoints) s_team[which] = 1u;  // any thread, the same value
    }
  };
  for (;;) {
    __syncthreads();  // the previous trajectory's state is no longer read
    if (tid == 0) {
      s_item = atomicAdd(&ctl->next[cls], 1u);
      s_r = s_small = s_count[0] = s_count[1] = s_team[0] = s_team[1] = 0u;
    }
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= n_local) break;
    worked = true;
    const uint32_t k = list[cls ? list_cap - 1 - item : item];
    const int64_t a = off ? off[k] : 0;
    const int len = (int)((off ? off[k + 1] : n) - a);
    const double2* P = xy + a;
    const double2 o = P[0];
    float r = 0.f;
    bool bad = false;
    for (int i = tid; i < len; i += nt) {
      const double2 p = P[i];
      const float2 x = split_double(p.x - o.x), y = split_double(p.y - o.y);
      // an infinite or undefined coordinate: the high word's exponent is full
      bad |= ((unsigned)__double2hiint(p.x) & 0x7ff00000u) == 0x7ff00000u ||
             ((unsigned)__double2hiint(p.y) & 0x7ff00000u) == 0x7ff00000u;
      q[i] = make_float4(x.x, y.x, x.y, y.y);
      r = fmaxf(r, fmaxf(fabsf(x.x), fabsf(y.x)));
      st[i] = i == 0 || i == len - 1 ? kKept : 0;
      lvl[i] = 0;
    }
    if (tid == 0) list_segment(0, len - 1, 0);
    if (bad) atomicOr(&scal->err, kErrNonFinite);
    const uint32_t rb = __reduce_max_sync(0xffffffffu, __float_as_uint(r));
    if (lane == 0) atomicMax(&s_r, rb);
    __syncthreads();
    // (hi is cut, not rounded: 2^-23 above it, inside the margins)
    const float R = __uint_as_float(s_r);
    const float uR = 8.f * u * u * R, tiny = fmaf(uR, uR, 1e-37f);
    for (int it = 0; it < len; ++it) {
      const uint32_t count = s_count[it & 1];
      if (!count) break;
      const uint32_t* cur = longs + (it & 1) * (m / 16);
      // the split of (s, e), by `size` warps of which this is the rank-th
      auto settle = [&](int s, int e, int at, int rank, int size) {
        if (at < 0) {
          for (int i = s + 1 + 32 * rank + lane; i < e; i += 32 * size) st[i] = kDone;
        } else {
          most = max(most, it + 2);
          if (rank == 0 && lane == 0) {
            st[at] = kKept;
            lvl[at] = (uint16_t)(it + 1);
            list_segment(s, at, (it & 1) ^ 1);
            list_segment(at, e, (it & 1) ^ 1);
          }
        }
      };
      if (s_team[it & 1] && 2 * (int)count <= warps) {
        const int size = warps / (int)count, j = warp / size;
        const bool none = j >= (int)count;
        const uint32_t w = cur[none ? 0 : j];
        const int s = (int)(w & 0xffffu), e = (int)(w >> 16), rank = warp - j * size;
        const int at = dp_split_team(P, q, s, e, none, none ? warp : j * size, none ? 0 : rank,
                                     none ? 1 : size, uR, tiny, eps_lo, eps_hi, eps, team);
        if (!none) settle(s, e, at, rank, size);
      } else {
        for (uint32_t j = warp; j < count; j += warps) {
          const int s = (int)(cur[j] & 0xffffu), e = (int)(cur[j] >> 16);
          settle(s, e, dp_split_warp(P, q, s, e, uR, tiny, eps_lo, eps_hi, eps), 0, 1);
        }
      }
      __syncthreads();
      if (tid == 0) s_count[it & 1] = s_team[it & 1] = 0u;  // the list after next
      __syncthreads();
    }
    const uint32_t ns = s_small;
    for (uint32_t j = tid; j < ns; j += nt) {
      const uint32_t w = small[j];
      most = max(most, dp_finish(P, q, st, lvl, (int)(w & 0xffffu), (int)(w >> 16), uR, tiny,
                                 eps_lo, eps_hi, eps));
    }
    __syncthreads();
    for (int i = tid; i < len; i += nt) flag[a + i] = st[i];
  }
  if (worked) {
    const int top = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) atomicMax(iterations, top);
  }
}

// Step 1.  Lanes of a warp hold consecutive points, so equal segment starts
// form runs of lanes: a shuffle scan takes each run's maximum and its last
// lane issues the atomic.
__device__ __forceinline__ void dp_ved(const double2* __restrict__ xy, int64_t n,
                                       const int32_t* __restrict__ s, const int32_t* __restrict__ e,
                                       const uint8_t* __restrict__ flag,
                                       const double* __restrict__ seglen, double* __restrict__ num,
                                       unsigned long long* __restrict__ segmax) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += stride) {
    const int64_t p = base + threadIdx.x;
    int64_t key = -1 - lane;  // lanes without a candidate never join a run
    unsigned long long v = 0ull;
    if (p < n && !(flag[p] & (kKept | kDone))) {
      const int32_t sp = s[p], ep = e[p];
      const double c = ved_num(xy[p], xy[sp], xy[ep], seglen[sp]);
      num[p] = c;
      key = sp;
      v = (unsigned long long)__double_as_longlong(c);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long vo = __shfl_up_sync(0xffffffffu, v, o);
      const int64_t ko = __shfl_up_sync(0xffffffffu, key, o);
      if (lane >= o && ko == key && vo > v) v = vo;
    }
    const int64_t knext = __shfl_down_sync(0xffffffffu, key, 1);
    const bool last = lane == 31 || knext != key;
    if (last && key >= 0 && v != 0ull) atomicMax(&segmax[key], v);
  }
}

// Step 2: the first point of each segment whose VED equals the segment's
// largest, when that exceeds eps.  A cross product below (1 - 1e-15) times the
// largest one gives a VED strictly below the largest after rounding (the
// division is correctly rounded and monotone), so only the others divide.
__device__ __forceinline__ void dp_arg(int64_t n, double eps, const int32_t* __restrict__ s,
                                       const uint8_t* __restrict__ flag,
                                       const double* __restrict__ seglen,
                                       const double* __restrict__ num,
                                       const unsigned long long* __restrict__ segmax,
                                       uint32_t* __restrict__ segarg) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
    if (flag[p] & (kKept | kDone)) continue;
    const int32_t sp = s[p];
    const double cmax = __longlong_as_double((long long)segmax[sp]);
    const double c = num[p];
    if (!(c >= __dmul_rn(cmax, 1.0 - 1e-15))) continue;
    const double len = seglen[sp];
    const double dmax = cmax == 0.0 ? 0.0 : ved_of(cmax, len);
    const double d = c == cmax ? dmax : ved_of(c, len);
    if (dmax > eps && d == dmax) atomicMin(&segarg[sp], (uint32_t)p);
  }
}

// Step 3: keep the split points, move the others' segment ends, close the
// segments without a split, clear the next iteration's slots.
__device__ __forceinline__ void dp_split(const double2* __restrict__ xy, int64_t n,
                                         int32_t* __restrict__ s, int32_t* __restrict__ e,
                                         uint8_t* __restrict__ flag,
                                         const uint32_t* __restrict__ segarg,
                                         double* __restrict__ seglen,
                                         unsigned long long* __restrict__ segmax_next,
                                         uint32_t* __restrict__ segarg_next,
                                         unsigned long long* __restrict__ kept_now) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  unsigned long long mine = 0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
    const uint8_t f = flag[p];
    if (f & (kKept | kDone)) continue;
    int32_t sp = s[p];
    const uint32_t k = segarg[sp];
    if (k == kNoArg) {
      flag[p] = f | kDone;
      continue;
    }
    if ((int64_t)k == p) {  // the lengths of the segments [s, p] and [p, e]
      flag[p] = kKept;
      const double2 q = xy[p];
      seglen[sp] = seg_len(xy[sp], q);
      seglen[p] = seg_len(q, xy[e[p]]);
      ++mine;
      continue;
    }
    if (p < (int64_t)k) e[p] = (int32_t)k;
    else s[p] = sp = (int32_t)k;
    segmax_next[sp] = 0ull;
    segarg_next[sp] = kNoArg;
  }
  if (mine) atomicAdd(kept_now, mine);
}

// Every iteration of the level loop in one cooperative launch (all CTAs
// resident).  counter[it & 1] counts the points iteration `it` keeps; the
// other slot is cleared after the first barrier of the iteration, when every
// CTA has read the previous iteration's count.  Each CTA leaves the loop on
// the same count, so all take the same barriers.  Every iteration keeps at
// least one point or ends the loop, so n + 1 iterations bound it.
__global__ void __launch_bounds__(256)
    k_dp_levels(const double2* __restrict__ xy, int64_t n, double eps, int32_t* __restrict__ s,
                int32_t* __restrict__ e, uint8_t* __restrict__ flag, double* __restrict__ num,
                double* __restrict__ seglen, unsigned long long* __restrict__ segmax,
                uint32_t* __restrict__ segarg, unsigned long long* __restrict__ counter,
                const DpCtl* __restrict__ ctl, int* __restrict__ iterations) {
  if (ctl->n_long == 0u && ctl->irregular == 0u) return;  // the same in every CTA
  cg::grid_group grid = cg::this_grid();
  __shared__ unsigned long long kept;
  int64_t it = 0;
  for (; it <= n; ++it) {
    const int b = (int)(it & 1);
    dp_ved(xy, n, s, e, flag, seglen, num, segmax + b * n);
    grid.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) counter[b ^ 1] = 0ull;
    dp_arg(n, eps, s, flag, seglen, num, segmax + b * n, segarg + b * n);
    grid.sync();
    dp_split(xy, n, s, e, flag, segarg + b * n, seglen, segmax + (b ^ 1) * n,
             segarg + (b ^ 1) * n, counter + b);
    grid.sync();
    if (threadIdx.x == 0) kept = __ldcg(counter + b);
    __syncthreads();
    const bool done = kept == 0ull;
    __syncthreads();  // `kept` is rewritten in the next iteration
    if (done) {
      ++it;
      break;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(iterations, (int)it);
}

// Compaction, kCompact points per CTA.  First the mask and each CTA's count...
constexpr int kCompactThreads = 256, kCompact = 2048;
__global__ void __launch_bounds__(kCompactThreads)
    k_dp_flags(const uint8_t* __restrict__ flag, int64_t n, uint8_t* __restrict__ keep,
               uint32_t* __restrict__ counts) {
  const int64_t base = (int64_t)blockIdx.x * kCompact;
  int mine = 0;
#pragma unroll
  for (int r = 0; r < kCompact / kCompactThreads; ++r) {
    const int64_t p = base + r * kCompactThreads + threadIdx.x;
    const int k = p < n ? (flag[p] & kKept) : 0;
    if (p < n) keep[p] = (uint8_t)k;
    mine += k;
  }
  __shared__ int total;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  mine = __reduce_add_sync(0xffffffffu, mine);
  if ((threadIdx.x & 31) == 0) atomicAdd(&total, mine);
  __syncthreads();
  // one more entry than CTAs, zero, so that the scan ends with the total
  if (threadIdx.x == 0) {
    counts[blockIdx.x] = (uint32_t)total;
    if (blockIdx.x == gridDim.x - 1) counts[gridDim.x] = 0u;
  }
}

// ... then, with the scan of the counts, each kept point to its place, and the
// number of kept points before each point (pos, when the offsets are wanted).
__global__ void __launch_bounds__(kCompactThreads)
    k_dp_compact(const double2* __restrict__ xy, int64_t n, const uint8_t* __restrict__ keep,
                 const uint32_t* __restrict__ first, double2* __restrict__ out,
                 uint32_t* __restrict__ pos, int* __restrict__ total) {
  __shared__ uint32_t warps[kCompactThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * kCompact;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blockIdx.x == 0 && threadIdx.x == 0) *total = (int)first[gridDim.x];
  if (!out && !pos) return;
  uint32_t before = first[blockIdx.x];
#pragma unroll
  for (int r = 0; r < kCompact / kCompactThreads; ++r) {
    const int64_t p = base + r * kCompactThreads + threadIdx.x;
    const bool k = p < n && keep[p];
    const unsigned m = __ballot_sync(0xffffffffu, k);
    if (lane == 0) warps[warp] = __popc(m);
    __syncthreads();
    uint32_t mine = before, all = 0;
    for (int w = 0; w < kCompactThreads / 32; ++w) {
      if (w < warp) mine += warps[w];
      all += warps[w];
    }
    mine += __popc(m & ((1u << lane) - 1u));
    if (p < n) {
      if (pos) pos[p] = mine;
      if (k && out) out[mine] = xy[p];
    }
    before += all;
    __syncthreads();
  }
  if (pos && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) pos[n] = before;
}

__global__ void k_dp_offsets(const uint32_t* __restrict__ pos, const int64_t* __restrict__ off,
                             int64_t ntraj, int64_t n, int64_t* __restrict__ out_off) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k <= ntraj; k += stride) {
    const int64_t o = off ? min(max(off[k], (int64_t)0), n) : (k == 0 ? 0 : n);
    out_off[k] = pos[o];
  }
}

int grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 8));
}

}  // namespace

namespace {

// Blocks of the compaction and the words it needs.
int64_t dp_blocks(int64_t n) { return std::max<int64_t>(1, (n + kCompact - 1) / kCompact); }

}  // namespace

size_t dp_workspace_bytes(int64_t n) {
  const size_t m = (size_t)n + 1, nb = (size_t)dp_blocks(n) + 1;
  return 256 * 16 + m * (4 + 4 + 1 + 16 + 8 + 8 + 8 + 4) + sizeof(uint32_t) * (m / 3 + 1) +
         sizeof(uint32_t) * 2 * nb + 4 * (scan_temp_words((int64_t)nb, 2048) + 64);
}

cudaError_t launch_dp(const double* xy, int64_t n, const int64_t* off, int64_t ntraj, double eps,
                      uint8_t* keep, double* out_xy, int64_t* out_off, void* ws,
                      CallScalars* scal, int64_t* n_kept, int* iterations, int* err_word,
                      cudaStream_t st) {
  const size_t m = (size_t)n + 1;
  char* w = static_cast<char*>(ws);
  size_t o = 0;
  auto take = [&](size_t bytes) { char* r = w + o; o = (o + bytes + 255) & ~(size_t)255; return r; };
  int32_t* s = reinterpret_cast<int32_t*>(take(4 * m));
  int32_t* e = reinterpret_cast<int32_t*>(take(4 * m));
  uint8_t* flag = reinterpret_cast<uint8_t*>(take(m));
  unsigned long long* segmax = reinterpret_cast<unsigned long long*>(take(16 * m));
  double* num = reinterpret_cast<double*>(take(8 * m));
  double* seglen = reinterpret_cast<double*>(take(8 * m));
  uint32_t* segarg = reinterpret_cast<uint32_t*>(take(8 * m));
  uint32_t* pos = reinterpret_cast<uint32_t*>(take(4 * m));
  const uint32_t list_cap = (uint32_t)(m / 3 + 1);
  uint32_t* list = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * list_cap));
  // counters, cleared together: points kept per iteration, the plan
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(take(16 + sizeof(DpCtl)));
  DpCtl* ctl = reinterpret_cast<DpCtl*>(counter + 2);
  const int64_t nb = dp_blocks(n);
  uint32_t* counts = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (nb + 1)));
  uint32_t* first = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (nb + 1)));
  uint32_t* scan_temp =
      reinterpret_cast<uint32_t*>(take(4 * (scan_temp_words(nb + 1, 2048) + 64)));
  const double2* P = reinterpret_cast<const double2*>(xy);
  int* iters_dev = &scal->pad[0];  // read back with the error word
  cudaError_t err = cudaSuccess;
  if (n > 0) {
    if ((err = cudaMemsetAsync(counter, 0, 16 + sizeof(DpCtl), st)) != cudaSuccess) return err;
    int dev = 0, per_sm = 0, sms = 0;
    if ((err = cudaGetDevice(&dev)) != cudaSuccess) return err;
    if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return err;
    // Trajectories of up to a quarter above the mean, the bulk of a call's, run
    // with the shared memory they need, so that many CTAs
    // share an SM; longer ones get the most a CTA can have, and those beyond
    // that go to the level kernel.
    const int64_t mean = n / std::max<int64_t>(ntraj, 1);
    int local_max = kLocalMax;
    int short_max = (int)std::min<int64_t>(kLocalMax,
                                           std::max<int64_t>(256, (5 * mean / 4 + 127) / 128 * 128));
    // Brackets cannot tell a straight track's roundings from a VED above an eps this
    // small (metres), and one SM's FP64 pipe is slower than the GPU's (straight tracks
    // at eps = 0, level kernel / local: one of 9000 points 0.88 / 4.5 ms, 20,000 of 40
    // 1.29 / 1.80); and the list holds 32-bit indices.
    if (eps < 1e-8 || ntraj > 0xffffffffll) local_max = short_max = 2;  // none is local
    k_dp_plan<<<(unsigned)((ntraj + 255) / 256), 256, 0, st>>>(
        P, off, ntraj, n, flag, scal, short_max, local_max, ctl, list, list_cap, iters_dev);
    k_dp_init<<<grid_for(n), 256, 0, st>>>(P, n, off, ntraj, s, e, flag, segmax, segarg, seglen,
                                           local_max, ctl, scal);
    note_launches(2);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    for (int cls = 0; cls < 2; ++cls) {
      const int m = cls ? local_max : short_max;
      // trajectories that can be on the list
      const int64_t most = std::min<int64_t>(ntraj, n / (cls ? short_max + 1 : 3));
      if (most < 1 || (cls && local_max <= short_max)) continue;
      // two warps for the usual track of 500 points (0.34 ms per call on 4000 of
      // them; 0.40 with one warp, 0.36 with four)
      const int threads = 32 * std::min(16, std::max(1, m / 320));
      const size_t smem = dp_local_smem(m);
      if ((err = cudaFuncSetAttribute(k_dp_local, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)dp_local_smem(kLocalMax))) !=
          cudaSuccess)
        return err;
      if ((err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_dp_local, threads,
                                                               smem)) != cudaSuccess)
        return err;
      if (per_sm < 1) return cudaErrorLaunchOutOfResources;
      const int gl = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * sms, most));
      k_dp_local<<<gl, threads, smem, st>>>(P, off, n, eps, m, cls, ctl, list, list_cap, flag,
                                            scal, iters_dev);
      note_launches(1);
      if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    // all CTAs of the cooperative launch must be resident at once
    if ((err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_dp_levels, 256, 0)) !=
        cudaSuccess)
      return err;
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    // up to four CTAs per SM: enough warps for the memory phases, few CTAs
    // at each barrier
    const int gl = (int)std::min<int64_t>((int64_t)std::min(per_sm, 4) * sms, (n + 255) / 256);
    void* args[] = {(void*)&P, (void*)&n, (void*)&eps, (void*)&s, (void*)&e, (void*)&flag,
                    (void*)&num, (void*)&seglen, (void*)&segmax, (void*)&segarg,
                    (void*)&counter, (void*)&ctl, (void*)&iters_dev};
    err = cudaLaunchCooperativeKernel((const void*)k_dp_levels, dim3(gl), dim3(256), args, 0, st);
    note_launches(1);
    if (err != cudaSuccess) return err;
  }
  k_dp_flags<<<(unsigned)nb, kCompactThreads, 0, st>>>(flag, n, keep, counts);
  note_launches(1);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if ((err = launch_exclusive_scan(counts, first, nb + 1, 2048, scan_temp, st)) != cudaSuccess)
    return err;
  k_dp_compact<<<(unsigned)nb, kCompactThreads, 0, st>>>(
      P, n, keep, first, reinterpret_cast<double2*>(out_xy), out_off ? pos : nullptr,
      &scal->pad[1]);
  note_launches(1);
  if (out_off) {
    k_dp_offsets<<<grid_for(ntraj + 1), 256, 0, st>>>(pos, off, ntraj, n, out_off);
    note_launches(1);
  }
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  // everything the host wants, in one copy and one wait
  CallScalars hs;
  if ((err = cudaMemcpyAsync(&hs, scal, sizeof(hs), cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return err;
  if ((err = cudaStreamSynchronize(st)) != cudaSuccess) return err;
  if (n_kept) *n_kept = (uint32_t)hs.pad[1];
  if (iterations) *iterations = hs.pad[0];
  *err_word = hs.err;
  return cudaSuccess;
}

}  // namespace kde
