// The paper's own GPU estimator (Sec. IV-B): the fixes are projected onto the
// count matrix M_D with integer atomic adds (Algorithm 3), cells skipped
// between consecutive fixes of one trajectory are filled by linear
// interpolation (Eq. InterX / InterY), and M_D is convolved with a
// window x window stencil of a Table 1 kernel (Eq. 7).
//
// Counting: the cell index is floor((x - o) / cell) with the FP64 division
// correctly rounded, and the interpolated cells are
// floor(i + (c/c_max) di + 1/2) with c = 1..c_max-1, evaluated with explicitly
// rounded FP64 operations (no fused multiply-add), so the counts are
// bit-identical to a CPU evaluation.  GB300 does 2 FP64 operations per SM and
// clock, so both are decided in FP32 and integers wherever those cannot
// differ from the FP64 evaluation, and in FP64 in the rest (one fix in a
// million; interpolated cells that fall half way between two).
// Integer atomics make the counts independent of scheduling.
//
// Convolution: the Table 1 kernels are products, so the 2-D stencil
// f(s,t) = k(s cell/h) k(t cell/h) / (N h^2) is applied as a row pass and a
// column pass, each thread computing several outputs per value it reads.
#include <math.h>

#include <algorithm>

#include "kde_internal.cuh"

namespace kde {
namespace {

constexpr int kMaxHalf = 127;  // window half-width limit (window <= 255)

// floor((v - o) / d) with the FP64 division correctly rounded, or -1 outside
// [0, n).  FP64 division is costly on this GPU, so the quotient is first
// taken as (v - o) * inv_d (inv_d = 1/d rounded): that product is within
// 3 ulp of the exact quotient, the rounded division within half an ulp, so
// unless the product lies within 4e-15 relative of an integer both have the
// same floor; only those rare cases divide.
__device__ __noinline__ int64_t cell_index(double v, double o, double d, double inv_d, int n) {
  const double t = __dsub_rn(v, o);
  const double q = __dmul_rn(t, inv_d);
  double f = floor(q);
  const double frac = q - f;  // exact for |q| < 2^52
  if (!(fmin(frac, 1.0 - frac) > 4e-15 * fmax(fabs(q), 1.0)))
    f = floor(__ddiv_rn(t, d));
  if (!(f >= 0.0) || f >= (double)n) return -1;
  return (int64_t)f;
}

// The same index from FP32: t = v - o as hi + lo, an estimate of the quotient,
// and the remainder r = t - i d, which one FMA gives to 2^-24 d (i d_hi is
// exact in it and nearly cancels hi).  Where r is inside (0, d) by more than
// the rounding of all of it, i is the floor of the exact quotient, which lies
// far from an integer, so the correctly rounded one has the same floor.  Near a
// cell edge (about 1e-6 of the fixes) and for quotients beyond 2^21 cell_index
// decides.
struct CellMap {
  double o, d, inv_d;
  float dh, dl, inv, margin;  // d = dh + dl, 1 / d, 2^-21 d
  int n;
};
__device__ __forceinline__ int cell_of(double v, const CellMap& m) {
  const double t = __dsub_rn(v, m.o);
  const float2 s = split_double(t);
  const float est = floorf(s.x * m.inv);
  const float r = fmaf(-est, m.dh, s.x) + fmaf(-est, m.dl, s.y);
  if (fabsf(est) < 2097152.f) {
    // the estimate is off by at most one
    float i = est, q = r;
    if (r < 0.f) {
      i -= 1.f;
      q += m.dh;
    } else if (r >= m.dh) {
      i += 1.f;
      q -= m.dh;
    }
    if (q > m.margin && m.dh - q > m.margin) return i >= 0.f && i < (float)m.n ? (int)i : -1;
  }
  return (int)cell_index(v, m.o, m.d, m.inv_d, m.n);
}

// Bits of the fixes that end a trajectory (their successor belongs to another
// one), from the offsets; *irregular is set when the offsets do not rise, and
// the counting then searches them per fix.
__global__ void k_traj_ends(const int64_t* __restrict__ off, int64_t ntraj, int64_t n,
                            uint32_t* __restrict__ ends, unsigned* __restrict__ irregular) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t e = -1;
  if (k < ntraj) {
    e = off[k + 1];
    if (e < off[k]) atomicOr(irregular, 1u);
    --e;
  }
  const bool in = e >= 0 && e < n;
  const uint32_t word = in ? (uint32_t)(e >> 5) : 0xffffffffu;
  const uint32_t bit = in ? 1u << (e & 31) : 0u;
  // neighbouring trajectories of a few fixes share words: one atomic per word
  const unsigned peers = __match_any_sync(0xffffffffu, word);
  const uint32_t bits = __reduce_or_sync(peers, bit);
  if (in && (threadIdx.x & 31) == __ffs(peers) - 1) atomicOr(ends + word, bits);
}

// The cells skipped between the cells (i, j) and (i1, j1), added to the
// counts; returns how many.  The coordinate that moves by c_max steps by one;
// the other one is floor(j + c dj / c_max + 1/2), a remainder in integers
// (Bresenham's).  The FP64 evaluation can differ only where that is an exact
// integer (a tie) and c / c_max is not exact, or for moves so long or cells so
// far that its rounding reaches 1 / (2 c_max); those are evaluated in FP64.
__device__ __forceinline__ int fill_gap(int i, int j, int i1, int j1, int nx,
                                        int* __restrict__ counts) {
  const int64_t di = (int64_t)i1 - i, dj = (int64_t)j1 - j;
  const int64_t adi = di < 0 ? -di : di, adj = dj < 0 ? -dj : dj;
  const int64_t cmax = adi > adj ? adi : adj;
  if (cmax < 2) return 0;
  auto exact = [&](int64_t c, int from, int64_t d) {
    const double t = __ddiv_rn((double)c, (double)cmax);
    return (int64_t)floor(__dadd_rn(__dadd_rn((double)from, __dmul_rn(t, (double)d)), 0.5));
  };
  if (cmax >= 1 << 18) {
    for (int64_t c = 1; c < cmax; ++c)
      atomicAdd(&counts[exact(c, j, dj) * nx + exact(c, i, di)], 1);
    return (int)(cmax - 1);
  }
  const int m = (int)cmax;
  const bool pow2 = (m & (m - 1)) == 0;
  const bool along_x = adi >= adj;  // equal: both step by one, whichever is taken
  const int step = along_x ? (di < 0 ? -1 : 1) : (dj < 0 ? -1 : 1);
  const int slope = 2 * (int)(along_x ? dj : di);
  int major = along_x ? i : j, minor = along_x ? j : i, rem = m;
  const int minor0 = minor;
  for (int c = 1; c < m; ++c) {
    major += step;
    rem += slope;
    if (rem >= 2 * m) {
      ++minor;
      rem -= 2 * m;
    } else if (rem < 0) {
      --minor;
      rem += 2 * m;
    }
    const int at = rem == 0 && !pow2 ? (int)exact(c, minor0, slope / 2) : minor;
    const int64_t cell = along_x ? (int64_t)at * nx + major : (int64_t)major * nx + at;
    atomicAdd(&counts[cell], 1);
  }
  return m - 1;
}

// A warp takes `rounds` x 32 consecutive fixes at a time, as many rounds as leave
// work for every warp (count_rounds); each fix's cell is found
// once, the cell before it comes from the neighbouring lane (lane 0: from the
// last round).  ends: bits of the fixes that end a trajectory; null (no
// scratch for them) or *irregular set: the offsets are searched per fix.
// Bound by instruction issue (slots 69% busy; DRAM 15%).  20M fixes x
// 4096^2, interpolated: 4.21 ms with every index and cell in FP64, the
// successor's cell found again and a search of the offsets per fix; 0.33 now.
__global__ void __launch_bounds__(256)
    k_count(const double2* __restrict__ xy, int64_t n, const int64_t* __restrict__ off,
            int64_t ntraj, const uint32_t* __restrict__ ends,
            const unsigned* __restrict__ irregular, const __grid_constant__ CellMap mx,
            const __grid_constant__ CellMap my, int interpolate, int rounds, int* __restrict__ counts,
            unsigned long long* __restrict__ added) {
  const int lane = threadIdx.x & 31, nx = mx.n;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const bool search = off && (!ends || *irregular);
  const int64_t last_end = off ? off[ntraj] : n;  // no fix from here on has a successor
  // a fix adds up to a side of the grid: their sum needs 64 bits
  unsigned long long total = 0;
  for (int64_t b = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32 * rounds;
       b < n; b += warps * 32 * rounds) {
    double2 v = b + lane < n ? xy[b + lane] : make_double2(0.0, 0.0);
    int last_i = -1, last_j = -1;  // cell of the fix before this round's first
    if (interpolate && b > 0 && lane == 31) {
      const double2 w = xy[b - 1];
      last_i = cell_of(w.x, mx);
      last_j = cell_of(w.y, my);
    }
    uint32_t last_ends = ends && interpolate && b > 0 ? ends[(b >> 5) - 1] : 0u;
    for (int r = 0; r < rounds; ++r) {
      const int64_t p = b + r * 32 + lane;
      if (b + r * 32 >= n) break;
      const double2 now = v;
      if (r + 1 < rounds && p + 32 < n) v = xy[p + 32];
      int i = -1, j = -1;
      if (p < n) {
        i = cell_of(now.x, mx);
        j = cell_of(now.y, my);
        if (i >= 0 && j >= 0) atomicAdd(&counts[(int64_t)j * nx + i], 1);
      }
      if (!interpolate) continue;
      int pi = __shfl_up_sync(0xffffffffu, i, 1), pj = __shfl_up_sync(0xffffffffu, j, 1);
      const int ci = __shfl_sync(0xffffffffu, last_i, 31), cj = __shfl_sync(0xffffffffu, last_j, 31);
      if (lane == 0) {
        pi = ci;
        pj = cj;
      }
      last_i = i;
      last_j = j;
      // does the fix before p end its trajectory?
      bool next = p > 0 && p < n && pi >= 0 && pj >= 0 && i >= 0 && j >= 0;
      if (off && !search) {
        const uint32_t word = ends[(b >> 5) + r];
        const uint32_t e = lane ? word >> (lane - 1) : last_ends >> 31;
        last_ends = word;
        next = next && !(e & 1u) && p < last_end;
      } else if (search && next) {
        int64_t lo = 0, hi = ntraj - 1;  // the last k with off[k] <= p - 1
        while (lo < hi) {
          const int64_t mid = (lo + hi + 1) >> 1;
          if (off[mid] <= p - 1) lo = mid; else hi = mid - 1;
        }
        next = p < off[lo + 1];
      }
      if (next) total += (unsigned)fill_gap(pi, pj, i, j, nx, counts);
    }
  }
  for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
  if (lane == 0 && total) atomicAdd(added, total);
}

// The stencil by distance back from an output's last cell: k[u] multiplies the
// value u cells after the first of its window; zeros up to a multiple of four.
struct Stencil {
  float k[2 * kMaxHalf + 2];
};

// Row pass: R(i, j) = sum_u k_u M(i - a + u, j) (cells outside the grid are
// zero), u falling.  LANES threads take 4 LANES columns of one row: a block's 128,
// or a warp's 32 where a row has no more than that many (four rows a block then).
// A thread computes four
// neighbouring ones, so each 16-byte read of the staged line feeds 16 FMAs (one
// output per thread read 4 bytes per FMA: 107 us on 4096^2 with 35 taps, 58
// now; 20 x 20000 with 97 taps: 16 so, 20 with a block per row, 17 now).  Rows
// are strided over gridDim.y (which is capped at 65535).
constexpr int kRowThreads = 128;
template <int LANES>
__global__ void __launch_bounds__(kRowThreads)
    k_conv_rows(const int* __restrict__ counts, int nx, int ny, int a,
                const __grid_constant__ Stencil st, float* __restrict__ R) {
  constexpr int kRows = kRowThreads / LANES, kTile = 4 * LANES, kLine = kTile + 2 * kMaxHalf + 6;
  __shared__ __align__(16) float lines[kRows][kLine];
  const int i0 = blockIdx.x * kTile, t = threadIdx.x % LANES, sub = threadIdx.x / LANES;
  float* line = lines[sub];
  const int taps4 = (2 * a + 4) / 4;  // groups of four taps
  const int width = min(kTile, nx - i0);
  auto sync = []() {
    if (LANES == 32) __syncwarp();
    else __syncthreads();
  };
  for (int64_t j = (int64_t)blockIdx.y * kRows + sub; j < ny; j += (int64_t)gridDim.y * kRows) {
    const int* row = counts + j * nx;
    for (int x = t; x < ((width + 3) & ~3) + 4 * taps4 + 4; x += LANES) {
      const int i = i0 - a + x;
      if (x < kLine) line[x] = (i >= 0 && i < nx && x < width + 2 * a) ? (float)row[i] : 0.f;
    }
    sync();
    if (4 * t < width) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      const float4* v4 = reinterpret_cast<const float4*>(line) + t;
      float4 hi = v4[taps4];
      for (int g = taps4 - 1; g >= 0; --g) {
        const float4 lo = v4[g];
        const float w[7] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z};
#pragma unroll
        for (int u = 3; u >= 0; --u) {
          const float k = st.k[4 * g + u];
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[c] = fmaf(k, w[c + u], acc[c]);
        }
        hi = lo;
      }
      float* out = R + j * nx + i0 + 4 * t;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (4 * t + c < width) out[c] = acc[c];
    }
    sync();
  }
}

// Column pass: out(i, j) = norm sum_u k_u R(i, j - a + u), u falling.  A block
// takes 32 C columns x kColRows rows; a thread C columns 32 apart and
// eight consecutive rows, and walks the rows of their common window once from
// its end: each value feeds eight FMAs, with coefficients that are zero outside
// an output's window (added zeros change nothing).  Step s of the walk needs the
// coefficients of distances s .. s + 7, which stay in registers, one new one a step.
// The block's rows stay in L1.  Staging 64 rows x 32 columns with one output per
// thread and step: 90 us on 4096^2 with 35 taps, 65 with C = 4 and eight coefficients
// read a step.  C = 1 where the grid has too few blocks of four columns a thread, or
// fewer than 33 columns (conv_columns).
constexpr int kColRows = 64;
template <int C>
__global__ void __launch_bounds__(256)
    k_conv_cols(const float* __restrict__ R, int nx, int ny, int a,
                const __grid_constant__ Stencil st, float norm, float* __restrict__ out) {
  // kz[8 + m] = k by distance m from the walk's first row; zeros around it
  __shared__ float kz[2 * kMaxHalf + 1 + 24];
  for (int x = threadIdx.x; x < 2 * kMaxHalf + 25; x += 256)
    kz[x] = x >= 8 && x - 8 <= 2 * a ? st.k[2 * a - (x - 8)] : 0.f;
  __syncthreads();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int i0 = blockIdx.x * (32 * C) + tx, j0 = blockIdx.y * kColRows + 8 * ty;
  if (i0 >= nx || j0 >= ny) return;
  float acc[8][C];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c) acc[r][c] = 0.f;
  // output row j0 + r takes the tap at distance s + r - 7 in step s, row top - s; the
  // coefficient of step s + r is in k[(s + r) % 8]
  const int top = j0 + 7 + a;
  const int begin = max(top - (ny - 1), 0) & ~7, end = min(8 + 2 * a, top + 1);  // the grid's rows
  float k[8];
#pragma unroll
  for (int r = 0; r < 7; ++r) k[r] = kz[1 + begin + r];
  for (int s0 = begin; s0 < end; s0 += 8) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int s = s0 + q, j = top - s;
      k[(q + 7) & 7] = kz[8 + s];
      float v[C];
#pragma unroll
      for (int c = 0; c < C; ++c)
        v[c] = j >= 0 && j < ny && i0 + 32 * c < nx ? __ldg(R + (int64_t)j * nx + i0 + 32 * c) : 0.f;
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) acc[r][c] = fmaf(k[(q + r) & 7], v[c], acc[r][c]);
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (j0 + r < ny && i0 + 32 * c < nx)
        out[(int64_t)(j0 + r) * nx + i0 + 32 * c] = acc[r][c] * norm;
}

// Rounds of k_count: 16 where every warp of the GPU gets that many (fewer fixes'
// cells are then found twice), fewer below, one under 311,000 fixes, whose gaps would
// otherwise be walked one after the other by a few warps (5000 fixes far apart on
// 512^2: 659 us with a thread per fix and FP64 cells, 1170 with 16 rounds, 173 now).
int count_rounds(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(16, n / (152 * 8 * 8 * 32)));
}

// Columns per thread of the column pass.
int conv_columns(int nx, int ny) {
  const int64_t blocks = (int64_t)((nx + 127) / 128) * ((ny + kColRows - 1) / kColRows);
  return nx > 32 && blocks >= 2 * 152 ? 4 : 1;
}

// One factor k(s) of a Table 1 kernel with its constant, in double (host side).
double table1_factor(int kid, double s) {
  const double a = fabs(s);
  const bool in = a <= 1.0;
  switch (kid) {
    case KDE_UNIFORM: return in ? 0.5 : 0.0;
    case KDE_TRIANGULAR: return in ? 1.0 - a : 0.0;
    case KDE_EPANECHNIKOV: return in ? 0.75 * (1.0 - s * s) : 0.0;
    case KDE_QUARTIC: return in ? 15.0 / 16.0 * (1.0 - s * s) * (1.0 - s * s) : 0.0;
    case KDE_TRIWEIGHT: {
      const double u = 1.0 - s * s;
      return in ? 35.0 / 32.0 * u * u * u : 0.0;
    }
    case KDE_TRICUBE: {
      const double u = 1.0 - a * a * a;
      return in ? 70.0 / 81.0 * u * u * u : 0.0;
    }
    case KDE_GAUSSIAN: return kernel_const_1d(KDE_GAUSSIAN) * exp(-0.5 * s * s);
    default: return in ? kernel_const_1d(KDE_COSINE) * cos(1.5707963267948966 * s) : 0.0;
  }
}

}  // namespace

size_t binned_ends_bytes(int64_t n) { return sizeof(uint32_t) * (size_t)((n + 31) / 32); }

int binned_window(int kid, double h, double cell, int window) {
  if (window > 0) return window;
  const double r = h / cell;
  const int a = kid == KDE_GAUSSIAN ? (int)ceil(4.0 * r) : (int)floor(r);
  return 2 * (a < kMaxHalf ? a : kMaxHalf) + 1;
}

cudaError_t launch_binned(const double* xy, int64_t n, const int64_t* off, int64_t ntraj,
                          double ox, double oy, double cell, int nx, int ny, double h, int kid,
                          int window, int interpolate, int* counts, float* rowbuf,
                          uint32_t* ends, unsigned long long* added, float* out, cudaStream_t s) {
  const int a = (window - 1) / 2;
  if (window < 1 || (window & 1) == 0 || a > kMaxHalf) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int) * (size_t)nx * ny, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(added, 0, 2 * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  // added: the count, then the irregular flag
  unsigned* irregular = reinterpret_cast<unsigned*>(added + 1);
  if (n > 0) {
    if (interpolate && off && ends) {
      if ((e = cudaMemsetAsync(ends, 0, binned_ends_bytes(n), s)) != cudaSuccess) return e;
      k_traj_ends<<<(unsigned)((ntraj + 255) / 256), 256, 0, s>>>(off, ntraj, n, ends, irregular);
      note_launches(1);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    auto map = [&](double o, int cells) {
      CellMap m;
      m.o = o;
      m.d = cell;
      m.inv_d = 1.0 / cell;
      m.dh = (float)cell;
      m.dl = (float)(cell - (double)m.dh);
      m.inv = (float)m.inv_d;
      m.margin = m.dh * 0x1p-21f;
      // cells too small or too large for FP32 go to the FP64 index
      if (!(cell > 1e-30 && cell < 1e30)) m.inv = INFINITY;
      m.n = cells;
      return m;
    };
    const int rounds = count_rounds(n);
    const int64_t per_block = 8 * 32 * rounds;
    const int64_t blocks = std::min<int64_t>((n + per_block - 1) / per_block, 152 * 8);
    k_count<<<(int)blocks, 256, 0, s>>>(reinterpret_cast<const double2*>(xy), n, off, ntraj, ends,
                                        irregular, map(ox, nx), map(oy, ny), interpolate, rounds,
                                        counts, added);
    note_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  Stencil st = {};
  for (int u = 0; u <= 2 * a; ++u) st.k[u] = (float)table1_factor(kid, (a - u) * cell / h);
  const float norm = n > 0 ? (float)(1.0 / ((double)n * h * h)) : 0.0f;
  if (nx <= 128)
    k_conv_rows<32><<<dim3(1, std::min((ny + 3) / 4, 65535)), kRowThreads, 0, s>>>(counts, nx, ny, a,
                                                                                 st, rowbuf);
  else
    k_conv_rows<128><<<dim3((nx + 511) / 512, std::min(ny, 65535)), kRowThreads, 0, s>>>(
        counts, nx, ny, a, st, rowbuf);
  note_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int cols = conv_columns(nx, ny);
  const dim3 tiles((nx + 32 * cols - 1) / (32 * cols), (ny + kColRows - 1) / kColRows);
  if (cols == 4) k_conv_cols<4><<<tiles, 256, 0, s>>>(rowbuf, nx, ny, a, st, norm, out);
  else k_conv_cols<1><<<tiles, 256, 0, s>>>(rowbuf, nx, ny, a, st, norm, out);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace kde
