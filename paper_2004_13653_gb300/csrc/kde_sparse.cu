// Block-sparse skipping for the Gaussian tensor-core path.
//
// In the factorisation F = c A B^T the operands are A[i,p] = 2^(15 - u^2) and
// B[j,p] = (w_p / w_max) 2^(15 - v^2) in FP16 (hi and lo parts for
// split-FP16), u and v the offsets between cell centre and point in units of
// h sqrt(2 ln 2) (the separable Gaussian of Table 1).  Beyond |u| = 6.45 the
// exact value is below 2^-26.6, so both FP16 parts round to zero: such a
// point contributes exactly nothing to any cell of a tile that lies that far
// from it along x or along y.  Skipping those (tile, point) pairs therefore
// changes no product, only which zeros are added.
//
// The points are sorted into bins of 8 to 32 cells a side (the cutoff path's
// stable radix sort, with that reach); a tile (128 x 128 or
// 256 x 256 cells) then needs only the bins
// within reach, i.e. one contiguous run of sorted points per bin row.  This
// file builds the work list (points per tile, cut into pieces of a fixed
// length, and the exclusive scan of the pieces per tile) and sums each
// tile's piece partials, in piece order, into the output.  The pieces of a
// tile all hold piece_len points except its last; the schedule lists the full
// pieces first and then the last pieces by decreasing length, so that dealing
// them to the CTA pairs in snake order balances the pairs' work.
#include "kde_internal.cuh"

namespace kde {
namespace {

__device__ __forceinline__ int inst_of_tile(const TcInst* __restrict__ tab, int ninst, int t) {
  int a = 0, b = ninst - 1;
  while (a < b) {
    const int mid = (a + b + 1) >> 1;
    if (tab[mid].tile_begin <= t) a = mid; else b = mid - 1;
  }
  return a;
}

// The points of a tile's bin rows, one warp per tile, the rows over its lanes
// (one thread per tile was a chain of a hundred dependent reads: 27 us for the
// 16 tiles of 1024^2).
__device__ __forceinline__ uint32_t tile_points(const TcInst* __restrict__ tab, int ninst, int t,
                                                int side) {
  const TcInst& I = tab[inst_of_tile(tab, ninst, t)];
  const int local = t - I.tile_begin;
  const int tm = local % I.tiles_m, tn = local / I.tiles_m;
  const BinRange br = tile_bins(I.cs, I.range_reach, I.inv_binw, I.nbx, I.nby, tm, tn, side);
  uint32_t total = 0;  // the sort holds fewer than 2^32 points
  if (br.lo_bx <= br.hi_bx)
    for (int by = br.lo_by + (threadIdx.x & 31); by <= br.hi_by; by += 32) {
      const int row = I.bin_begin + by * I.nbx;
      total += __ldg(I.start + row + br.hi_bx + 1) - __ldg(I.start + row + br.lo_bx);
    }
  return __reduce_add_sync(0xffffffffu, total);
}

// The tiles' points, piece counts and counts of full pieces.  npieces and
// nfull have tiles_total + 1 entries; the last are zero so that the exclusive
// scans end with the totals.
__global__ void k_sparse_totals(const TcInst* __restrict__ tab, int ninst, SparseCtl sp,
                                uint32_t* __restrict__ tile_total, uint32_t* __restrict__ npieces,
                                uint32_t* __restrict__ nfull) {
  const int t = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (t > sp.tiles_total) return;
  uint32_t total = 0;
  if (t < sp.tiles_total) total = tile_points(tab, ninst, t, sp.side);
  if ((threadIdx.x & 31) != 0) return;
  if (t < sp.tiles_total) tile_total[t] = total;
  npieces[t] = (uint32_t)(((uint64_t)total + sp.piece_len - 1) / sp.piece_len);
  nfull[t] = total / (uint32_t)sp.piece_len;
}

// Lists the tiles whose last piece is short, longest first: a counting sort
// on the piece's length in 512 classes (64-point MMA stages for the longest
// pieces the planner makes; one CTA; the order among tails of the same class
// is whatever the atomics give, which changes no result).
constexpr int kTailClasses = 512;
constexpr int kTailKeys = kTailClasses + 1;  // keys 1 .. kTailClasses
constexpr int kTailThreads = 1024;
static_assert(kTailKeys <= kTailThreads, "one key per thread in the scan");

// class of a short piece of rem points, 1 <= rem < L
__device__ __forceinline__ int tail_key(uint32_t rem, uint32_t L) {
  return 1 + (int)(((uint64_t)(rem - 1) * kTailClasses) / L);
}

__device__ __forceinline__ void list_tails(const SparseCtl& sp, uint32_t (&cnt)[kTailKeys],
                                           uint32_t (&warp_sum)[kTailThreads / 32]) {
  const int tid = threadIdx.x;
  const uint32_t L = (uint32_t)sp.piece_len;
  if (tid < kTailKeys) cnt[tid] = 0;
  __syncthreads();
  for (int t = tid; t < sp.tiles_total; t += kTailThreads) {
    const uint32_t rem = sp.tile_total[t] % L;
    if (rem) atomicAdd(&cnt[tail_key(rem, L)], 1u);
  }
  __syncthreads();
  // exclusive scan with the longest key first: thread r holds key kTailKeys-1-r
  const int key = kTailKeys - 1 - tid;
  const uint32_t c = tid < kTailKeys ? cnt[key] : 0u;
  uint32_t v = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
    if ((tid & 31) >= o) v += n;
  }
  if ((tid & 31) == 31) warp_sum[tid >> 5] = v;
  __syncthreads();
  if (tid < 32) {
    uint32_t w = warp_sum[tid];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t n = __shfl_up_sync(0xffffffffu, w, o);
      if (tid >= o) w += n;
    }
    warp_sum[tid] = w;  // inclusive over warps
  }
  __syncthreads();
  const uint32_t before = v - c + ((tid >> 5) ? warp_sum[(tid >> 5) - 1] : 0u);
  __syncthreads();
  if (tid < kTailKeys) cnt[key] = before;  // now the cursor of each key
  __syncthreads();
  uint32_t* tail = const_cast<uint32_t*>(sp.tail_tile);
  for (int t = tid; t < sp.tiles_total; t += kTailThreads) {
    const uint32_t rem = sp.tile_total[t] % L;
    if (rem) tail[atomicAdd(&cnt[tail_key(rem, L)], 1u)] = t;
  }
}

__global__ void __launch_bounds__(kTailThreads) k_sparse_tails(SparseCtl sp) {
  __shared__ uint32_t cnt[kTailKeys];
  __shared__ uint32_t warp_sum[kTailThreads / 32];
  list_tails(sp, cnt, warp_sum);
}

// The work list of at most kTailThreads tiles in one CTA: totals (a warp per
// tile; with have_totals k_sparse_totals has done them), both exclusive scans
// (a tile per thread) and the tails.  Five launches of a few microseconds each
// become one (1024^2, 16 tiles: 35 us -> 12 us), or two beyond 32 tiles, whose
// bin ranges, FP64, would queue on the one SM's FP64 pipe (256 tiles: 84 us).
__global__ void __launch_bounds__(kTailThreads)
    k_sparse_plan(const TcInst* __restrict__ tab, int ninst, SparseCtl sp,
                  bool have_totals, uint32_t* __restrict__ tile_total,
                  uint32_t* __restrict__ piece_begin, uint32_t* __restrict__ full_begin) {
  __shared__ uint32_t cnt[kTailKeys];
  __shared__ uint32_t warp_sum[kTailThreads / 32];
  __shared__ uint32_t totals[kTailThreads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (have_totals) {
    if (tid < sp.tiles_total) totals[tid] = tile_total[tid];
  } else {
    for (int t = warp; t < sp.tiles_total; t += kTailThreads / 32) {
      const uint32_t total = tile_points(tab, ninst, t, sp.side);
      if (lane == 0) totals[t] = total;
    }
  }
  __syncthreads();
  const uint32_t L = (uint32_t)sp.piece_len;
  const uint32_t total = tid < sp.tiles_total ? totals[tid] : 0u;
  if (tid < sp.tiles_total && !have_totals) tile_total[tid] = total;
  const uint32_t full = total / L, pieces = full + (total % L ? 1u : 0u);
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    const uint32_t c = which ? full : pieces;
    uint32_t v = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += n;
    }
    if (lane == 31) warp_sum[warp] = v;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int w = 0; w < kTailThreads / 32; ++w) {
      if (w < warp) before += warp_sum[w];
      all += warp_sum[w];
    }
    uint32_t* out = which ? full_begin : piece_begin;
    if (tid < sp.tiles_total) out[tid] = before + v - c;
    if (tid == 0) out[sp.tiles_total] = all;
    __syncthreads();
  }
  list_tails(sp, cnt, warp_sum);  // reads tile_total, written before the barriers above
}

// out cell (i, j) of tile t = sum over the tile's pieces, in order.  Grid:
// (tiles, side^2 / kRedCells); a thread sums four adjacent columns of one row,
// eight pieces' loads in flight at a time (the adds stay in piece order).
// Bound by HBM (256 KB per piece); a dense cluster's tile holds most of the
// pieces, so its rows are spread over 128 blocks and each thread keeps enough
// bytes in flight: 1.47M points x 1024^2, 16 tiles: 323 us with one column per
// thread, 16 rows per block and one load at a time.
constexpr int kRedThreads = 128, kRedCells = 4 * kRedThreads;
__global__ void __launch_bounds__(kRedThreads)
    k_sparse_reduce(const TcInst* __restrict__ tab, int ninst, SparseCtl sp) {
  const int t = blockIdx.x;
  const TcInst& I = tab[inst_of_tile(tab, ninst, t)];
  const int local = t - I.tile_begin;
  const int tm = local % I.tiles_m, tn = local / I.tiles_m;
  const int cell = blockIdx.y * kRedCells + 4 * threadIdx.x;  // of the tile
  const int il = cell % sp.side, i = tm * sp.side + il;
  const int jl = cell / sp.side, j = tn * sp.side + jl;
  const int64_t cells = (int64_t)sp.side * sp.side;
  if (i >= I.nx || j >= I.ny) return;
  const int p0 = bounded_piece(sp.piece_begin[t], sp.max_pieces);
  const int p1 = bounded_piece(sp.piece_begin[t + 1], sp.max_pieces);
  const float* src = sp.part + cell;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr int kAhead = 8;
  for (int p = p0; p < p1; p += kAhead) {
    float4 v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (p + u < p1) v[u] = __ldcs(reinterpret_cast<const float4*>(src + (p + u) * cells));
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (p + u < p1) {
        acc.x += v[u].x;
        acc.y += v[u].y;
        acc.z += v[u].z;
        acc.w += v[u].w;
      }
  }
  float* out = I.part + (int64_t)j * I.nx + i;
  const float r[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
  for (int c = 0; c < 4; ++c)  // out is 4-byte aligned only, and nx any number
    if (i + c < I.nx) out[c] = r[c];
}

}  // namespace

size_t sparse_scan_words(int tiles_total) {
  return scan_temp_words((int64_t)tiles_total + 1, 2048) + 64;
}

cudaError_t launch_sparse_plan(const TcInst* tab, int ninst, const SparseCtl& sp,
                               uint32_t* npieces, uint32_t* nfull, uint32_t* scan_temp,
                               CallScalars* err, cudaStream_t s) {
  (void)err;
  if (sp.piece_len <= 0) return cudaErrorInvalidValue;
  const int m = sp.tiles_total + 1;
  const bool one_cta = sp.tiles_total <= kTailThreads, split = sp.tiles_total > 32;
  cudaError_t e = cudaSuccess;
  if (split) {
    k_sparse_totals<<<(m + 7) / 8, 256, 0, s>>>(
        tab, ninst, sp, const_cast<uint32_t*>(sp.tile_total), npieces, nfull);
    note_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (one_cta) {
    k_sparse_plan<<<1, kTailThreads, 0, s>>>(tab, ninst, sp, split,
                                             const_cast<uint32_t*>(sp.tile_total),
                                             const_cast<uint32_t*>(sp.piece_begin),
                                             const_cast<uint32_t*>(sp.full_begin));
    note_launches(1);
    return cudaGetLastError();
  }
  e = launch_exclusive_scan(npieces, const_cast<uint32_t*>(sp.piece_begin), m, 2048, scan_temp, s);
  if (e != cudaSuccess) return e;
  e = launch_exclusive_scan(nfull, const_cast<uint32_t*>(sp.full_begin), m, 2048, scan_temp, s);
  if (e != cudaSuccess) return e;
  k_sparse_tails<<<1, kTailThreads, 0, s>>>(sp);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_sparse_reduce(const TcInst* tab, int ninst, const SparseCtl& sp,
                                 cudaStream_t s) {
  k_sparse_reduce<<<dim3(sp.tiles_total, sp.side * sp.side / kRedCells), kRedThreads, 0, s>>>(
      tab, ninst, sp);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace kde
