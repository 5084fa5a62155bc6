// Path (c): the compact kernels of Table 1 evaluated over their support only.
//
// With the indicator of Eq. 8 a point contributes to the cells within one
// bandwidth of it.  Every point gets the key of its sort bin (4, 8 or
// 16 cells a side, cutoff_sort_bin; points farther than a bandwidth
// outside the grid are dropped), the (key, index) pairs are sorted with a
// stable LSD radix sort, and each 16x16-cell output block is then computed by
// one CTA that reads the points of the sort bins within reach of its cells,
// in sorted order: its eight warps take 32-point batches in turn, keep the
// points within reach of the block, tabulate the x and y kernel factors of the
// block's 16 columns and 16 rows for 16 of them at a time in shared memory, and
// each thread adds the outer products into its eight cells.  The
// blocks run heaviest first; a block with thousands of points within reach may be
// split into four row slices, one CTA each, light blocks share a CTA two at a
// time, four warps each, and blocks that no point reaches get their zeros.  Nothing is accumulated with atomics, and the
// order of every sum is fixed, so results are reproducible bit for bit.  The
// same sort, with a wider reach, orders the points of the
// block-sparse tensor-core path.
#include "kde_internal.cuh"
#include "kernel_factors.cuh"
#include "tc_ptx.cuh"

namespace kde {
namespace {

constexpr int kBin = kCutoffBin;    // cells per output block side
constexpr int kGroupThreads = 32;   // a point group is one warp: 8 cells per thread
constexpr int kGroups = 8;          // point groups per CTA (one output block)
constexpr int kSortThreads = 512;   // 16 warps
constexpr int kSortRounds = 8;      // 32-element rounds per warp
constexpr int kSortChunk = kSortThreads * kSortRounds;  // 4096 keys per block
constexpr int kMaxPasses = 4;     // 8-bit digits of 32-bit keys
constexpr int kBatch = 32;          // points read at a time (one per lane)
constexpr int kStep = 16;           // points whose factors are tabulated at a time

template <class T>
__device__ __forceinline__ int find_by(const T* tab, int ninst, int64_t v, int64_t T::*field) {
  int lo = 0, hi = ninst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].*field <= v) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Radix buckets per pass: the 256 values of an 8-bit digit, then one bucket
// for keys with a bit set at or above `top` = 8 x passes.  Only the key that
// marks padding and unreachable points (total_bins) can have one, when it
// needs a bit more than every valid key; it then sorts after every digit in
// each pass, so the valid keys alone decide the number of passes.
constexpr int kDigits = 257;
static_assert(kSortThreads >= kDigits, "one thread per radix bucket in the look-back");

__device__ __forceinline__ uint32_t radix_digit(uint32_t key, int shift, int top) {
  return (top < 32 && (key >> top) != 0u) ? 256u : (key >> shift) & 255u;
}

// Bin key of each point of every instance (points centred and scaled):
// key = bin_begin + by * nbx + bx, or total_bins for padding and for points
// that cannot reach their grid.  vals = the point's index in the prepared
// arrays.  Each CTA also counts the digits of every radix pass of its keys
// (lanes that share a digit add once) and adds them to the per-pass
// histograms ghist[pass][kDigits].
__global__ void __launch_bounds__(256)
    k_bin_keys(const CutInst* __restrict__ tab, int ninst, int64_t m,
               const float4* __restrict__ prepared, uint32_t total_bins, int passes,
               uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
               uint32_t* __restrict__ ghist) {
  __shared__ uint32_t h[kMaxPasses][kDigits];
  for (int i = threadIdx.x; i < kMaxPasses * kDigits; i += blockDim.x) (&h[0][0])[i] = 0;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  // warp-uniform trip count, so every lane takes part in the matches
  for (int64_t g0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); g0 < m; g0 += stride) {
    const int64_t g = g0 + lane;
    const bool valid = g < m;
    uint32_t key = total_bins;
    if (valid) {
      const CutInst& I = tab[find_by(tab, ninst, g, &CutInst::cut_begin)];
      const int64_t p = g - I.cut_begin;
      if (p < I.n) {
        // FP32 throughout (FP64 is slow here): the keys can be one bin off near
        // a bin edge, which the ranges' widened reach covers
        const float4 q = prepared[I.prep_begin + p];
        const float X = q.x + q.y, Y = q.z + q.w;
        // a point reaches the grid only if it lies within the reach of it
        if (X >= I.key_lo && Y >= I.key_lo && X <= I.key_hx && Y <= I.key_hy) {
          const int bx = min(max((int)floorf(X * I.key_inv), 0), I.nbx - 1);
          const int by = min(max((int)floorf(Y * I.key_inv), 0), I.nby - 1);
          key = (uint32_t)I.bin_begin + (uint32_t)by * I.nbx + bx;
        }
      }
      keys[g] = key;
      vals[g] = (uint32_t)(I.prep_begin + p);
    }
    const unsigned act = __ballot_sync(0xffffffffu, valid);
    for (int pass = 0; pass < passes; ++pass) {
      const uint32_t d = radix_digit(key, 8 * pass, 8 * passes);
      const unsigned peers = __match_any_sync(0xffffffffu, valid ? d : 0xffffffffu) & act;
      if (valid && lane == __ffs(peers) - 1) atomicAdd(&h[pass][d], (uint32_t)__popc(peers));
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * kDigits; i += blockDim.x) {
    const uint32_t c = (&h[0][0])[i];
    if (c) atomicAdd(&ghist[i], c);
  }
}

// Rank of each key's digit among equal digits earlier in this block's chunk:
// each warp walks its 256 keys (kv, loaded beforehand) in rounds of 32, peers
// found with match_any, per-warp digit counts kept in shared memory.
// Deterministic.
__device__ __forceinline__ void rank_digits(const uint32_t (&kv)[kSortRounds], int64_t m,
                                            int64_t base, int shift, int top,
                                            uint32_t (*cnt)[kDigits], uint32_t (&digit)[kSortRounds],
                                            uint32_t (&rank)[kSortRounds]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const int64_t e = base + (int64_t)warp * 32 * kSortRounds + r * 32 + lane;
    const bool valid = e < m;
    const uint32_t d = valid ? radix_digit(kv[r], shift, top) : 0u;
    const uint32_t active = __ballot_sync(0xffffffffu, valid);
    uint32_t peers = 0, old = 0;
    if (valid) {
      peers = __match_any_sync(active, d);
      old = cnt[warp][d];
    }
    __syncwarp();
    if (valid && lane == 31 - __clz(peers)) cnt[warp][d] = old + __popc(peers);
    __syncwarp();
    digit[r] = valid ? d : 0xffffffffu;
    rank[r] = old + __popc(peers & lt);
  }
}

// Look-back status of one (chunk, digit) of a radix pass: bits 61-63 the pass
// number plus one (0 or another pass: not yet published by this pass), bit 60
// set when the value is the inclusive prefix over chunks 0..c, clear when it
// is the chunk's own count; bits 0-39 the value.
constexpr unsigned long long kStatusIncl = 1ull << 60;
constexpr unsigned long long kStatusValue = (1ull << 40) - 1;
constexpr int kRoleLookback = 31;  // timeout role id of the look-back wait

__device__ __forceinline__ unsigned long long status_word(int pass, bool incl, uint64_t v) {
  return ((unsigned long long)(pass + 1) << 61) | (incl ? kStatusIncl : 0ull) | v;
}

// One stable counting pass over 8 bits of the keys and the bucket above them
// (`top` = 8 x passes; Merrill and Garland's
// single-pass prefix scan with decoupled look-back, applied per digit).  CTAs
// take 4096-key chunks in the order they start (a counter), so every chunk a
// CTA waits for belongs to a CTA that is already running.  Each CTA ranks its
// keys per digit (stable: warps in order, lanes in order), publishes its
// per-digit counts, then walks back over earlier chunks until it meets an
// inclusive prefix, publishes its own inclusive prefix and scatters: position
// = (keys of smaller digits) + (same digit in earlier chunks) + rank.  The
// last pass writes the permuted points and weights instead of the indices
// (last = 1), or beside them (2).
// A wait that does not end within the limit records a timeout in err; the
// positions are then bounded, not correct.
__global__ void __launch_bounds__(kSortThreads)
    k_radix_pass(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals, int64_t m,
                 int pass, int top, const uint32_t* __restrict__ ghist,
                 uint32_t* __restrict__ chunk_ctr,
                 unsigned long long* __restrict__ status, uint32_t* __restrict__ keys_out,
                 uint32_t* __restrict__ vals_out, const float4* __restrict__ prepared,
                 const float* __restrict__ wts, float4* __restrict__ spts, float* __restrict__ sw,
                 int last, CallScalars* __restrict__ err, uint64_t limit_ns) {
  __shared__ uint32_t cnt[kSortThreads / 32][kDigits];
  __shared__ uint32_t base[kDigits];
  __shared__ uint32_t wsum[kSortThreads / 32];
  __shared__ uint32_t chunk_s;
  if (threadIdx.x == 0) chunk_s = atomicAdd(&chunk_ctr[pass], 1u);
  for (int i = threadIdx.x; i < (kSortThreads / 32) * kDigits; i += kSortThreads)
    (&cnt[0][0])[i] = 0;
  __syncthreads();
  const uint32_t chunk = chunk_s;
  const int shift = 8 * pass;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t e0 = (int64_t)chunk * kSortChunk + (int64_t)warp * 32 * kSortRounds + lane;
  // every key and index of this thread in flight at once
  uint32_t kv[kSortRounds], vv[kSortRounds];
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const int64_t e = e0 + r * 32;
    kv[r] = e < m ? keys[e] : 0u;
    vv[r] = e < m ? vals[e] : 0u;
  }
  uint32_t digit[kSortRounds], rank[kSortRounds];
  rank_digits(kv, m, (int64_t)chunk * kSortChunk, shift, top, cnt, digit, rank);
  __syncthreads();
  // the first kDigits threads own one bucket each
  const bool dig = threadIdx.x < kDigits;
  const int d = dig ? (int)threadIdx.x : 0;
  uint32_t total = 0;
  if (dig) {
    for (int w = 0; w < kSortThreads / 32; ++w) {
      const uint32_t c = cnt[w][d];
      cnt[w][d] = total;  // exclusive prefix over the warps
      total += c;
    }
  }
  volatile unsigned long long* st = status + (size_t)chunk * kDigits + d;
  if (dig) *st = status_word(pass, chunk == 0, total);
  uint64_t excl = 0;
  if (dig && chunk > 0) {
    // four earlier chunks per step, their words loaded together; the walk
    // ends at the first inclusive prefix (chunk 0 publishes one at once)
    constexpr int kLook = 4;
    const uint64_t t0 = tc::globaltimer_ns();
    int64_t c = (int64_t)chunk - 1;
    for (uint32_t it = 1;; ++it) {
      unsigned long long v[kLook];
#pragma unroll
      for (int j = 0; j < kLook; ++j)
        v[j] = c - j >= 0
                   ? *(volatile unsigned long long*)(status + (size_t)(c - j) * kDigits + d)
                   : 0ull;
      bool done = false;
      int j = 0;
      for (; j < kLook; ++j) {
        if ((int)(v[j] >> 61) != pass + 1) break;  // not yet published
        excl += v[j] & kStatusValue;
        if (v[j] & kStatusIncl) {
          done = true;
          break;
        }
      }
      if (done) break;
      c -= j;
      if (j == 0 && (it & 63) == 0 &&
          (tc::globaltimer_ns() - t0 > limit_ns || it > (1u << 30))) {
        if (atomicOr(&err->err, kErrTimeout | kErrSortTimeout) == 0)
          atomicExch(&err->timeout_where, kRoleLookback);
        break;
      }
    }
    *st = status_word(pass, true, excl + total);
  }
  // keys of smaller digits: exclusive scan of this pass's histogram
  const uint32_t gh = dig ? ghist[pass * kDigits + d] : 0u;
  uint32_t inc = gh;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  uint32_t before = 0;
  for (int w = 0; w < warp; ++w) before += wsum[w];
  if (dig) base[d] = before + inc - gh + (uint32_t)excl;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    if (digit[r] == 0xffffffffu) continue;
    const uint32_t pos = base[digit[r]] + cnt[warp][digit[r]] + rank[r];
    if (pos >= m) continue;  // only after a timed-out wait
    keys_out[pos] = kv[r];
    const uint32_t v = vv[r];
    if (last) {
      spts[pos] = prepared[v];
      sw[pos] = wts[v];
      if (last == 2) vals_out[pos] = v;
    } else {
      vals_out[pos] = v;
    }
  }
}

// start[k] = first position whose key >= k in the sorted keys (k = 0..nbins).
__global__ void k_bin_bounds(const uint32_t* __restrict__ skeys, int64_t m, int nbins,
                             uint32_t* __restrict__ start) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k > nbins) return;
  int64_t lo = 0, hi = m;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (skeys[mid] < (uint32_t)k) lo = mid + 1; else hi = mid;
  }
  start[k] = (uint32_t)lo;
}


// Shared-memory tables of one point group: points within reach that wait for
// their turn (x and y, hi and lo; weights), and the factors of kStep of them.
// A row of factors is four floats longer than its 16 so that eight lanes'
// 16-byte stores, a row each, take all the banks.
constexpr int kRow = kBin + 4;
struct GroupTables {
  float2 P[2][kBatch + kStep];
  float W[kBatch + kStep];
  __align__(16) float K[2][kStep][kRow];
};

// Accumulate the outer products of the first cnt <= kStep waiting points into a
// thread's cells: columns cx, cx+1 of RPL rows from cy0 (acc[2 r + c]); RPL = 4
// for a whole 16-row block, 1 for a 4-row slice of a heavy block.  Product
// kernels from tabulated factors, radial kernels from tabulated squared offsets
// and the profile per pair.  Per point one 8-byte and one 4*RPL-byte table read
// feed 2*RPL FMAs.
template <int KID, bool RADIAL, int RPL>
__device__ __forceinline__ void accumulate(const GroupTables& T, int cnt, int cx, int cy0,
                                           float (&acc)[2 * RPL]) {
  static_assert(RPL == 4 || RPL == 1, "rows per lane");
  auto load_y = [&](int c, float (&y)[RPL]) {
    if constexpr (RPL == 4) {
      const float4 v = *reinterpret_cast<const float4*>(&T.K[1][c][cy0]);
      y[0] = v.x;
      y[1] = v.y;
      y[2] = v.z;
      y[3] = v.w;
    } else {
      y[0] = T.K[1][c][cy0];
    }
  };
  int c = 0;
  if (!RADIAL) {  // two points per step so their table reads are in flight together
    for (; c + 2 <= cnt; c += 2) {
      float2 kx[2];
      float y[2][RPL];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        kx[u] = *reinterpret_cast<const float2*>(&T.K[0][c + u][cx]);
        load_y(c + u, y[u]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
          acc[2 * r] = fmaf(kx[u].x, y[u][r], acc[2 * r]);
          acc[2 * r + 1] = fmaf(kx[u].y, y[u][r], acc[2 * r + 1]);
        }
      }
    }
  }
  for (; c < cnt; ++c) {
    const float2 kx = *reinterpret_cast<const float2*>(&T.K[0][c][cx]);
    float y[RPL];
    load_y(c, y);
    if (RADIAL) {
      const float w = T.W[c];
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        acc[2 * r] = fmaf(w, kradial<KID>(kx.x + y[r]), acc[2 * r]);
        acc[2 * r + 1] = fmaf(w, kradial<KID>(kx.y + y[r]), acc[2 * r + 1]);
      }
    } else {
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        acc[2 * r] = fmaf(kx.x, y[r], acc[2 * r]);
        acc[2 * r + 1] = fmaf(kx.y, y[r], acc[2 * r + 1]);
      }
    }
  }
}

// The factors of the first cnt <= kStep waiting points, lanes l and l + 16 for
// point l's columns and rows: the offset from cell j is that from the item's
// first cell, g0, plus j times the cell's side (pair_offset).  A slice has 4
// rows.
template <int KID, bool RADIAL, int RPL>
__device__ __forceinline__ void tabulate(GroupTables& T, int cnt, int lane, float2 g0, float cs_hi,
                                         float cs_lo) {
  const int axis = lane >> 4, pt = lane & (kStep - 1);
  if (pt < cnt) {
    const float2 p = T.P[axis][pt];
    const float w = axis && !RADIAL ? T.W[pt] : 1.0f;
    const float2 d0 = pair_offset(g0, p);
    const float dh = d0.x, dl = d0.y;
    float4* row = reinterpret_cast<float4*>(&T.K[axis][pt][0]);
#pragma unroll
    for (int q = 0; q < kBin / 4; ++q) {
      if (RPL == 1 && q > 0 && axis) break;
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float j = (float)(4 * q + e);
        const float u = fmaf(j, cs_hi, dh) + fmaf(j, cs_lo, dl);
        v[e] = RADIAL ? u * u : w * kfactor<KID>(u);
      }
      row[q] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// The sort bins whose points can reach output block (bx, by), with the
// widened reach: the points left out have |u| or |v| above 1 in FP32 too, so
// their factors are exactly zero, and those whose FP32 key put them a bin
// further are still in.
__device__ __forceinline__ BinRange output_block_bins(const CutInst& I, int bx, int by) {
  return block_bins(I.cs, I.range_reach, I.inv_binw, I.nbx, I.nby, bx * kBin, by * kBin, kBin);
}

// The instance of global output block blk, and the block's position in it.
__device__ __forceinline__ const CutInst& output_block(const CutInst* __restrict__ tab, int ninst,
                                                       int blk, int& bx, int& by) {
  int lo = 0, hi = ninst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].out_begin <= blk) lo = mid; else hi = mid - 1;
  }
  const CutInst& I = tab[lo];
  const int local = blk - I.out_begin;
  bx = local % I.obx;
  by = local / I.obx;
  return I;
}

// Weight class of a block from the points within its reach (larger is
// heavier): two classes per power of two.
__device__ __forceinline__ int weight_key(uint32_t total) {
  if (total == 0) return 0;
  const int b = 31 - __clz(total);
  return 1 + 2 * b + (b >= 1 ? (int)((total >> (b - 1)) & 1u) : 0);
}

// Blocks with at least 4096 points within reach (weight class 25 and up) of
// an instance whose supports allow it are computed as four items of four rows
// each, so a dense cluster's block is spread over four CTAs instead of
// holding one for the whole launch; their order keys sit above all others, so
// they come first.  The split depends only on the block's own point count
// and its instance, so a block is computed the same way in every run and in a
// batch as on its own.
constexpr int kHeavyKey = 25;  // weight_key(4096)
// Blocks with fewer than 192 points within reach (weight class 15 and below,
// empty blocks included) are computed two to a CTA, four point groups each:
// eight groups would leave most of their warps without a batch.  Like the
// split of heavy blocks, this depends only on the block's own count.
constexpr int kLightKey = 15;  // weight_key(191)
__device__ __forceinline__ int order_key(const CutInst& I, uint32_t total) {
  const int k = weight_key(total);
  return I.slice && k >= kHeavyKey ? kCutOrderClasses + k : k;
}

// Points within reach of each output block, the block's range of sort bins
// (found once here, in FP64, so the gather itself needs no FP64), and the
// count of blocks per weight class.  The rows' runs are read two at a time so
// their loads overlap.
__global__ void k_cut_block_totals(const CutInst* __restrict__ tab, int ninst,
                                   const uint32_t* __restrict__ start, int nblocks,
                                   uint32_t* __restrict__ totals, int4* __restrict__ ranges,
                                   uint32_t* __restrict__ ocount) {
  const int blk = blockIdx.x * blockDim.x + threadIdx.x;
  if (blk >= nblocks) return;
  int bx, by;
  const CutInst& I = output_block(tab, ninst, blk, bx, by);
  const BinRange br = output_block_bins(I, bx, by);
  ranges[blk] = make_int4(br.lo_bx, br.hi_bx, br.lo_by, br.hi_by);
  uint32_t total = 0;
  if (!range_empty(br)) {
    int r = br.lo_by;
    for (; r + 1 <= br.hi_by; r += 2) {
      const uint32_t* a = start + I.bin_begin + r * I.nbx;
      const uint32_t* b = a + I.nbx;
      const uint32_t a0 = __ldg(a + br.lo_bx), a1 = __ldg(a + br.hi_bx + 1);
      const uint32_t b0 = __ldg(b + br.lo_bx), b1 = __ldg(b + br.hi_bx + 1);
      total += (a1 - a0) + (b1 - b0);
    }
    if (r <= br.hi_by) {
      const uint32_t* a = start + I.bin_begin + r * I.nbx;
      total += __ldg(a + br.hi_bx + 1) - __ldg(a + br.lo_bx);
    }
  }
  totals[blk] = total;
  atomicAdd(&ocount[order_key(I, total)], 1u);
}

// The output blocks in decreasing weight class (a counting sort; within a
// class the order is whatever the atomics give).  Each block computes only its
// own cells, so the order changes the schedule, never a result: the heaviest
// blocks (dense clusters) start first instead of wherever raster order puts
// them.
__global__ void k_cut_order_scatter(const CutInst* __restrict__ tab, int ninst,
                                    const uint32_t* __restrict__ totals, int nblocks,
                                    uint32_t* __restrict__ ocount, uint32_t* __restrict__ order) {
  __shared__ uint32_t first[kCutOrderKeys];
  if (threadIdx.x == 0) {
    uint32_t acc = 0;
    for (int k = kCutOrderKeys - 1; k >= 0; --k) {
      first[k] = acc;
      acc += ocount[k];
    }
    // the blocks to be split into slices come first, then the others, the light
    // ones and those without a point: the gather needs where each kind begins
    if (blockIdx.x == 0) {
      ocount[2 * kCutOrderKeys] = first[kCutOrderClasses - 1];
      ocount[2 * kCutOrderKeys + 1] = first[kLightKey];
      ocount[2 * kCutOrderKeys + 2] = first[0];
    }
  }
  __syncthreads();
  const int blk = blockIdx.x * blockDim.x + threadIdx.x;
  if (blk >= nblocks) return;
  int bx, by;
  const int key = order_key(output_block(tab, ninst, blk, bx, by), __ldg(totals + blk));
  order[first[key] + atomicAdd(&ocount[kCutOrderKeys + key], 1u)] = (uint32_t)blk;
}

constexpr int kCutCtasPerSm = 4;
constexpr int kSliceRows = 4;
// dynamic shared memory of the gather: the groups' tables, then their running sums
constexpr size_t kCutTablesBytes = sizeof(GroupTables) * kGroups;
constexpr size_t kCutSmemBytes = kCutTablesBytes + sizeof(float2) * kGroups * 8 * kGroupThreads;
constexpr int kSlices = kBin / kSliceRows;  // items per heavy block

// The work of one item, for one kernel: rows y_off..y_off + 4 RPL - 1 of the
// block (RPL = 4: all 16 rows; RPL = 1: a 4-row slice).  The points that can
// reach those rows are the runs of the sort bins in range br, one run per bin
// row; their concatenation is cut into kBatch-point batches, and group g of
// the block's NG takes batches g, g+NG, g+2NG, ... (fetching the next while computing
// the current; the warp synchronises only itself).  The bins hold half as many
// points again as reach the item at a reach of 3 cells: the others, whose
// factors are zeros, are dropped, and the rest wait until there are kStep.
// After 32 points the products go into the (hi, lo) running sums of the cells
// with a two-sum; the running sums live in shared memory (run[r * 32] for cell r
// of this lane), which keeps the kernel at 64 registers and four CTAs per SM.
// Bound by shared memory's 128 bytes per clock to the registers and by the
// latency of the point reads: with every point of the bins computed, and its
// factors made a cell per lane from a broadcast of the point, 4M points x 1024^2
// took 664 us per call at a reach of 3 cells, 1080 at 6 and 1292 at 12; now 543,
// 781 and 936.
template <int KID, bool RADIAL, int RPL, int NG>
__device__ __forceinline__ void cutoff_group(const CutInst& I, const float4* __restrict__ P,
                                             const float* __restrict__ W,
                                             const uint32_t* __restrict__ start, int bx, int by,
                                             int y_off, const BinRange& br, int64_t total, int g,
                                             int lane, GroupTables& T, float2* run) {
  static_assert(kGroupThreads == 2 * kStep && kBatch == kGroupThreads && kBatch % kStep == 0,
                "table roles");
  const int nx = I.nx, ny = I.ny;
  const int x0 = bx * kBin, y0 = by * kBin + y_off;
  const int cx = 2 * (lane & 7), cy0 = RPL * (lane >> 3);
  if (total == 0 || y0 >= ny) return;  // a ragged block's slice may have no row
  const float2 g0 = lane < kStep ? I.gxt[x0] : I.gyt[y0];
  // the item's reach, widened as the bin ranges are: points beyond it have a
  // factor of exactly zero at every cell
  float x_lo, x_hi, y_lo, y_hi;
  {
    const float2 a = I.gxt[x0], b = I.gxt[min(x0 + kBin - 1, nx - 1)];
    const float2 c = I.gyt[y0], d = I.gyt[min(y0 + 4 * RPL - 1, ny - 1)];
    x_lo = (a.x + a.y) - I.drop_reach;
    x_hi = (b.x + b.y) + I.drop_reach;
    y_lo = (c.x + c.y) - I.drop_reach;
    y_hi = (d.x + d.y) + I.drop_reach;
  }
  const float cs_hi = I.cs_hi, cs_lo = I.cs_lo;
  RunCursor32 cur;
  cur.init(start, I.bin_begin, I.nbx, br);
  constexpr uint32_t kStride = NG * kBatch;
  const uint32_t total32 = (uint32_t)total;
  uint32_t v = g * kBatch + lane;  // this lane's point of the warp's current batch
  float4 pf = make_float4(0.f, 0.f, 0.f, 0.f);
  float wf = 0.f;
  if (v < total32) {
    const uint32_t p = cur.map(v);
    pf = P[p];
    wf = W[p];
  }
  float acc[2 * RPL];
#pragma unroll
  for (int r = 0; r < 2 * RPL; ++r) acc[r] = 0.f;
  int held = 0, waiting = 0;  // points in acc, and in the tables
  auto flush = [&]() {
#pragma unroll
    for (int r = 0; r < 2 * RPL; ++r) {
      float2 x = run[r * kGroupThreads];
      two_sum_acc(x, acc[r]);
      run[r * kGroupThreads] = x;
      acc[r] = 0.f;
    }
  };
  for (uint32_t b0 = g * kBatch;; b0 += kStride, v += kStride) {
    const bool more = b0 < total32;
    if (more) {
      const float X = pf.x + pf.y, Y = pf.z + pf.w;
      const bool in = v < total32 && X >= x_lo && X <= x_hi && Y >= y_lo && Y <= y_hi;
      const uint32_t mask = __ballot_sync(0xffffffffu, in);
      if (in) {
        const int e = waiting + __popc(mask & ((1u << lane) - 1u));
        T.P[0][e] = make_float2(pf.x, pf.y);
        T.P[1][e] = make_float2(pf.z, pf.w);
        T.W[e] = wf;
      }
      waiting += __popc(mask);
      __syncwarp();
      if (v + kStride < total32) {  // next batch, in flight
        const uint32_t p = cur.map(v + kStride);
        pf = P[p];
        wf = W[p];
      }
    }
    while (waiting >= (more ? kStep : 1)) {  // at the end, the points left too
      const int cnt = min(waiting, kStep);
      tabulate<KID, RADIAL, RPL>(T, cnt, lane, g0, cs_hi, cs_lo);
      __syncwarp();
      accumulate<KID, RADIAL, RPL>(T, cnt, cx, cy0, acc);
      held += cnt;
      waiting -= cnt;
      if (held >= kBatch) {
        flush();
        held = 0;
      }
      // the points left, at most 31, move to the front
      float2 px = make_float2(0.f, 0.f), py = px;
      float w = 0.f;
      if (lane < waiting) {
        px = T.P[0][lane + kStep];
        py = T.P[1][lane + kStep];
        w = T.W[lane + kStep];
      }
      __syncwarp();
      if (lane < waiting) {
        T.P[0][lane] = px;
        T.P[1][lane] = py;
        T.W[lane] = w;
      }
      __syncwarp();
    }
    if (!more) break;
  }
  flush();
}

// Points of the sort bins in range br (the runs of its bin rows).
__device__ __forceinline__ uint32_t range_total(const uint32_t* __restrict__ start, int row0,
                                                int nbx, const BinRange& br) {
  uint32_t total = 0;
  if (range_empty(br)) return 0;
  for (int r = br.lo_by; r <= br.hi_by; ++r) {
    const uint32_t* a = start + row0 + r * nbx;
    total += __ldg(a + br.hi_bx + 1) - __ldg(a + br.lo_bx);
  }
  return total;
}

template <int RPL, int NG>
__device__ __forceinline__ void group_dispatch(const CutInst& I, const float4* __restrict__ P,
                                               const float* __restrict__ W,
                                               const uint32_t* __restrict__ start, int bx, int by,
                                               int y_off, const BinRange& br, int64_t total, int g,
                                               int lane, GroupTables& T, float2* run) {
  switch (I.kid) {
#define KDE_CUT(K)                                                                       \
  case K:                                                                                \
    cutoff_group<K, false, RPL, NG>(I, P, W, start, bx, by, y_off, br, total, g, lane, T, run); \
    break;                                                                               \
  case kRadial + K:                                                                      \
    cutoff_group<K, true, RPL, NG>(I, P, W, start, bx, by, y_off, br, total, g, lane, T, run); \
    break;
    KDE_CUT(KDE_UNIFORM)
    KDE_CUT(KDE_TRIANGULAR)
    KDE_CUT(KDE_EPANECHNIKOV)
    KDE_CUT(KDE_QUARTIC)
    KDE_CUT(KDE_TRIWEIGHT)
    KDE_CUT(KDE_TRICUBE)
    KDE_CUT(KDE_COSINE)
#undef KDE_CUT
    default: break;
  }
}

// One item by a CTA of kGroups one-warp point groups.  A whole
// block's eight cells per thread, or a slice's two, are summed over the groups
// in group order at the end, so every cell is computed by one CTA in a fixed
// order and results are reproducible bit for bit.  Blocks of 16 cells spread a
// dense region over many CTAs; the finer sort bins keep the points an item
// reads close to those its cells' supports actually reach.
struct ItemShared {
  int4 rg[2];
  uint32_t total[2];
  int blk[2];
  int64_t next;  // the CTA's next item
};
// thread 0 takes the CTA's next item
__device__ __forceinline__ void take_next(uint32_t* ctr, ItemShared& S) {
  if (threadIdx.x == 0) S.next = (int64_t)gridDim.x + atomicAdd(ctr, 1u);
}

// two light blocks: half h = g / 4 takes the block at order position
// pos0 + h with its four groups
__device__ __forceinline__ void light_item(const CutInst* __restrict__ tab, int ninst,
                                           const float4* __restrict__ P,
                                           const float* __restrict__ W,
                                           const uint32_t* __restrict__ start,
                                           const uint32_t* __restrict__ order,
                                           const uint32_t* __restrict__ totals,
                                           const int4* __restrict__ ranges, int64_t pos0,
                                           int64_t end, GroupTables& T,
                                           float2 (*part)[8][kGroupThreads], ItemShared& S) {
  const int g = threadIdx.x / kGroupThreads, lane = threadIdx.x % kGroupThreads;
  const int half = g >> 2, gh = g & 3;
  const int64_t pos = pos0 + half;
  const bool has = pos < end;
  if (has && gh == 0 && lane == 0) {
    const int blk = (int)__ldg(order + pos);
    S.blk[half] = blk;
    S.rg[half] = __ldg(ranges + blk);
    S.total[half] = __ldg(totals + blk);
  }
  __syncthreads();
  if (has) {
    int bx, by;
    const CutInst& I = output_block(tab, ninst, S.blk[half], bx, by);
    const int4 rg = S.rg[half];
    const BinRange br = {rg.x, rg.y, rg.z, rg.w};
#pragma unroll
    for (int r = 0; r < 8; ++r) part[g][r][lane] = make_float2(0.f, 0.f);
    group_dispatch<4, 4>(I, P, W, start, bx, by, 0, br, S.total[half], gh, lane, T,
                         &part[g][0][lane]);
  }
  __syncthreads();  // every group's running sums are final
  if (has) {
    // group gh of the half combines cells 2 gh and 2 gh + 1 of every
    // thread's eight over the half's four groups, in order
    int bx, by;
    const CutInst& I = output_block(tab, ninst, S.blk[half], bx, by);
    const int cx = 2 * (lane & 7), cy0 = 4 * (lane >> 3);
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int r = 2 * gh + rr;
      float2 sum = part[4 * half][r][lane];
#pragma unroll
      for (int h = 1; h < 4; ++h) {
        const float2 o = part[4 * half + h][r][lane];
        two_sum_acc(sum, o.x);
        sum.y += o.y;
      }
      const int x = bx * kBin + cx + (r & 1), y = by * kBin + cy0 + (r >> 1);
      if (x < I.nx && y < I.ny) I.out[(int64_t)y * I.nx + x] = (sum.x + sum.y) * I.scale;
    }
  }
}

// a whole block (slice < 0) or a slice of one
__device__ __forceinline__ void block_item(const CutInst* __restrict__ tab, int ninst,
                                           const float4* __restrict__ P,
                                           const float* __restrict__ W,
                                           const uint32_t* __restrict__ start, int blk, int slice,
                                           const uint32_t* __restrict__ totals,
                                           const int4* __restrict__ ranges, GroupTables& T,
                                           float2 (*part)[8][kGroupThreads], uint32_t* ctr,
                                           ItemShared& S) {
  const int g = threadIdx.x / kGroupThreads, lane = threadIdx.x % kGroupThreads;
  int bx, by;
  const CutInst& I = output_block(tab, ninst, blk, bx, by);
  if (threadIdx.x == 0) {
    if (slice < 0) {
      S.rg[0] = __ldg(ranges + blk);
      S.total[0] = __ldg(totals + blk);
    } else {  // the slice's own bin range and point count
      const BinRange b = block_bins_rect(I.cs, I.range_reach, I.inv_binw, I.nbx, I.nby, bx * kBin,
                                         by * kBin + slice * kSliceRows, kBin, kSliceRows);
      S.rg[0] = make_int4(b.lo_bx, b.hi_bx, b.lo_by, b.hi_by);
      S.total[0] = range_total(start, I.bin_begin, I.nbx, b);
    }
  }
  __syncthreads();
  const int4 rg = S.rg[0];
  const BinRange br = {rg.x, rg.y, rg.z, rg.w};
  const int64_t total = S.total[0];
  if (slice < 0) {
#pragma unroll
    for (int r = 0; r < 8; ++r) part[g][r][lane] = make_float2(0.f, 0.f);
    group_dispatch<4, kGroups>(I, P, W, start, bx, by, 0, br, total, g, lane, T,
                               &part[g][0][lane]);
    __syncthreads();  // every group's running sums are final
    take_next(ctr, S);
    // group g combines cell r = g of every thread's eight, over the groups in
    // order (the same order for every block and run)
    static_assert(kGroups == 8, "one cell of eight per group");
    const int r = g;
    const int cx = 2 * (lane & 7), cy0 = 4 * (lane >> 3);
    float2 sum = part[0][r][lane];
#pragma unroll
    for (int h = 1; h < kGroups; ++h) {
      const float2 o = part[h][r][lane];
      two_sum_acc(sum, o.x);
      sum.y += o.y;
    }
    const int x = bx * kBin + cx + (r & 1), y = by * kBin + cy0 + (r >> 1);
    if (x < I.nx && y < I.ny) I.out[(int64_t)y * I.nx + x] = (sum.x + sum.y) * I.scale;
  } else {
    part[g][0][lane] = make_float2(0.f, 0.f);
    part[g][1][lane] = make_float2(0.f, 0.f);
    group_dispatch<1, kGroups>(I, P, W, start, bx, by, slice * kSliceRows, br, total, g, lane, T,
                               &part[g][0][lane]);
    __syncthreads();
    take_next(ctr, S);
    if (threadIdx.x < 2 * kGroupThreads) {  // 64 cells, one thread each
      const int l = threadIdx.x >> 1, r = threadIdx.x & 1;
      float2 sum = part[0][r][l];
#pragma unroll
      for (int h = 1; h < kGroups; ++h) {
        const float2 o = part[h][r][l];
        two_sum_acc(sum, o.x);
        sum.y += o.y;
      }
      const int x = bx * kBin + 2 * (l & 7) + r, y = by * kBin + slice * kSliceRows + (l >> 3);
      if (x < I.nx && y < I.ny) I.out[(int64_t)y * I.nx + x] = (sum.x + sum.y) * I.scale;
    }
  }
}

// The items, taken from a counter by CTAs that stay: first the four slices of
// every heavy block, then the other blocks, each in the order list's
// heaviest-first order, then the light blocks two at a time, groups 0-3 on the
// first and 4-7 on the second, and last the blocks that no point reaches, whose
// zeros a warp writes, 32 blocks an item.  The counts are known on the device
// only; a CTA for every item there could be was 65,536 launches at 4096^2, most
// of which found nothing to do.
constexpr int kEmptyPerItem = 32;
__global__ void __launch_bounds__(kGroups * kGroupThreads, 4)
    k_cutoff(const CutInst* __restrict__ tab, int ninst, const float4* __restrict__ P,
             const float* __restrict__ W, const uint32_t* __restrict__ start,
             const uint32_t* __restrict__ order, const uint32_t* __restrict__ totals,
             const int4* __restrict__ ranges, uint32_t* __restrict__ counts, int nblocks,
             const CallScalars* __restrict__ err) {
  // the groups' tables, then their running sums (cell r of lane l of group g
  // at part[g][r][l])
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ ItemShared S;
  GroupTables* tables = reinterpret_cast<GroupTables*>(smem);
  float2 (*part)[8][kGroupThreads] =
      reinterpret_cast<float2 (*)[8][kGroupThreads]>(smem + kCutTablesBytes);
  const int g = threadIdx.x / kGroupThreads, lane = threadIdx.x % kGroupThreads;
  // after a timed-out sort the bin starts may not rise, and positions taken
  // from them could leave the sorted points: compute nothing (the call
  // reports the timeout)
  if (*reinterpret_cast<const volatile int*>(&err->err) & kErrSortTimeout) return;
  // blocks to split, and the order positions of the first light and empty ones
  const int64_t heavy = __ldg(counts), light = __ldg(counts + 1), empty = __ldg(counts + 2);
  const int64_t slices = kSlices * heavy, singles = slices + (light - heavy);
  const int64_t pairs = singles + (empty - light + 1) / 2;
  const int64_t items = pairs + (nblocks - empty + kEmptyPerItem - 1) / kEmptyPerItem;
  int64_t item = blockIdx.x;
  while (item < items) {
    // a CTA takes its next item when its long item ends (one taken before would
    // wait for it: 4M points x 1024^2 at a reach of 14 cells 1243 us against
    // 1056), and while it computes a short one
    if (item >= singles) take_next(counts + 3, S);
    if (item < singles) {
      const bool slice = item < slices;
      const int64_t pos = slice ? item / kSlices : heavy + (item - slices);
      block_item(tab, ninst, P, W, start, (int)__ldg(order + pos),
                 slice ? (int)(item % kSlices) : -1, totals, ranges, tables[g], part, counts + 3, S);
    } else if (item < pairs) {
      light_item(tab, ninst, P, W, start, order, totals, ranges, light + 2 * (item - singles),
                 empty, tables[g], part, S);
    } else {
      for (int k = g; k < kEmptyPerItem; k += kGroups) {
        const int64_t pos = empty + kEmptyPerItem * (item - pairs) + k;
        if (pos >= nblocks) break;
        int bx, by;
        const CutInst& I = output_block(tab, ninst, (int)__ldg(order + pos), bx, by);
        const int x = bx * kBin + (lane & 15);
        for (int r = lane >> 4; r < kBin; r += 2) {
          const int y = by * kBin + r;
          if (x < I.nx && y < I.ny) I.out[(int64_t)y * I.nx + x] = 0.f * I.scale;
        }
      }
    }
    __syncthreads();  // the item's shared memory is free, and S.next there
    item = S.next;
    __syncthreads();
  }
}

int grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

}  // namespace

CutoffGeom cutoff_geometry(int nx, int ny, double cs, double reach, int bin) {
  CutoffGeom g;
  g.bin = bin;
  g.nbx = (nx + bin - 1) / bin;
  g.nby = (ny + bin - 1) / bin;
  g.nbins = g.nbx * g.nby;
  g.inv_binw = 1.0 / (bin * cs);
  g.ext_x = nx * cs + reach;
  g.ext_y = ny * cs + reach;
  return g;
}

// Sort bins of 8 cells, 16 beyond a reach of 12.  A block reads the points of
// about (16 + 2 reach + bin)^2 cells and computes the (16 + 2 reach)^2 cells'
// that reach it; finer bins mean more bins to sort and to find, and three radix
// passes sooner.  4-, 8- and 16-cell bins, us per call: 1M points x 1024^2 at a
// reach of 3 cells 199 / 203 / 223, x 2048^2 275 / 254 / 258, 8M x 4096^2 1385 /
// 1270 / 1258, 200,000 x 4096^2 at 14 cells 430 / 376 / 342, 8M 2594 / 2434 /
// 2324.  4-cell bins only where the reach is short (a block then reads fewest
// points beyond it), the points many and the bins still two passes' worth.
int cutoff_sort_bin(int64_t n, int nx, int ny, double reach_cells) {
  const int64_t bins4 = (int64_t)((nx + 3) / 4) * ((ny + 3) / 4);
  const bool fine = reach_cells <= 4.0 && n >= (1 << 18) && n >= 8 * bins4 && bins4 <= 65536;
  int bin = fine ? 4 : reach_cells <= 12.0 ? 8 : 16;
  while (bin < 64 && ((int64_t)(nx + bin - 1) / bin) * ((ny + bin - 1) / bin) > (1 << 24)) bin *= 2;
  return bin;
}

// The four slices read (4 + 2 reach + bin) / (16 + 2 reach + bin) of the block's
// points each: up to 6 cells of reach that costs little; beyond, they pay where
// the grid has too few blocks to fill the GPU (200,000 points x 256^2 at 8
// cells: 178 us whole, 139 sliced; 1M x 1024^2 at 14 cells: 352 and 470).
bool cutoff_slices(int nx, int ny, double reach_cells) {
  const double blocks = ((nx + kBin - 1) / kBin) * (double)((ny + kBin - 1) / kBin);
  return reach_cells <= 6.0 || blocks * reach_cells <= 8192.0;
}

CutoffSizes cutoff_sizes(int64_t m, int64_t total_bins) {
  CutoffSizes z;
  z.nchunks = (int)((m + kSortChunk - 1) / kSortChunk);
  // the valid keys 0..total_bins - 1 set the passes; the marker total_bins
  // takes the bucket above the digits where it needs one more bit
  int bits = 1;
  while ((1ll << bits) < (long long)total_bins) ++bits;
  z.passes = (bits + 7) / 8;
  // look-back status (one 64-bit word per chunk and bucket), the per-pass
  // bucket histograms and the per-pass chunk counters, cleared together
  z.hist_words = (size_t)2 * kDigits * z.nchunks + (size_t)kMaxPasses * kDigits + kMaxPasses;
  return z;
}

cudaError_t launch_bin_sort(const CutInst* tab, int ninst, int64_t m, int64_t total_bins,
                            const float4* prepared, const float* prepared_w, const CutoffSizes& z,
                            CutoffScratch ws, cudaStream_t s, bool indices) {
  if (ninst <= 0 || m <= 0) return cudaSuccess;
  if (z.passes < 1 || z.passes > kMaxPasses) return cudaErrorInvalidValue;
  unsigned long long* status = reinterpret_cast<unsigned long long*>(ws.hist);
  uint32_t* ghist = ws.hist + (size_t)2 * kDigits * z.nchunks;
  uint32_t* chunk_ctr = ghist + kMaxPasses * kDigits;
  cudaError_t e = cudaMemsetAsync(ws.hist, 0, sizeof(uint32_t) * z.hist_words, s);
  if (e != cudaSuccess) return e;
  k_bin_keys<<<grid_for(m), 256, 0, s>>>(tab, ninst, m, prepared, (uint32_t)total_bins, z.passes,
                                         ws.keys[0], ws.vals[0], ghist);
  note_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  int cur = 0;
  for (int pass = 0; pass < z.passes; ++pass) {
    const int last = pass == z.passes - 1 ? (indices ? 2 : 1) : 0;
    k_radix_pass<<<z.nchunks, kSortThreads, 0, s>>>(ws.keys[cur], ws.vals[cur], m, pass,
                                                    8 * z.passes, ghist, chunk_ctr, status,
                                                    ws.keys[cur ^ 1],
                                                    ws.vals[cur ^ 1], prepared, prepared_w, ws.spts,
                                                    ws.sw, last, ws.err, tc::kWaitLimitNs);
    note_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    cur ^= 1;
  }
  k_bin_bounds<<<(int)((total_bins + 1 + 255) / 256), 256, 0, s>>>(ws.keys[cur], m,
                                                                   (int)total_bins, ws.start);
  note_launches(1);
  return cudaGetLastError();
}

size_t lookback_probe_words() {
  return 4 * 2 * kSortChunk + 2 * 2 * kDigits + kDigits + kMaxPasses;
}

cudaError_t launch_lookback_timeout_probe(uint32_t* buf, CallScalars* err, uint64_t limit_ns,
                                          cudaStream_t s) {
  // zero keys in two chunks; the chunk counter starts at 1, so the one
  // CTA takes chunk 1 and waits for a chunk 0 that never publishes
  constexpr int64_t m = 2 * kSortChunk;
  uint32_t* keys = buf;
  uint32_t* vals = keys + m;
  uint32_t* keys_out = vals + m;
  uint32_t* vals_out = keys_out + m;
  unsigned long long* status = reinterpret_cast<unsigned long long*>(vals_out + m);
  uint32_t* ghist = reinterpret_cast<uint32_t*>(status + 2 * kDigits);
  uint32_t* chunk_ctr = ghist + kDigits;
  cudaError_t e = cudaMemsetAsync(buf, 0, sizeof(uint32_t) * lookback_probe_words(), s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(chunk_ctr, 1, 1, s);  // the counter's lowest byte: 1
  if (e != cudaSuccess) return e;
  k_radix_pass<<<1, kSortThreads, 0, s>>>(keys, vals, m, 0, 8, ghist, chunk_ctr, status, keys_out,
                                          vals_out, nullptr, nullptr, nullptr, nullptr, 0, err,
                                          limit_ns);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_cutoff_eval(const CutInst* tab, int ninst, int64_t cut_bins, int64_t slice_bins,
                               const CutoffScratch& ws, int sms, cudaStream_t s) {
  if (ninst <= 0 || cut_bins <= 0) return cudaSuccess;
  if (cut_bins > 0x7fffffff || !ws.err) return cudaErrorInvalidValue;
  const int nb = (int)cut_bins, grid = (nb + 255) / 256;
  // per-key counts and cursors of the order, then the gather's item counter
  cudaError_t e = cudaMemsetAsync(ws.ocount, 0, sizeof(uint32_t) * kCutOcountWords, s);
  if (e != cudaSuccess) return e;
  k_cut_block_totals<<<grid, 256, 0, s>>>(tab, ninst, ws.start, nb, ws.totals, ws.ranges,
                                          ws.ocount);
  k_cut_order_scatter<<<grid, 256, 0, s>>>(tab, ninst, ws.totals, nb, ws.ocount, ws.order);
  // as many CTAs as stay on the GPU, or as there can be items: every block, and
  // three more for each block of a slicing instance that may turn out heavy
  const int64_t ctas = std::min((int64_t)nb + (int64_t)(kSlices - 1) * slice_bins,
                                (int64_t)kCutCtasPerSm * sms);
  if ((e = cudaFuncSetAttribute(k_cutoff, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kCutSmemBytes)) != cudaSuccess)
    return e;
  k_cutoff<<<(unsigned)ctas, kGroups * kGroupThreads, kCutSmemBytes, s>>>(
      tab, ninst, ws.spts, ws.sw, ws.start, ws.order, ws.totals, ws.ranges,
      ws.ocount + 2 * kCutOrderKeys, nb, ws.err);
  note_launches(3);
  return cudaGetLastError();
}

}  // namespace kde
