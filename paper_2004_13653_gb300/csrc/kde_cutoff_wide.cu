// Path (c), product kernels over supports of many cells: 32 x 32-cell tiles.
//
// The gather of kde_cutoff.cu computes 16 x 16-cell blocks: per 32 points a
// warp tabulates 32 factors a point and then adds 256 products a point, eight
// per lane, so half of its instructions make factors and the products are
// bound by their table reads (a float2 and a float4 per eight FMAs; shared memory
// delivers 128 bytes per clock to the registers, broadcasts included).  Over
// a support of many cells a point belongs to few enough 32 x 32 tiles,
// (1 + 2 reach / 32)^2, that four times the block pays: 64 factors a point for
// 1024 products, 32 per lane as 16 packed FMAs for three float4 reads.
//
// A tile's points are the runs of its bin rows in the shared sort, cut into
// pieces of piece_len points by the work list of kde_sparse.cu.  A CTA computes
// one piece: its eight warps take batches of 32 points in turn, each for the
// whole tile.  A warp drops the points of its batch that lie beyond the reach of
// the tile (their factors are zeros) and keeps the others until there are 16;
// then its half-warps make their column and row factors, a point per lane, so
// that only the stores go through shared memory, and the products go into the
// lanes' 8 x 4 cells.  After 32 points those FP32 sums go into the cells'
// (hi, lo) running sums; the warps' sums are added in warp order and the
// pieces' in piece order, so every result is the same in every run, and in a
// batch as on its own.
//
// 1M points x 1000 x 900, reach 40 cells, quartic: 1150 us in 16 x 16 blocks,
// 838 with the factors tabulated a cell per lane (each point read as a
// broadcast), 670 now: the three float4 reads a point keep shared memory's data
// pipe 94% busy, the FMA pipe (a packed FMA is two cycles) 70%.
#include "kde_internal.cuh"
#include "kernel_factors.cuh"

namespace kde {
namespace {

constexpr int kSide = kWideSide;
constexpr int kWarps = 8, kThreads = 32 * kWarps;
constexpr int kBatch = 32;
constexpr int kCellsPerTile = kSide * kSide;
static_assert(kSide == 32, "a lane tabulates one column and one row");

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

// One warp's tables: points within reach that wait for their turn (their x and
// y, hi and lo, and weights), the factors of kStep of them at a time, and the
// running sums of the warp's cells (pair k of lane l, two cells' hi and two
// cells' lo, at run[k][l]).  A row of factors is four floats longer than its 32
// so that the lanes' 16-byte stores, a row each, take all the banks.
constexpr int kStep = 16;
constexpr int kRow = kSide + 4;
struct WarpTables {
  float2 P[2][kBatch + kStep];
  float W[kBatch + kStep];
  __align__(16) float K[2][kStep][kRow];
  float4 run[kCellsPerTile / 64][32];
};
constexpr size_t kSmemBytes = kWarps * sizeof(WarpTables);

// A warp's cells: lane l holds columns cx .. cx + 7 of rows cy .. cy + 3, in
// pairs along x.
struct Cells {
  float2 v[4][4];  // [row][column pair]
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[r][j] = make_float2(0.f, 0.f);
  }
};

// run += acc by two-sums; acc = 0
__device__ __forceinline__ void flush(WarpTables& T, int lane, Cells& acc) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 x = T.run[4 * r + j][lane];
      const float2 a = make_float2(x.x, x.y), b = acc.v[r][j];
      const float2 s = p_add(a, b), bb = p_sub(s, a);
      const float2 lo = p_add(make_float2(x.z, x.w), p_add(p_sub(a, p_sub(s, bb)), p_sub(b, bb)));
      T.run[4 * r + j][lane] = make_float4(s.x, s.y, lo.x, lo.y);
      acc.v[r][j] = make_float2(0.f, 0.f);
    }
}

// A point's factors at a lane's columns and rows.
struct Factors {
  float4 x0, x1, y;
};
__device__ __forceinline__ Factors load_factors(const WarpTables& T, int c, int cx, int cy) {
  Factors f;
  f.x0 = *reinterpret_cast<const float4*>(&T.K[0][c][cx]);
  f.x1 = *reinterpret_cast<const float4*>(&T.K[0][c][cx + 4]);
  f.y = *reinterpret_cast<const float4*>(&T.K[1][c][cy]);
  return f;
}

__device__ __forceinline__ void point_products(const Factors& f, Cells& acc) {
  const float2 x[4] = {make_float2(f.x0.x, f.x0.y), make_float2(f.x0.z, f.x0.w),
                       make_float2(f.x1.x, f.x1.y), make_float2(f.x1.z, f.x1.w)};
  const float y[4] = {f.y.x, f.y.y, f.y.z, f.y.w};
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float2 yy = make_float2(y[r], y[r]);
#pragma unroll
    for (int j = 0; j < 4; ++j) acc.v[r][j] = p_fma(x[j], yy, acc.v[r][j]);
  }
}

// The products of the first m <= kStep waiting points.  Lanes l and l + 16 make
// point l's 32 column and 32 row factors: the offset from cell j is that from
// the tile's first cell plus j times the cell's side (pair_offset).
template <int KID>
__device__ __forceinline__ void step(WarpTables& T, int m, int lane, float2 g0, float cs_hi,
                                     float cs_lo, int cx, int cy, Cells& acc) {
  const int axis = lane >> 4, pt = lane & (kStep - 1);
  if (pt < m) {
    const float2 p = T.P[axis][pt];
    const float w = axis ? T.W[pt] : 1.0f;
    const float2 d0 = pair_offset(g0, p);
    const float dh = d0.x, dl = d0.y;
    float4* row = reinterpret_cast<float4*>(&T.K[axis][pt][0]);
#pragma unroll
    for (int q = 0; q < kSide / 4; ++q) {
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; e += 2) {
        const float2 j = make_float2((float)(4 * q + e), (float)(4 * q + e + 1));
        const float2 u = p_add(p_fma(j, make_float2(cs_hi, cs_hi), make_float2(dh, dh)),
                               p_fma(j, make_float2(cs_lo, cs_lo), make_float2(dl, dl)));
        v[e] = w * kfactor<KID>(u.x);
        v[e + 1] = w * kfactor<KID>(u.y);
      }
      row[q] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
  __syncwarp();
  int c = 0;
  for (; c + 2 <= m; c += 2) {
    const Factors a = load_factors(T, c, cx, cy);
    const Factors b = load_factors(T, c + 1, cx, cy);
    point_products(a, acc);
    point_products(b, acc);
  }
  if (c < m) point_products(load_factors(T, c, cx, cy), acc);
  __syncwarp();  // the tables are consumed
}

// The batches of one warp: points begin + 32 (warp + 8 k) of the tile's runs,
// up to end.
template <int KID>
__device__ __forceinline__ void warp_piece(const TcInst& I, const BinRange& br, int tm, int tn,
                                           uint32_t begin, uint32_t end, int warp, int lane,
                                           WarpTables& T) {
  const float2 g0 = lane < 16 ? I.gxt[tm * kSide] : I.gyt[tn * kSide];
  const float cs_hi = I.cs_hi, cs_lo = I.cs_lo;
  // the tile's reach, widened as the bin ranges are: FP32 coordinates beyond it
  // have a factor of exactly zero at every cell
  const float rr = (float)I.range_reach;
  const float x_lo = (float)((tm * kSide + 0.5) * I.cs) - rr;
  const float x_hi = (float)((tm * kSide + kSide - 0.5) * I.cs) + rr;
  const float y_lo = (float)((tn * kSide + 0.5) * I.cs) - rr;
  const float y_hi = (float)((tn * kSide + kSide - 0.5) * I.cs) + rr;
  const int cx = 8 * (lane & 3), cy = 4 * (lane >> 2);
  const uint32_t lt = (1u << lane) - 1u;

  Cells acc;
  acc.clear();
#pragma unroll
  for (int k = 0; k < kCellsPerTile / 64; ++k) T.run[k][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  int held = 0, waiting = 0;  // points in acc, and in the tables

  RunCursor32 cur;
  cur.init(I.start, I.bin_begin, I.nbx, br);
  constexpr uint32_t kStride = kWarps * kBatch;
  uint32_t v = begin + warp * kBatch + lane;
  float4 pf = make_float4(0.f, 0.f, 0.f, 0.f);
  float wf = 0.f;
  if (v < end) {
    const uint32_t p = cur.map(v);
    pf = I.pts[p];
    wf = I.wts[p];
  }
  for (uint32_t b0 = begin + warp * kBatch; b0 < end; b0 += kStride, v += kStride) {
    const float X = pf.x + pf.y, Y = pf.z + pf.w;
    const bool in = v < end && X >= x_lo && X <= x_hi && Y >= y_lo && Y <= y_hi;
    const uint32_t mask = __ballot_sync(0xffffffffu, in);
    if (in) {
      const int e = waiting + __popc(mask & lt);
      T.P[0][e] = make_float2(pf.x, pf.y);
      T.P[1][e] = make_float2(pf.z, pf.w);
      T.W[e] = wf;
    }
    waiting += __popc(mask);
    __syncwarp();
    if (v + kStride < end) {  // next batch, in flight
      const uint32_t p = cur.map(v + kStride);
      pf = I.pts[p];
      wf = I.wts[p];
    }
    while (waiting >= kStep) {
      if (held == kBatch) {
        flush(T, lane, acc);
        held = 0;
      }
      step<KID>(T, kStep, lane, g0, cs_hi, cs_lo, cx, cy, acc);
      held += kStep;
      waiting -= kStep;
      // the points left, at most 31, move to the front
      float2 px, py;
      float w = 0.f;
      px = py = make_float2(0.f, 0.f);
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
  }
  if (waiting) {
    if (held == kBatch) flush(T, lane, acc);
    step<KID>(T, waiting, lane, g0, cs_hi, cs_lo, cx, cy, acc);
  }
  flush(T, lane, acc);
}

// The work item at schedule position pos: full pieces first (tile by tile),
// then the tiles' short last pieces, longest first.
struct Piece {
  const TcInst* I;
  int tm, tn, pieces;     // the tile, and how many pieces it has
  int64_t k_begin, vend;  // positions in the tile's runs
  int64_t slot;           // the piece's partial tile
};
__device__ __forceinline__ Piece list_piece(const TcInst* __restrict__ tab, int ninst,
                                            const SparseCtl& sp, int pos) {
  const int n_full = (int)__ldg(sp.full_begin + sp.tiles_total);
  int t, p = -1;
  if (pos < n_full) {
    int lo = 0, hi = sp.tiles_total - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if ((int)__ldg(sp.full_begin + mid) <= pos) lo = mid; else hi = mid - 1;
    }
    t = lo;
    p = pos - (int)__ldg(sp.full_begin + t);
  } else {
    t = (int)__ldg(sp.tail_tile + (pos - n_full));
  }
  const int first = (int)__ldg(sp.piece_begin + t);
  Piece r;
  r.pieces = (int)__ldg(sp.piece_begin + t + 1) - first;
  if (p < 0) p = r.pieces - 1;
  int a = 0, b = ninst - 1;
  while (a < b) {
    const int mid = (a + b + 1) >> 1;
    if (tab[mid].tile_begin <= t) a = mid; else b = mid - 1;
  }
  r.I = tab + a;
  const int local = t - r.I->tile_begin;
  r.tm = local % r.I->tiles_m;
  r.tn = local / r.I->tiles_m;
  r.k_begin = (int64_t)p * sp.piece_len;
  r.vend = min((int64_t)__ldg(sp.tile_total + t), r.k_begin + (int64_t)sp.piece_len);
  r.slot = (int64_t)first + p;
  return r;
}

// One CTA per piece; those past the work list return at once (the grid is its
// bound, known on the host).  A tile of one piece is written to the output here,
// the pieces of others to their partial tiles of (hi, lo) sums.
__global__ void __launch_bounds__(kThreads, 2)
    k_cutoff_wide(const TcInst* __restrict__ tab, int ninst, const __grid_constant__ SparseCtl sp,
                  float2* __restrict__ part, CallScalars* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem[];
  WarpTables* tables = reinterpret_cast<WarpTables*>(smem);
  __shared__ BinRange s_br;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // after a timed-out sort its bin starts are not trusted, and a list longer
  // than the partial buffer is an error: compute nothing
  const uint32_t listed = __ldg(sp.piece_begin + sp.tiles_total);
  if (*reinterpret_cast<const volatile int*>(&err->err) & kErrSortTimeout) return;
  if (listed > (uint32_t)sp.max_pieces) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&err->err, kErrBadArg);
    return;
  }
  if (blockIdx.x >= listed) return;
  const Piece pc = list_piece(tab, ninst, sp, blockIdx.x);
  const TcInst& I = *pc.I;
  if (threadIdx.x == 0)
    s_br = tile_bins(I.cs, I.range_reach, I.inv_binw, I.nbx, I.nby, pc.tm, pc.tn, kSide);
  __syncthreads();
  const BinRange br = s_br;
  const uint32_t begin = (uint32_t)pc.k_begin, end = (uint32_t)pc.vend;
  switch (I.kid) {
#define KDE_WIDE(K) \
  case K: warp_piece<K>(I, br, pc.tm, pc.tn, begin, end, warp, lane, tables[warp]); break;
    KDE_WIDE(KDE_UNIFORM)
    KDE_WIDE(KDE_TRIANGULAR)
    KDE_WIDE(KDE_EPANECHNIKOV)
    KDE_WIDE(KDE_QUARTIC)
    KDE_WIDE(KDE_TRIWEIGHT)
    KDE_WIDE(KDE_TRICUBE)
    KDE_WIDE(KDE_COSINE)
#undef KDE_WIDE
    default: return;
  }
  __syncthreads();
  for (int cell = threadIdx.x; cell < kCellsPerTile; cell += kThreads) {
    const int col = cell % kSide, row = cell / kSide;
    // lane (col / 8, row / 4) holds the cell in half col & 1 of pair 4 (row & 3) + (col & 7) / 2
    const int at = ((4 * (row & 3) + (col & 7) / 2) * 32 + (row / 4) * 4 + col / 8) * 4 + (col & 1);
    float2 sum = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float* r = &tables[w].run[0][0].x;
      two_sum_acc(sum, r[at]);
      sum.y += r[at + 2];
    }
    if (pc.pieces == 1) {
      const int x = pc.tm * kSide + col, y = pc.tn * kSide + row;
      if (x < I.nx && y < I.ny) I.part[(int64_t)y * I.nx + x] = (sum.x + sum.y) * I.base_scale;
    } else {
      part[pc.slot * kCellsPerTile + cell] = sum;
    }
  }
}

// The other tiles' output: their pieces' sums, in piece order (none: zeros).
constexpr int kRedThreads = 256;
__global__ void __launch_bounds__(kRedThreads)
    k_wide_reduce(const TcInst* __restrict__ tab, int ninst, SparseCtl sp,
                  const float2* __restrict__ part) {
  const int t = blockIdx.x;
  const int p0 = bounded_piece(sp.piece_begin[t], sp.max_pieces);
  const int p1 = bounded_piece(sp.piece_begin[t + 1], sp.max_pieces);
  if (p1 - p0 == 1) return;
  int a = 0, b = ninst - 1;
  while (a < b) {
    const int mid = (a + b + 1) >> 1;
    if (tab[mid].tile_begin <= t) a = mid; else b = mid - 1;
  }
  const TcInst& I = tab[a];
  const int local = t - I.tile_begin;
  const int cell = blockIdx.y * kRedThreads + threadIdx.x;
  const int x = (local % I.tiles_m) * kSide + cell % kSide;
  const int y = (local / I.tiles_m) * kSide + cell / kSide;
  if (x >= I.nx || y >= I.ny) return;
  float2 sum = make_float2(0.f, 0.f);
  constexpr int kAhead = 8;  // loads in flight; the sums stay in piece order
  for (int p = p0; p < p1; p += kAhead) {
    float2 v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (p + u < p1) v[u] = __ldcs(part + (int64_t)(p + u) * kCellsPerTile + cell);
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (p + u < p1) {
        two_sum_acc(sum, v[u].x);
        sum.y += v[u].y;
      }
  }
  I.part[(int64_t)y * I.nx + x] = (sum.x + sum.y) * I.base_scale;
}

}  // namespace

cudaError_t launch_wide_reduce(const TcInst* tab, int ninst, const SparseCtl& sp, cudaStream_t s) {
  k_wide_reduce<<<dim3(sp.tiles_total, kCellsPerTile / kRedThreads), kRedThreads, 0, s>>>(
      tab, ninst, sp, reinterpret_cast<const float2*>(sp.part));
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_cutoff_wide(const TcInst* tab, int ninst, const SparseCtl& sp, CallScalars* err,
                               cudaStream_t s) {
  if (ninst < 1 || sp.side != kSide || sp.tiles_total < 1 || sp.piece_len < 1 || sp.max_pieces < 1)
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k_cutoff_wide, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemBytes);
  if (e != cudaSuccess) return e;
  float2* part = reinterpret_cast<float2*>(sp.part);
  k_cutoff_wide<<<sp.max_pieces, kThreads, kSmemBytes, s>>>(tab, ninst, sp, part, err);
  note_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return launch_wide_reduce(tab, ninst, sp, s);
}

}  // namespace kde
