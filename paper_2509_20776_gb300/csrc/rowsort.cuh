// The Build step (Sec. 3.1, Algorithm 2's fill pass and the per-row sort): every output row
// takes its source entries, relabelled, and is sorted by column.
//   * Rows of at most TMAX entries (512, or 1024 with the run-time tile shape 1) go in tiles
//     of consecutive rows, k_seg_sort<SsTile / SsTileL>: the tile reads its rows' source
//     entries itself (column, relabel lookup, value), sorts them in shared memory and
//     writes them once.
//   * Rows of TMAX < L <= SS_RUN_MAX entries go alone, read and written the same way:
//     k_seg_sort<SsRunS / SsRunM / SsRun> by their length.
//   * Longer rows are cut by key range, chunk by chunk, into runs of at most SS_RUN_MAX
//     entries (k_long_hist, k_long_scatter and, where a key range can overflow a run,
//     k_split_fine), and the runs sorted by the same kernels.
// Rows that lie in the output already (a sort alone) take the same kernels with the output
// as their source; a gather without a sort is k_gather_chunks.  One pass over the row
// pointer (RowsPartition) finds the tiles' first rows and lists the rows that fit none.
#pragma once

#include <type_traits>

#include "scan.cuh"

namespace sp {

constexpr int SS_HEAVY = 128;                  // default (and smallest) heavy-bucket threshold
constexpr int SS_LEVELS = 3;                   // levels a heavy bucket is bucketed again

// A sort configuration: B threads hold ITEMS entries each of an item of at most CAP = B *
// ITEMS entries, MINB CTAs per SM.  A tile holds the rows whose partition coordinate (the
// row's output position + W for every earlier row) lies in a window of WIN, so at most
// ROWS = WIN / W rows; of those it sorts the rows of at most TMAX entries, as many whole
// rows at a time as fit in CAP (a second round takes what a window's last rows add).
template <int BLOCK_, int ITEMS_, int MINB_, bool TILES_ = false>
struct SsCfg {
  static constexpr int B = BLOCK_, ITEMS = ITEMS_, CAP = B * ITEMS, MINB = MINB_;
  static constexpr int TMAX = CAP / 2, WIN = CAP, W = 4, ROWS = WIN / W;
  static constexpr int RPT = (ROWS + B - 1) / B;  // rows a thread sets up
  static constexpr int WORDS = CAP / 32;   // row-start bitmap words
  static constexpr bool kTiles = TILES_;   // items are tiles (else: single runs)
  static_assert((CAP & (CAP - 1)) == 0, "a row's window by a shift");
  static_assert(B % 32 == 0 && B * MINB <= 2048, "whole warps, resident CTAs");
  static_assert(CAP <= 4096 && ROWS < 65536 / 2, "packed positions and counts");
};
// Shapes by measurement (R-MAT scale 25, 1.05 G entries, whole permutation with the long
// rows' split of one CTA per row; gather and sort apart: 21.0 ms):
// few entries per thread and many threads -- 256 x 4 at 5 CTAs per SM 17.6 ms, 6 CTAs 18.4,
// 4 CTAs 18.4, 128 x 8 at 8 CTAs 24.0, 64 x 16 31 (longer unrolled code, and the lookups of a
// thread in flight at once evict one another's lines from the L1 that shared memory leaves).
using SsTile = SsCfg<256, 4, 5, true>;   // tiles of rows of at most 512 entries
using SsTileL = SsCfg<256, 8, 4, true>;  // tile shape 1: rows of at most 1024 entries (8-byte values: 3 CTAs)
using SsRun = SsCfg<512, 8, 2>;          // single runs of at most 4096 entries
using SsRunM = SsCfg<256, 8, 4>;         // of at most 2048
using SsRunS = SsCfg<256, 4, 5>;         // of at most 1024
constexpr int SS_SMALL_RUN = SsRunS::CAP, SS_MID_RUN = SsRunM::CAP;
constexpr int SS_RUN_MAX = 4096;           // longest row sorted alone
constexpr long long SS_ONE_LAUNCH = 1 << 17;  // sorts of at most this many entries take one launch for all runs
static_assert(SsRun::CAP == SS_RUN_MAX, "run capacity");
static_assert(SsTile::W == SsTileL::W && SsTile::WIN <= SsTileL::WIN, "one bound on the number of tiles");

// Where a run's entries are: in the output arrays or in the temporary arrays (keys as
// uint32, values) at the run's output offset, or still at the row's source.
enum BufId : int { BUF_TEMP = 0, BUF_OUT = 1, BUF_SRC = 2 };

struct FinalEntry {  // a run of at most SS_RUN_MAX entries left to sort
  long long off;     // output offset
  int len;
  int buf;
  long long row;     // BUF_SRC: the output row
};
// The run lists: slices of one array, by what sorts them -- runs of at most SS_WARP_RUN
// entries a warp (k_sort_warp_runs; only where a caller queues them: an empty slice passes
// them on), of at most SS_SMALL_RUN, SS_MID_RUN, SS_RUN_MAX entries a CTA of SsRunS,
// SsRunM, SsRun -- each with its own count and bound.
constexpr int SS_WARP_RUN = 128;
constexpr int RUNS_BAD = 8;    // of the counters: the row pointer does not ascend (RowsPartition)
struct RunLists {
  FinalEntry* list;
  unsigned* n;               // 4 counts (the first of the counters)
  long long c0, c1, c2, c3;  // capacity of each slice
  __device__ __forceinline__ FinalEntry* slice(int k) const { return list + (k > 0 ? c0 : 0) + (k > 1 ? c1 : 0) + (k > 2 ? c2 : 0); }
  __device__ __forceinline__ long long cap(int k) const { return k == 0 ? c0 : k == 1 ? c1 : k == 2 ? c2 : c3; }
};
__device__ __forceinline__ void queue_run(const RunLists& rl, const FinalEntry& e, DevStatus* st, long long err) {
  const int k = e.len <= SS_WARP_RUN && rl.c0 > 0 ? 0 : e.len <= SS_SMALL_RUN ? 1 : e.len <= SS_MID_RUN ? 2 : 3;
  const unsigned q = atomicAdd(rl.n + k, 1u);
  if (q < rl.cap(k)) rl.slice(k)[q] = e;
  else dev_fail(st, SP_ERR_INTERNAL, err);
}
struct HugeEntry {     // a run longer than SS_RUN_MAX
  long long off;       // output offset
  long long len;
  long long row;       // BUF_SRC: the output row
  int buf;             // where its entries are
  unsigned arrived;    // chunks whose histogram is written (k_long_hist)
  int bad;             // a key outside the matrix (reported): not cut
  int pad;
};
struct LongChunk {     // SL_CH entries of a row longer than SS_RUN_MAX
  unsigned huge;       // its slot of the huge list
  unsigned chunk;
};
constexpr int SL_CH = 4096;

// What a pass over the output rows queues for the sort: rows of at most SS_RUN_MAX entries
// as runs, longer ones for the key-range split, chunk by chunk.  The capacities bound what
// nnz entries can hold (huge_cap rows longer than SS_RUN_MAX, lchunk_cap chunks of them).  Rows
// that lie on one another (a row pointer that does not ascend) can hold more: such a row is
// reported, and the chunks it has already taken from the list are marked as nobody's.
constexpr unsigned SL_NONE = 0xFFFFFFFFu;
struct SortLists {
  RunLists runs;
  HugeEntry* huge;
  unsigned* huge_n;
  long long huge_cap;
  LongChunk* lchunk;
  unsigned* lchunk_n;
  long long lchunk_cap;
};
__device__ __forceinline__ void queue_row(const SortLists& sl, long long off, long long L, int buf, long long row,
                                          DevStatus* st, long long err) {
  if (L <= SS_RUN_MAX) {
    queue_run(sl.runs, FinalEntry{off, int(L), buf, row}, st, err);
    return;
  }
  const unsigned h = atomicAdd(sl.huge_n, 1u), nc = unsigned((L + SL_CH - 1) / SL_CH);
  const unsigned c = atomicAdd(sl.lchunk_n, nc);
  const bool fits = h < sl.huge_cap && (long long)c + nc <= sl.lchunk_cap;
  if (fits) sl.huge[h] = HugeEntry{off, L, row, buf, 0u, 0, 0};
  else dev_fail(st, SP_ERR_INTERNAL, err);
  for (long long k = 0; k < nc && c + k < sl.lchunk_cap; ++k) sl.lchunk[c + k] = LongChunk{fits ? h : SL_NONE, unsigned(k)};
}

constexpr int GC_BLOCK = 256;                  // gather: threads per CTA
constexpr int GC_CH = 4096;                    // gather: output positions per CTA
constexpr int GC_ITEMS = GC_CH / GC_BLOCK;
constexpr int GC_MINB = 5;                     // gather: resident CTAs per SM (persistent grid)
constexpr int GC_H = 4;                        // gather: positions a thread loads before it stores

// ---- partition ----------------------------------------------------------------------
// Row r has the coordinate c(r) = vp[r] + W * r; tile t holds the rows with c(r) in
// [t * 2^wlog, (t + 1) * 2^wlog): a closed form of the row pointer, so no scan of weights is
// needed and the number of tiles is known on the host (a window inside a longer row is an
// empty tile).  Gather chunk k starts at the row holding output position k * GC_CH.
// The row pointer is clamped to [0, nnz], so no run or chunk reaches outside the output
// arrays.  It need not ascend: a scan that gave up waiting (SP_ERR_TIMEOUT) takes the prefix it
// missed as 0, so the pointer drops, or jumps, where one of the scan's own tiles ends, and some
// of tile_first and chunk_first stays unwritten; a caller's own row pointer may hold anything.
// The scan or k_partition marks either in *bad, and the kernels that go by the pointer from row
// to row (tiles, gather) then do nothing; the rows listed here are each of one value and its
// successor, so they are sound by themselves.  (A test of the rows of every tile instead cost
// 2 to 3 % of a permutation of rows of 8 to 32.)
struct RowsPartition {
  long long nrows, nnz;
  long long ntiles;         // tile_first holds ntiles + 1 entries
  long long* tile_first;    // null: no tiles (nothing is sorted)
  long long nchunks;
  long long* chunk_first;   // null: no gather chunks
  SortLists lists;          // rows that fit no tile
  int buf;                  // where the rows' entries are: BUF_SRC or BUF_OUT
  int wlog, tmax;           // the tile shape's window (its logarithm) and longest row
  unsigned* bad;            // cleared before; null: nothing goes by it
  DevStatus* st;
  // row r at output positions [o0, o1), 0 <= o0
  __device__ void operator()(long long r, long long o0, long long o1) const {
    o0 = o0 < nnz ? o0 : nnz;
    o1 = o1 < nnz ? o1 : nnz;
    const long long L = o1 - o0;
    if (tile_first) {
      constexpr int W = SsTile::W;
      if (r == 0)  // (a row pointer may start above 0)
        for (long long t = 0; t <= (o0 >> wlog) && t < ntiles; ++t) tile_first[t] = 0;
      // the tiles that start after this row: their first row is r + 1
      long long t = ((o0 + W * r) >> wlog) + 1, t_hi = (o1 + W * (r + 1)) >> wlog;
      if (r + 1 == nrows || t_hi > ntiles) t_hi = ntiles;
      for (; t <= t_hi; ++t) tile_first[t] = r + 1;
      if (L > tmax) queue_row(lists, o0, L, buf, r, st, -15);
    }
    if (chunk_first && L > 0) {
      long long k_hi = (unsigned long long)(o1 - 1) / GC_CH;
      if (k_hi > nchunks - 1) k_hi = nchunks - 1;
      for (long long k = (unsigned long long)(o0 + GC_CH - 1) / GC_CH; k <= k_hi; ++k) chunk_first[k] = r;
    }
    if (chunk_first && r + 1 == nrows)  // none, unless the lengths do not add up to nnz
      for (long long k = (unsigned long long)(o1 + GC_CH - 1) / GC_CH; k < nchunks; ++k) chunk_first[k] = nrows;
  }
};

template <int kDummy = 0>
__global__ void k_partition(RowsPartition part, const long long* __restrict__ vp) {
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < part.nrows;
       r += (long long)gridDim.x * blockDim.x) {
    long long o0 = vp[r], o1 = vp[r + 1];
    if (o0 < 0 || o1 < o0 || o1 > part.nnz) {  // only a caller's own row pointer
      dev_fail(part.st, SP_ERR_NOT_CANONICAL, r);
      if (part.bad) *part.bad = 1u;
    }
    part(r, o0 < 0 ? 0 : o0, o1 < 0 ? 0 : o1);
  }
}

// Scan output of a row pointer (vp, mirrored into a typed array) that partitions its rows
// on the way.
template <class T>
struct StorePartition {
  long long* vp;
  T* out;  // may be null
  RowsPartition part;
  DevStatus* st;
  __device__ void operator()(long long i, long long v, long long vn) const {
    vp[i] = v;
    if (out) {
      if (sizeof(T) == 4 && v > 0x7fffffffll) dev_fail(st, SP_ERR_OVERFLOW, i);
      out[i] = T(v);
    }
    if (i < part.nrows) part(i, v, vn);
  }
};

// ---- conflict-free block scans over shared arrays ------------------------------------------
// Each warp owns a contiguous segment of n / (B / 32) entries and walks it 32 entries at a
// time (lane l reads word base + l: no bank conflicts), carrying its running value; the
// warps' segment totals are combined by one warp.  n must be a multiple of B.
template <int B>
__device__ uint32_t smem_excl_sum_w(uint32_t* a, int n, uint32_t* tmp) {
  constexpr int NW = B / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, seg = n / NW;
  uint32_t* s = a + w * seg;
  uint32_t tot = 0;
  for (int x = lane; x < seg; x += 32) tot += s[x];
  tot = warp_sum(tot);
  if (lane == 0) tmp[w] = tot;
  __syncthreads();
  if (w == 0) {
    const uint32_t v = lane < NW ? tmp[lane] : 0u;
    const uint32_t inc = warp_incl_sum(v);
    if (lane < NW) tmp[lane] = inc - v;
    if (lane == NW - 1) tmp[NW] = inc;
  }
  __syncthreads();
  uint32_t carry = tmp[w];
  for (int x = lane; x < seg; x += 32) {
    const uint32_t v = s[x];
    const uint32_t inc = warp_incl_sum(v);
    s[x] = carry + inc - v;
    carry += __shfl_sync(0xffffffffu, inc, 31);
  }
  const uint32_t total = tmp[NW];
  __syncthreads();
  return total;
}

template <int B>
__device__ void smem_incl_max_w(uint32_t* a, int n, uint32_t* tmp) {
  constexpr int NW = B / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, seg = n / NW;
  uint32_t* s = a + w * seg;
  uint32_t mx = 0;
  for (int x = lane; x < seg; x += 32) mx = s[x] > mx ? s[x] : mx;
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) tmp[w] = mx;
  __syncthreads();
  if (w == 0) {
    const uint32_t v = lane < NW ? tmp[lane] : 0u;
    uint32_t inc = warp_incl_max(v);
    uint32_t ex = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) ex = 0u;
    if (lane < NW) tmp[lane] = ex;
  }
  __syncthreads();
  uint32_t carry = tmp[w];
  for (int x = lane; x < seg; x += 32) {
    const uint32_t inc = warp_incl_max(s[x]);
    const uint32_t r = inc > carry ? inc : carry;
    s[x] = r;
    carry = __shfl_sync(0xffffffffu, r, 31);
  }
  __syncthreads();
}

// ---- sources -------------------------------------------------------------------------
// Where an output row's entries are and how their columns are relabelled:
//   struct Gs {
//     using CI, VT;                            // column / value words
//     const long long* srcs() const;           // source start of every output row (packed
//                                              // with whatever view() needs)
//     GsView<CI, VT> view(long long src, long long L) const;  // the row's first entry
//     uint32_t map(unsigned mid, uint32_t c) const;  // new column (0xFFFFFFFF: c lies
//                                              // outside the matrix)
//     CI map_ci(unsigned mid, CI c) const;     // the same in the column's own width
//   };
template <class CI, class VT>
struct GsView {
  const CI* c;   // null: the row's source is inconsistent (a library bug)
  const VT* v;
  unsigned mid;  // which relabelling
};
// A stored column as a 32-bit key; a 64-bit one outside [0, 2^32) becomes the key
// 0xFFFFFFFF, which is outside every matrix that the sort takes.
__device__ __forceinline__ uint32_t ss_key(int32_t c) { return uint32_t(c); }
__device__ __forceinline__ uint32_t ss_key(uint32_t c) { return c; }
__device__ __forceinline__ uint32_t ss_key(int64_t c) {
  return (uint64_t(c) >> 32) ? 0xFFFFFFFFu : uint32_t(c);
}

// Rows that lie in the output already, as the source of the sort.
template <class CIt, class VTt>
struct RowsInPlace {
  using CI = CIt;
  using VT = VTt;
  static constexpr bool kInPlace = true;
  const long long* vp;
  const CI* c_;
  const VT* v_;
  __device__ const long long* srcs() const { return vp; }
  __device__ GsView<CI, VT> view(long long src, long long) const { return {c_ + src, v_ + src, 0u}; }
  __device__ uint32_t map(unsigned, uint32_t c) const { return c; }
};
template <class Gs, class = void>
struct in_place : std::false_type {};
template <class Gs>
struct in_place<Gs, std::void_t<decltype(Gs::kInPlace)>> : std::bool_constant<Gs::kInPlace> {};

// ---- gather without a sort ----------------------------------------------------------------
// Chunk k is GC_CH consecutive output positions, starting inside row chunk_first[k].  bad (may
// be null): the row pointer does not ascend (see RowsPartition).
template <class Gs>
__global__ void __launch_bounds__(GC_BLOCK, GC_MINB) k_gather_chunks(Gs gs, const long long* __restrict__ vp,
                                                            long long nrows, long long total,
                                                            const long long* __restrict__ chunk_first,
                                                            long long nchunks, const unsigned* __restrict__ bad,
                                                            typename Gs::CI* __restrict__ out_col,
                                                            typename Gs::VT* __restrict__ out_val, DevStatus* st) {
  using CI = typename Gs::CI;
  using VT = typename Gs::VT;
  constexpr int B = GC_BLOCK, ITEMS = GC_ITEMS;
  __shared__ uint32_t owner[GC_CH];
  __shared__ GsView<CI, VT> r_v[B];  // the row's source
  __shared__ long long r_o0[B];
  __shared__ long long r_o1[B];
  __shared__ uint32_t tmp32[B / 32 + 1];
  __shared__ long long s_last;  // output end of the batch's last row
  __shared__ int s_single;      // the batch's first row covers the whole chunk
  const int t = threadIdx.x;
  // row r's output range [o0, o1) and source start
  auto setup = [&](long long r, long long& a, long long& b, long long& s) {
    a = total;
    b = total;
    s = 0;
    if (r < nrows) {
      a = vp[r];
      b = vp[r + 1];
      s = gs.srcs()[r];
    }
  };
  // persistent: chunks blockIdx.x, + gridDim.x, ...; a batch is B consecutive rows.  The
  // next batch's row setup is loaded while this batch's entries are in flight.
  long long c = blockIdx.x;
  if (c >= nchunks) return;
  const bool skip = bad && *bad != 0u;  // (read beside the first chunk's row)
  long long rb = chunk_first[c];
  if (skip) return;
  long long o0, o1, so;
  setup(rb + t, o0, o1, so);
  for (;;) {
    const long long c0 = c * (long long)GC_CH, c1 = c0 + GC_CH < total ? c0 + GC_CH : total;
    const long long cn = c + gridDim.x;
    const long long rb_next_chunk = cn < nchunks ? chunk_first[cn] : 0;
    bool active = rb + t < nrows && o1 > o0 && o1 > c0 && o0 < c1;
    if (active) {
      r_v[t] = gs.view(so, o1 - o0);
      if (!r_v[t].c) {
        dev_fail(st, SP_ERR_INTERNAL, -13);
        active = false;
      }
      r_o0[t] = o0;
      r_o1[t] = o1;
    }
    if (t == B - 1) s_last = o1;
    if (t == 0) s_single = active && o0 <= c0 && o1 >= c1;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) owner[t + j * B] = 0;
    __syncthreads();
    // a chunk inside one long row (most of a long row's chunks) needs no owner search
    const bool single = s_single;
    if (!single) {
      if (active) owner[(o0 > c0 ? o0 : c0) - c0] = uint32_t(t + 1);
      __syncthreads();
      smem_incl_max_w<B>(owner, GC_CH, tmp32);
    }
    // the chunk ends with this batch once its last row reaches the end of the chunk
    const bool last_batch = rb + B - 1 >= nrows - 1 || s_last >= c1;
    const bool more = !last_batch || cn < nchunks;
    const long long rb_next = last_batch ? rb_next_chunk : rb + B;
    long long n0 = 0, n1 = 0, ns = 0;
    if (more) setup(rb_next + t, n0, n1, ns);
    // all loads, then all stores (the compiler cannot move stores above later loads)
    constexpr int H = GC_H;
#pragma unroll
    for (int h = 0; h < ITEMS; h += H) {
      CI cv[H];
      VT v[H];
      int kk[H];
      long long off[H];
      bool ok[H];
#pragma unroll
      for (int u = 0; u < H; ++u) {
        const int x = t + (h + u) * B;
        const long long g = c0 + x;
        const int ow = single ? 1 : int(owner[x]);
        ok[u] = false;
        off[u] = 0;
        kk[u] = 0;
        if (g < c1 && ow > 0) {
          const int k = ow - 1;
          const long long o = r_o0[k];
          // positions past this batch of rows belong to the next batch
          if (g >= o && g < r_o1[k]) {
            ok[u] = true;
            kk[u] = k;
            off[u] = g - o;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < H; ++u) cv[u] = ok[u] ? ld_stream(r_v[kk[u]].c + off[u]) : CI(0);
#pragma unroll
      for (int u = 0; u < H; ++u)
        if (ok[u]) v[u] = ld_stream(r_v[kk[u]].v + off[u]);
#pragma unroll
      for (int u = 0; u < H; ++u)
        if (ok[u]) cv[u] = gs.map_ci(r_v[kk[u]].mid, cv[u]);
#pragma unroll
      for (int u = 0; u < H; ++u) {
        if (!ok[u]) continue;
        const long long g = c0 + t + (h + u) * B;
        st_stream(out_col + g, cv[u]);
        st_stream(out_val + g, v[u]);
      }
    }
    __syncthreads();
    if (!more) break;
    if (last_batch) c = cn;
    rb = rb_next;
    o0 = n0;
    o1 = n1;
    so = ns;
  }
}

// ---- approximate square-root bucketing of the row sort -----------------------------------
// Bucket of key k in a row of L entries: L buckets spaced evenly in an approximate square
// root of k over the row's key range [0, kmax].  The root is the exponent-halving bit trick
// on the float of k (exact at even powers of two, up to 6% high in between): monotone in k
// (every step is), so buckets stay in key order; the scale L / root(kmax) maps [0, kmax]
// onto the L buckets.  The square root keeps buckets balanced both for uniformly relabelled
// columns and for labels crowded at the low end (degree-descending orderings).
__device__ __forceinline__ float ss_root(uint32_t k) {
  return __uint_as_float((__float_as_uint(__uint2float_rn(k)) >> 1) + 0x1FC00000u);
}
// 1 / root(kmax): the scale of a range [0, kmax] over L buckets is L * ss_inv_root(kmax)
__device__ __forceinline__ float ss_inv_root(uint32_t kmax) { return kmax ? 1.0f / ss_root(kmax) : 0.0f; }
// bucket of `key` given the row's scale and last bucket L - 1
__device__ __forceinline__ uint32_t ss_bucket(uint32_t key, float scale, uint32_t last) {
  const uint32_t b = __float2uint_rz(ss_root(key) * scale);
  return b < last ? b : last;
}

// ---- key-range split of long rows ------------------------------------------------------
// A row of more than SS_RUN_MAX entries is cut by key into runs of at most SS_RUN_MAX
// entries, chunk by chunk of SL_CH entries so that a hub row is spread over the chip (one
// CTA per row took up to 2.4 ms for a row of 640 K entries, and set the time of this phase
// on every power-law matrix of a few M entries):
//   k_long_hist    reads a chunk (at the row's source, relabelled, its keys written to the
//                  row's place in the output; or in the output already) and counts its keys
//                  in 2^10 buckets evenly spaced over [0, 2^key_bits).  The CTA that
//                  finishes a row's last chunk adds up the counts and forms groups:
//                  consecutive small buckets whose starts fall in one GROUP_CAP window are
//                  one run; a bucket of more than GROUP_CAP entries is a run of its own,
//                  or (more than SS_RUN_MAX entries) goes to the fine split.
//                  A row whose counts do not add up to its length is reported and left out:
//                  its entries were outside the matrix, or another row lies on it (a row
//                  pointer that does not ascend), so its groups could reach past its end.
//   k_long_scatter moves a chunk's entries to their groups in the temporary arrays: staged
//                  in shared memory by group, then each group's share written as one piece
//                  at a place taken from the group's cursor.
//   k_split_fine   one CTA per oversized bucket (skewed keys): 2^13 buckets over the
//                  bucket's own [min, max] keys, from the temporary to the output arrays.
//                  A coarse bucket spans 2^(key_bits - 10) <= 2^22 keys, so a fine bucket
//                  spans at most 2^9 < SS_RUN_MAX keys: with keys unique within a row it
//                  holds fewer than SS_RUN_MAX entries and no third split is needed; with
//                  key_bits <= 22 no coarse bucket can be oversized and it is not launched.
//                  (Only keys that repeat within a row, which no canonical matrix has, make a
//                  bucket larger: SP_ERR_INTERNAL, from k_long_hist where no fine split follows.)
// The runs are then sorted by k_seg_sort.
constexpr int SL_NBL = 10, SL_NB = 1 << SL_NBL;
constexpr int SL_HB = 256, SL_HMINB = 5;  // k_long_hist
constexpr int SL_SB = 512;                // k_long_scatter
template <class VT>
constexpr int sl_sminb() { return sizeof(VT) == 4 ? 3 : 2; }
constexpr int SF_NBL = 13, SF_B = 512, SF_MINB = 2, SF_U = 4;  // k_split_fine
constexpr int SS_RUN_LOG = 12;             // SS_RUN_MAX = 2^SS_RUN_LOG
static_assert((1 << SS_RUN_LOG) == SS_RUN_MAX, "run capacity is a power of two");
static_assert(32 - SL_NBL - SF_NBL <= SS_RUN_LOG, "fine-split buckets fit a run");
// whether a coarse bucket can hold more than SS_RUN_MAX distinct keys
__host__ __device__ constexpr bool fine_split_follows(int key_bits) { return key_bits > SL_NBL + SS_RUN_LOG; }
constexpr int GROUP_CAP = SS_SMALL_RUN;    // small buckets grouped up to this start window: runs of at most SS_MID_RUN
// A row's groups: at most one per GROUP_CAP window of starts, one per bucket of more than
// GROUP_CAP entries and one after each such bucket: 3 L / GROUP_CAP + 1 < L / SL_GSLOT - 1
// for L > SS_RUN_MAX, so a row's cursors fit the slots [off / SL_GSLOT, (off + L) / SL_GSLOT).
constexpr int SL_GSLOT = 256;
static_assert(GROUP_CAP == 4 * SL_GSLOT && SS_RUN_MAX > 3 * GROUP_CAP, "cursor slots");
// A chunk's histogram (SL_NB 16-bit counts) goes to its row's part of the temporary keys,
// which nothing else uses before the scatter: ceil(L / SL_CH) * SL_NB / 2 <= L words.
static_assert(SL_CH / (SL_NB / 2) >= 2, "chunk histograms fit the temporary keys");

// The group of bucket 32 w + lane of a long row, minus none before the first: starts = lane's
// word of the bitmap of the buckets that start a group, before = the starts in earlier words (a
// warp holds the bitmap, one word per lane).  All lanes call it.
static_assert(SL_NB == 32 * 32, "a warp holds a row's bitmap");
__device__ __forceinline__ uint32_t group_of_bucket(uint32_t starts, uint32_t before, int w) {
  const int lane = threadIdx.x & 31;
  const uint32_t b = __shfl_sync(0xffffffffu, starts, w), p = __shfl_sync(0xffffffffu, before, w);
  return p + __popc(b & (0xFFFFFFFFu >> (31 - lane))) - 1u;
}

// Groups of a split: hist (exclusive starts of nb buckets, SIZE of them scanned, the rest
// empty; total L) -> a bucket is big, or the head of a group.  All threads of the CTA call
// it; prv and nxb hold SIZE words.  Afterwards emit(x, big, start, end) is called for every
// big bucket and every group (end: the next group's or big bucket's start).
template <int B, int SIZE, class Emit>
__device__ void split_groups(const uint32_t* hist, uint32_t* prv, uint32_t* nxb, uint32_t* tmp32, int nb, uint32_t L,
                             Emit&& emit) {
  const int t = threadIdx.x;
  // bucket x holds [hist[x], end(x)); bucket order is key order
  auto bend = [&](int x) { return x + 1 < nb ? hist[x + 1] : L; };
  // previous non-empty bucket (inclusive max-scan of x+1 over non-empty buckets)
  for (int x = t; x < SIZE; x += B) prv[x] = (x < nb && bend(x) > hist[x]) ? uint32_t(x + 1) : 0u;
  __syncthreads();
  smem_incl_max_w<B>(prv, SIZE, tmp32);
  // A bucket of more than GROUP_CAP entries ("big") stands alone; a small non-empty bucket
  // starts a new group ("head") unless the previous non-empty bucket is small and starts in
  // the same GROUP_CAP window.
  auto kind = [&](int x, bool& big, bool& head) {
    const uint32_t sb = hist[x], cc = x < nb ? bend(x) - sb : 0u;
    big = cc > uint32_t(GROUP_CAP);
    head = false;
    if (cc > 0 && !big) {
      const uint32_t pv = x > 0 ? prv[x - 1] : 0u;
      if (pv == 0) {
        head = true;
      } else {
        const int y = int(pv) - 1;
        head = bend(y) - hist[y] > uint32_t(GROUP_CAP) || (hist[y] / GROUP_CAP) != (sb / GROUP_CAP);
      }
    }
  };
  // next group boundary after each bucket: suffix min of boundary starts, as a prefix
  // max over the reversed array of (L - start)
  for (int x = t; x < SIZE; x += B) {
    bool big, head;
    kind(x, big, head);
    nxb[SIZE - 1 - x] = (big || head) ? L - hist[x] : 0u;
  }
  __syncthreads();
  smem_incl_max_w<B>(nxb, SIZE, tmp32);
  for (int x = t; x < SIZE; x += B) {
    bool big, head;
    kind(x, big, head);
    if (!big && !head) continue;
    const uint32_t nx = (x + 1 < SIZE) ? nxb[SIZE - 1 - (x + 1)] : 0u;
    emit(x, big, hist[x], big ? bend(x) : (nx ? L - nx : L));
  }
}

template <class Gs>
__global__ void __launch_bounds__(SL_HB, SL_HMINB)
    k_long_hist(Gs gs, SortLists sl, uint32_t* __restrict__ tkey, typename Gs::CI* __restrict__ out_col,
                uint32_t* __restrict__ gstart, uint32_t* __restrict__ cursor, HugeEntry* __restrict__ nxt,
                unsigned* nxt_n, long long nxt_cap, int key_bits, DevStatus* st) {
  using CI = typename Gs::CI;
  constexpr int B = SL_HB, NB = SL_NB, ITEMS = SL_CH / B, H = 4;
  __shared__ uint32_t hist[NB], prv[NB], nxb[NB];
  __shared__ uint32_t tmp32[B / 32 + 1];
  __shared__ int s_last;
  __shared__ unsigned long long s_total;
  const int t = threadIdx.x;
  const uint32_t kmax = key_bits >= 32 ? 0xFFFFFFFFu : (1u << key_bits) - 1u;
  const int nbl = key_bits < SL_NBL ? key_bits : SL_NBL, sh = key_bits - nbl, nb = 1 << nbl;
  long long n = *sl.lchunk_n;
  if (n > sl.lchunk_cap) n = sl.lchunk_cap;
  for (long long k = blockIdx.x; k < n; k += gridDim.x) {
    const LongChunk lc = sl.lchunk[k];
    if (lc.huge == SL_NONE) continue;
    HugeEntry* const hp = sl.huge + lc.huge;
    const long long off = hp->off, L = hp->len, e0 = (long long)lc.chunk * SL_CH;
    const int len = L - e0 < SL_CH ? int(L - e0) : SL_CH;
    const unsigned nc = unsigned((L + SL_CH - 1) / SL_CH);
    for (int x = t; x < NB; x += B) hist[x] = 0;
    if (t == 0) s_total = 0;
    __syncthreads();
    const bool here = in_place<Gs>::value || hp->buf != BUF_SRC;
    GsView<CI, typename Gs::VT> gv{out_col + off, nullptr, 0u};
    if (!here) gv = gs.view(gs.srcs()[hp->row], L);
    bool bad = false;
    if (!gv.c) {
      if (t == 0) dev_fail(st, SP_ERR_INTERNAL, -13);
      bad = true;
    } else {
      CI* const oc = out_col + off + e0;
      const CI* const cp = gv.c + e0;
#pragma unroll
      for (int h = 0; h < ITEMS; h += H) {
        uint32_t key[H];
#pragma unroll
        for (int u = 0; u < H; ++u) {
          const int x = t + (h + u) * B;
          key[u] = x < len ? ss_key(ld_stream(cp + x)) : 0u;
        }
        if (!here) {
#pragma unroll
          for (int u = 0; u < H; ++u) key[u] = gs.map(gv.mid, key[u]);
        }
#pragma unroll
        for (int u = 0; u < H; ++u) {
          const int x = t + (h + u) * B;
          if (x >= len) continue;
          if (!here) st_stream(oc + x, CI(key[u]));
          if (key[u] <= kmax) {
            atomicAdd(&hist[key[u] >> sh], 1u);
          } else {  // a column outside [0, ncols)
            dev_fail(st, SP_ERR_INDEX_RANGE, off + e0 + x);
            bad = true;
          }
        }
      }
    }
    if (bad) hp->bad = 1;
    __syncthreads();
    uint32_t* const ch = tkey + off;  // chunk c's histogram at c * NB / 2
    for (int w = t; w < NB / 2; w += B)
      __stcg(ch + (long long)lc.chunk * (NB / 2) + w, hist[2 * w] | (hist[2 * w + 1] << 16));
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(&hp->arrived, 1u) == nc - 1;
    __syncthreads();
    if (!s_last) continue;
    // the row's last chunk: add up the counts and form the groups
    __threadfence();
    if (__ldcg(&hp->bad)) continue;  // uniform: written before the last arrival
    unsigned long long mine = 0;
    for (int w = t; w < NB / 2; w += B) {
      uint32_t lo = 0, hi = 0;
#pragma unroll 4
      for (unsigned c = 0; c < nc; ++c) {
        const uint32_t v = __ldcg(ch + (long long)c * (NB / 2) + w);
        lo += v & 0xFFFFu;
        hi += v >> 16;
      }
      hist[2 * w] = lo;
      hist[2 * w + 1] = hi;
      mine += (unsigned long long)lo + hi;
    }
    mine = warp_sum(mine);
    if ((t & 31) == 0) atomicAdd(&s_total, mine);
    __syncthreads();
    const bool whole = s_total == (unsigned long long)L;
    __syncthreads();  // s_total is cleared for the next chunk
    if (!whole) {
      if (t == 0) {
        dev_fail(st, SP_ERR_INTERNAL, -5);
        hp->bad = 1;
      }
      continue;
    }
    smem_excl_sum_w<B>(hist, NB, tmp32);
    uint32_t* const cur = cursor + off / SL_GSLOT;
    split_groups<B, NB>(hist, prv, nxb, tmp32, nb, uint32_t(L), [&](int, bool big, uint32_t s, uint32_t e) {
      if (e - s <= uint32_t(SS_RUN_MAX)) {
        queue_run(sl.runs, FinalEntry{off + s, int(e - s), BUF_TEMP, 0}, st, -6);
      } else if (!fine_split_follows(key_bits)) {  // repeated keys
        dev_fail(st, SP_ERR_INTERNAL, -7);
      } else {
        const unsigned q = atomicAdd(nxt_n, 1u);  // the fine split finds its key range itself
        if (q < nxt_cap) nxt[q] = HugeEntry{off + s, (long long)(e - s), 0, BUF_TEMP, 0u, 0, 0};
        else dev_fail(st, SP_ERR_INTERNAL, -7);
      }
    });
    __syncthreads();  // prv has been read
    // the buckets that start a group, for the scatter, and every group's cursor
    uint32_t* const gs_bits = gstart + (long long)lc.huge * (NB / 32);
    for (int x = t; x < NB; x += B) {
      const uint32_t a = nxb[NB - 1 - x], b = x + 1 < NB ? nxb[NB - 1 - (x + 1)] : 0u;
      const uint32_t bits = __ballot_sync(0xffffffffu, a != b);  // the suffix minimum changes exactly at a start
      if ((x & 31) == 0) prv[x >> 5] = gs_bits[x >> 5] = bits;
    }
    __syncthreads();
    const uint32_t starts = prv[t & 31], count = __popc(starts), before = warp_incl_sum(count) - count;
    for (int x = t; x < NB; x += B) {
      const uint32_t g = group_of_bucket(starts, before, x >> 5);
      if ((prv[x >> 5] >> (x & 31)) & 1u) cur[g] = hist[x];
    }
    __syncthreads();
  }
}

template <class VT>
constexpr size_t long_scatter_smem() {
  return size_t(SL_NB) * (4 + 4 + 2) + size_t(SL_CH) * (4 + sizeof(VT));
}
template <class Gs>
__global__ void __launch_bounds__(SL_SB, sl_sminb<typename Gs::VT>())
    k_long_scatter(Gs gs, SortLists sl, uint32_t* __restrict__ tkey, typename Gs::VT* __restrict__ tval,
                   const typename Gs::CI* __restrict__ out_col, const typename Gs::VT* __restrict__ out_val,
                   const uint32_t* __restrict__ gstart, uint32_t* __restrict__ cursor, int key_bits) {
  using VT = typename Gs::VT;
  constexpr int B = SL_SB, NB = SL_NB, U = SL_CH / B;
  extern __shared__ __align__(16) unsigned char smem[];
  VT* sv = reinterpret_cast<VT*>(smem);                        // the chunk's values by group
  uint32_t* sk = reinterpret_cast<uint32_t*>(sv + SL_CH);      // and keys
  uint32_t* lh = sk + SL_CH;                                   // its count, then start, in each group
  uint32_t* gb = lh + NB;                                      // where its share of the group goes
  uint16_t* gm = reinterpret_cast<uint16_t*>(gb + NB);         // group of each bucket
  __shared__ uint32_t tmp32[B / 32 + 1];
  const int t = threadIdx.x;
  const int sh = key_bits - (key_bits < SL_NBL ? key_bits : SL_NBL);
  // (clamped: a key may have changed since its chunk was counted, where rows lie on each other)
  auto group = [&](uint32_t key) -> uint32_t {
    const uint32_t x = key >> sh, g = gm[x < NB ? x : NB - 1];
    return g < NB ? g : NB - 1;
  };
  long long n = *sl.lchunk_n;
  if (n > sl.lchunk_cap) n = sl.lchunk_cap;
  for (long long k = blockIdx.x; k < n; k += gridDim.x) {
    const LongChunk lc = sl.lchunk[k];
    if (lc.huge == SL_NONE) continue;
    const HugeEntry he = sl.huge[lc.huge];
    if (he.bad) continue;
    const long long e0 = (long long)lc.chunk * SL_CH;
    const int len = he.len - e0 < SL_CH ? int(he.len - e0) : SL_CH;
    const VT* vp = out_val + he.off;
    if (!in_place<Gs>::value && he.buf == BUF_SRC) vp = gs.view(gs.srcs()[he.row], he.len).v;
    const uint32_t starts = gstart[(long long)lc.huge * (NB / 32) + (t & 31)], count = __popc(starts),
                   before = warp_incl_sum(count) - count;
    for (int x = t; x < NB; x += B) {
      lh[x] = 0;
      gm[x] = uint16_t(group_of_bucket(starts, before, x >> 5));
    }
    uint32_t key[U], pk[U];  // group << 16 | rank in the group's share of the chunk
    VT val[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = t + u * B;
      key[u] = x < len ? ss_key(ld_stream(out_col + he.off + e0 + x)) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = t + u * B;
      val[u] = x < len ? ld_stream(vp + e0 + x) : VT(0);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      pk[u] = 0xFFFFFFFFu;
      if (t + u * B >= len) continue;
      const uint32_t g = group(key[u]);
      pk[u] = (g << 16) | atomicAdd(&lh[g], 1u);
    }
    __syncthreads();
    uint32_t* const cur = cursor + he.off / SL_GSLOT;
    for (int g = t; g < NB; g += B) gb[g] = lh[g] ? atomicAdd(cur + g, lh[g]) : 0u;
    smem_excl_sum_w<B>(lh, NB, tmp32);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (pk[u] == 0xFFFFFFFFu) continue;
      const uint32_t q = lh[pk[u] >> 16] + (pk[u] & 0xFFFFu);
      sk[q] = key[u];
      sv[q] = val[u];
    }
    __syncthreads();
    for (int i = t; i < len; i += B) {
      const uint32_t kk = sk[i], g = group(kk);
      const uint32_t q = gb[g] + (uint32_t(i) - lh[g]);
      if (q >= uint32_t(he.len)) continue;
      st_stream(tkey + he.off + q, kk);
      st_stream(tval + he.off + q, sv[i]);
    }
    __syncthreads();
  }
}

constexpr size_t split_fine_smem() { return size_t(1 << SF_NBL) * 4 * 3; }
template <class CI, class VT>
__global__ void __launch_bounds__(SF_B, SF_MINB)
    k_split_fine(const HugeEntry* __restrict__ runs, const unsigned* __restrict__ nruns_p, long long runs_cap,
                 unsigned* ticket, const uint32_t* __restrict__ tkey, const VT* __restrict__ tval,
                 CI* __restrict__ out_col, VT* __restrict__ out_val, RunLists rl, DevStatus* st) {
  constexpr int B = SF_B, U = SF_U, NBM = 1 << SF_NBL;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* hist = reinterpret_cast<uint32_t*>(smem);  // bucket sizes, then starts, then cursors
  uint32_t* prv = hist + NBM;
  uint32_t* nxb = prv + NBM;
  __shared__ uint32_t tmp32[B / 32 + 1];
  __shared__ unsigned s_item;
  const int t = threadIdx.x;
  long long count = *nruns_p;
  if (count > runs_cap) count = runs_cap;
  for (;;) {
    if (t == 0) s_item = atomicAdd(ticket, 1u);
    __syncthreads();
    const long long item = s_item;
    if (item >= count) break;
    const long long g0 = runs[item].off, L = runs[item].len;
    const uint32_t* skp = tkey + g0;
    const VT* svp = tval + g0;
    // the bucket's own key range
    uint32_t mn = 0xFFFFFFFFu, mx = 0u;
    for (long long e0 = t; e0 < L; e0 += (long long)B * U) {
      uint32_t k[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (e0 + (long long)u * B < L) k[u] = ld_stream(skp + e0 + (long long)u * B);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (e0 + (long long)u * B < L) {
          mn = k[u] < mn ? k[u] : mn;
          mx = k[u] > mx ? k[u] : mx;
        }
    }
    mn = __reduce_min_sync(0xFFFFFFFFu, mn);
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if ((t & 31) == 0) {
      tmp32[t >> 5] = mn;
      hist[t >> 5] = mx;  // hist is cleared below
    }
    __syncthreads();
    mn = 0xFFFFFFFFu;
    mx = 0u;
    for (int w = 0; w < B / 32; ++w) {
      mn = tmp32[w] < mn ? tmp32[w] : mn;
      mx = hist[w] > mx ? hist[w] : mx;
    }
    __syncthreads();
    const uint32_t lo = mn, span = mx >= mn ? mx - mn : 0u;  // keys in [lo, lo + span]
    const int wb = span ? 32 - __clz(span) : 0;               // 2^wb > span
    const int nbl = wb < SF_NBL ? wb : SF_NBL, nb = 1 << nbl, sh = wb - nbl;
    for (int x = t; x < NBM; x += B) hist[x] = 0;
    __syncthreads();
    // pass 1: bucket sizes
    for (long long e0 = t; e0 < L; e0 += (long long)B * U) {
      uint32_t k[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (e0 + (long long)u * B < L) k[u] = ld_stream(skp + e0 + (long long)u * B);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (e0 + (long long)u * B < L) atomicAdd(&hist[(k[u] - lo) >> sh], 1u);
    }
    __syncthreads();
    smem_excl_sum_w<B>(hist, NBM, tmp32);
    split_groups<B, NBM>(hist, prv, nxb, tmp32, nb, uint32_t(L), [&](int, bool, uint32_t s, uint32_t e) {
      if (e - s <= uint32_t(SS_RUN_MAX)) queue_run(rl, FinalEntry{g0 + s, int(e - s), BUF_OUT, 0}, st, -6);
      else dev_fail(st, SP_ERR_INTERNAL, -7);  // repeated keys (reported where the map was built)
    });
    __syncthreads();
    // pass 2 (hist now serves as the bucket cursors): scatter entry by entry
    for (long long e0 = t; e0 < L; e0 += (long long)B * U) {
      uint32_t k[U];
      VT v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (e0 + (long long)u * B < L) k[u] = ld_stream(skp + e0 + (long long)u * B);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (e0 + (long long)u * B < L) v[u] = ld_stream(svp + e0 + (long long)u * B);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (e0 + (long long)u * B >= L) continue;
        const uint32_t q = atomicAdd(&hist[(k[u] - lo) >> sh], 1u);
        if (q >= uint32_t(L)) continue;
        st_stream(out_col + g0 + q, CI(k[u]));
        st_stream(out_val + g0 + q, v[u]);
      }
    }
    __syncthreads();
  }
}

// ---- the sort of tiles and runs ----------------------------------------------------------

template <class Cfg, class VT>
__host__ __device__ constexpr size_t ss_smem_bytes() {
  // values (sorted), keys (bucket order, then sorted), bucket counters; tiles add the row
  // tables and the row-start bitmap with its word prefix
  return size_t(Cfg::CAP) * (sizeof(VT) + 4 + 4) +
         (Cfg::kTiles ? size_t(Cfg::ROWS) * 32 + size_t(Cfg::WORDS) * 8 : 0);
}

// Resident CTAs per SM: MINB, or as many as their shared memory leaves room for (228 KB per SM,
// 1 KB of it per CTA for the system; the arrays above and the kernel's own).  Tile shape 1 with
// 8-byte values holds 3, not 4.
template <class Cfg, class VT>
constexpr int ss_minb() {
  const size_t per = ss_smem_bytes<Cfg, VT>() + (Cfg::kTiles ? size_t(Cfg::ROWS + 1) * 16 : 0) + 256 + 1024;
  const int fit = int(228 * 1024 / per);
  return fit < Cfg::MINB ? fit : Cfg::MINB;
}

struct SsRow {     // a tile's row (one 16-byte word)
  uint32_t rdel;   // output offset from base - packed start
  uint32_t ps_L;   // packed start | length << 16
  float scale;     // bucket scale
  unsigned mid;    // which relabelling
};

// Exclusive scan of the bucket counters cnt[0, B * ITEMS) in place, thread t owning ITEMS
// consecutive ones; each becomes start | count << 16 (both at most CAP <= 4096).
template <int B, int ITEMS>
__device__ __forceinline__ void ss_scan(uint32_t* cnt, uint32_t* tmp) {
  static_assert(ITEMS % 4 == 0 && B * ITEMS <= 4096, "16-byte words; 16-bit halves");
  constexpr int NW = B / 32, Q = ITEMS / 4;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint4* c4 = reinterpret_cast<uint4*>(cnt) + t * Q;
  uint32_t s = 0;
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    const uint4 v = c4[j];
    s += v.x + v.y + v.z + v.w;
  }
  const uint32_t inc = warp_incl_sum(s);
  if (lane == 31) tmp[w] = inc;
  __syncthreads();
  uint32_t run = inc - s;
#pragma unroll
  for (int k = 0; k < NW - 1; ++k) run += k < w ? tmp[k] : 0u;
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    uint4 v = c4[j];
    uint32_t c;
    c = v.x, v.x = run | (c << 16), run += c;
    c = v.y, v.y = run | (c << 16), run += c;
    c = v.z, v.z = run | (c << 16), run += c;
    c = v.w, v.w = run | (c << 16), run += c;
    c4[j] = v;
  }
  __syncthreads();
}

template <int B, int ITEMS>
__device__ __forceinline__ void ss_clear(uint32_t* cnt) {
  uint4* c4 = reinterpret_cast<uint4*>(cnt) + threadIdx.x * (ITEMS / 4);
#pragma unroll
  for (int j = 0; j < ITEMS / 4; ++j) c4[j] = make_uint4(0, 0, 0, 0);
}

// Rank of `key` among its bucket's keys sk[s, s + c): the first four without a loop (most
// buckets hold one or two keys, and a warp would loop to its largest), the rest in one.
__device__ __forceinline__ uint32_t ss_rank(const uint32_t* sk, uint32_t s, uint32_t c, uint32_t key) {
  const uint32_t* b = sk + s;
  uint32_t p = s;
  if (c > 1u) {
    const uint32_t k0 = b[0], k1 = b[1];
    p += (k0 < key) + (k1 < key);
  }
  if (c > 2u) p += b[2] < key;
  if (c > 3u) {
    p += b[3] < key;
#pragma unroll 1
    for (uint32_t q = 4; q < c; ++q) p += b[q] < key;
  }
  return p;
}

// Work items: tiles [0, ntiles) of the partition, or the runs of one slice of the run
// lists: whole rows at their source, rows in the output arrays, and the split's runs in the
// output or in the temporary arrays.  Every item's entries are loaded before any of them is
// written, so a run is sorted in place.
//
// The bucket sort: an entry's bucket counter (shared memory) returns its arrival number,
// one block scan turns the counters into bucket starts, the entry's key is put at start +
// arrival, and its owner (the thread that loaded it, which keeps key and bucket in
// registers) ranks it among its bucket's keys, one on average.  Keys and
// values then go to their sorted position in shared memory and are written coalesced.
// A bucket of more than `heavy` keys (skewed keys): a tile writes it in bucket order and
// queues it as a run; a run buckets it again over its own key range, in the counters of
// its own positions, for up to SS_LEVELS levels (the last ranks whatever is left).
//
// A position past the item's end carries a padding entry: its bucket is the counter of its
// own position, which no bucket uses, so it passes through the sort in place and every pass
// runs without a bounds check; only loads and stores look at the length.
//
// What bounds it: shared-memory wavefronts and issue slots (profiles of a tile sort: rows of
// 512 entries 80 % of the LSU data pipe, 53 % of issue, 22 % of the DRAM copy rate; 2 M random
// rows of R-MAT scale 25, where the lookups miss L2, 60, 55 and 28 %), and for a matrix whose
// column map exceeds L2 the random lookups.  So the gather is part of the sort (one
// pass over the entries instead of two), an entry stays with its thread from load to
// staging, and buckets hold one key on average.  Uniform rows of 32 over 2^25 columns: 25.8
// -> 16.4 ms per permutation, of which the lookups alone take 12.9 in a plain gather; rows
// of 512 over 2^21 columns: 17.5 -> 11.3 ms; R-MAT scale 25: 21.0 -> 17.6 ms (17.1 with the
// long rows split chunk by chunk and the partition part of the scan).
template <class Cfg, class Gs>
__global__ void __launch_bounds__(Cfg::B, ss_minb<Cfg, typename Gs::VT>())
    k_seg_sort(Gs gs, const long long* __restrict__ vp, long long nnz, const long long* __restrict__ tile_first,
               long long ntiles,
               RunLists rl, int slice, const uint32_t* __restrict__ tkey_g,
               const typename Gs::VT* __restrict__ tval_g, typename Gs::CI* __restrict__ out_col,
               typename Gs::VT* __restrict__ out_val, int key_bits, int heavy, DevStatus* st) {
  using CI = typename Gs::CI;
  using VT = typename Gs::VT;
  constexpr int B = Cfg::B, ITEMS = Cfg::ITEMS, CAP = Cfg::CAP, ROWS = Cfg::ROWS, WORDS = Cfg::WORDS, RPT = Cfg::RPT;
  extern __shared__ __align__(16) unsigned char smem[];
  VT* sval = reinterpret_cast<VT*>(smem);
  uint32_t* skey = reinterpret_cast<uint32_t*>(smem + size_t(CAP) * sizeof(VT));
  uint32_t* cnt = skey + CAP;
  // tiles only (runs allocate none of these)
  SsRow* rows = reinterpret_cast<SsRow*>(cnt + CAP);
  ulonglong2* rptr = reinterpret_cast<ulonglong2*>(rows + ROWS);  // the row's column / value pointers - packed start
  uint32_t* bits = reinterpret_cast<uint32_t*>(rptr + ROWS);      // row starts
  uint32_t* wpre = bits + WORDS;                                  // row starts in earlier words
  __shared__ uint32_t tmp32[B / 32 + 1];
  __shared__ uint32_t s_min[2], s_max[2];
  __shared__ int s_cut, s_cutE;
  // tiles: row pointers vp[r0 .. r1] and source starts of the next tile, copied in while
  // this one is sorted
  __shared__ long long pre_o[Cfg::kTiles ? ROWS + 1 : 1], pre_s[Cfg::kTiles ? ROWS + 1 : 1];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const uint32_t kmax = key_bits >= 32 ? 0xFFFFFFFFu : (1u << key_bits) - 1u;
  const float isr = ss_inv_root(kmax);
  long long nitems, n1 = 0, n2 = 0;
  if constexpr (Cfg::kTiles) {
    nitems = ntiles;
  } else {
    // (an overflow was reported by the producer)
    auto count = [&](int k) -> long long { return rl.n[k] < rl.cap(k) ? rl.n[k] : rl.cap(k); };
    if (slice >= 0) {
      nitems = count(slice);
    } else {
      n1 = count(1);
      n2 = n1 + count(2);
      nitems = n2 + count(3);
    }
  }
  // run i of the slice (slice < 0: of slices 1, 2 and 3 together)
  auto run_at = [&](long long i) -> FinalEntry {
    if (slice >= 0) return rl.slice(slice)[i];
    return i < n1 ? rl.slice(1)[i] : i < n2 ? rl.slice(2)[i - n1] : rl.slice(3)[i - n2];
  };
  if (blockIdx.x >= nitems) return;

  // the next item's descriptor is loaded one item ahead, so its latency hides behind
  // the current item's sort
  long long pf0 = 0;           // tiles: first row
  int pfn = 0;                 // and number of rows
  FinalEntry pfe{0, 0, 0, 0};  // runs
  // tiles: the ranges of this CTA's next 32 tiles, one per lane, and which hold rows (a
  // window inside a longer row is empty; on a power-law matrix half of them are, and one
  // dependent load per empty tile took 1 ms of a scale-25 permutation)
  long long lf0 = 0;
  int ln = 0, lbase = 0;  // (ntiles < 2^31: checked by the launch)
  unsigned lmask = 0;
  // tiles: the next tile's first row and number of rows in (pf0, pfn), or false
  auto next_tile = [&]() -> bool {
    while (lmask == 0) {
      if (lbase >= nitems) return false;
      const int i = lbase + lane * int(gridDim.x);
      ln = 0;
      if (i >= 0 && i < nitems) {
        lf0 = tile_first[i];
        ln = int(tile_first[i + 1] - lf0);
      }
      lmask = __ballot_sync(0xffffffffu, ln > 0);
      lbase = lbase > 0x7fffffff - 32 * int(gridDim.x) ? 0x7fffffff : lbase + 32 * int(gridDim.x);
    }
    const int k = __ffs(lmask) - 1;
    lmask &= lmask - 1;
    pf0 = __shfl_sync(0xffffffffu, lf0, k);
    pfn = __shfl_sync(0xffffffffu, ln, k);
    return true;
  };
  // tiles: start copying the row pointers of the tile in (pf0, pfn)
  auto prefetch_rows = [&](bool any) {
    if (any) {
      const int n = pfn < ROWS ? pfn : ROWS;
      for (int x = t; x <= n; x += B) {
        cp_async8(pre_o + x, vp + pf0 + x);
        if (x < n) cp_async8(pre_s + x, gs.srcs() + pf0 + x);
      }
    }
    cp_async_commit();
  };
  bool more_tiles = false;
  if constexpr (Cfg::kTiles) {
    const bool bad = rl.n[RUNS_BAD] != 0u;  // (read beside the first tiles' ranges)
    lbase = blockIdx.x;
    more_tiles = next_tile();
    if (bad) return;
    prefetch_rows(more_tiles);
  } else {
    pfe = run_at(blockIdx.x);
    if (t < 2) {
      s_min[t] = 0xFFFFFFFFu;
      s_max[t] = 0u;
    }
  }
  int par = 0;
  int ra = 0;  // tiles: the round's first row
  for (long long item = blockIdx.x; Cfg::kTiles ? more_tiles : item < nitems;) {
    const long long nx = item + gridDim.x;
    long long base;
    int E, nrow = 0, rnext = 0;
    uint32_t key[ITEMS], seg[ITEMS];  // seg: bucket | arrival << 16, then start | count << 16
    VT val[ITEMS];
    uint32_t out[Cfg::kTiles ? ITEMS : 1];  // tiles: the position's output offset from base
    // the row of packed entry x of a tile: the row starts at or before x
    auto row_of = [&](int x) -> uint32_t {
      const int w = x >> 5;
      return wpre[w] + __popc(bits[w] & (0xFFFFFFFFu >> (31 - (x & 31)))) - 1u;
    };
    if constexpr (Cfg::kTiles) {
      nrow = pfn;
      if (nrow > ROWS) {  // cannot happen: see RowsPartition
        if (t == 0) dev_fail(st, SP_ERR_INTERNAL, -17);
        nrow = ROWS;
      }
      cp_async_wait_all();  // this tile's row pointers
      __syncthreads();      // and the previous round's last reads of the tables
      ss_clear<B, ITEMS>(cnt);
      for (int w = t; w < WORDS; w += B) bits[w] = 0;
      base = pre_o[0];
      uint32_t L[RPT], off[RPT], mine = 0;
      long long src[RPT];
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        const int r = ra + t * RPT + k;
        L[k] = off[k] = 0;
        if (r < nrow) {
          const long long o0 = pre_o[r], l = pre_o[r + 1] - o0;
          off[k] = uint32_t(o0 - base);  // < WIN
          src[k] = pre_s[r];
          if (l > 0 && l <= Cfg::TMAX && o0 + l <= nnz) L[k] = uint32_t(l);
        }
        mine += L[k] ? ((L[k] << 16) | 1u) : 0u;
      }
      // packed start (high half) and rank among the item's rows (low half)
      const uint32_t inc = warp_incl_sum(mine);
      if (lane == 31) tmp32[wid] = inc;
      __syncthreads();
      uint32_t pre = inc - mine, tot = 0;
#pragma unroll
      for (int k = 0; k < B / 32; ++k) {
        const uint32_t x = tmp32[k];
        pre += k < wid ? x : 0u;
        tot += x;
      }
      E = int(tot >> 16);
      rnext = nrow;
      if (E == 0) {  // only longer (or empty) rows: the next tile
        ra = 0;
        __syncthreads();  // pre_o has been read
        more_tiles = next_tile();
        prefetch_rows(more_tiles);
        continue;
      }
      if (E > CAP) {  // the rows that fit now, the others in another round
        uint32_t q = pre >> 16;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          if (q <= uint32_t(CAP) && q + L[k] > uint32_t(CAP)) {
            s_cut = ra + t * RPT + k;
            s_cutE = int(q);
          }
          q += L[k];
        }
        __syncthreads();
        rnext = s_cut;
        E = s_cutE;
      }
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        const uint32_t ps = pre >> 16, pe = ps + L[k], i = pre & 0xFFFFu;
        if (L[k] == 0 || pe > uint32_t(E)) continue;
        GsView<CI, VT> gv = gs.view(src[k], L[k]);
        if (!gv.c) {
          dev_fail(st, SP_ERR_INTERNAL, -13);
          gv = GsView<CI, VT>{out_col, out_val, 0u};  // readable: at most nnz entries in
        }
        rows[i] = SsRow{off[k] - ps, ps | (L[k] << 16), float(L[k]) * isr, gv.mid};
        rptr[i] = make_ulonglong2((unsigned long long)(gv.c - ps), (unsigned long long)(gv.v - ps));
        atomicOr(&bits[ps >> 5], 1u << (ps & 31));
        // the words whose first entry comes after this row's first: i + 1 starts before them
        for (uint32_t w = (ps >> 5) + 1; (w << 5) <= pe && w < WORDS; ++w) wpre[w] = i + 1;
        if (i == 0) wpre[0] = 0;
        pre += (L[k] << 16) | 1u;
      }
      __syncthreads();
      if (rnext == nrow) {  // the last round: the next tile's row pointers arrive during this sort
        more_tiles = next_tile();
        prefetch_rows(more_tiles);
      }
      // load: key, value and bucket of every entry
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const int x = t + j * B;
        seg[j] = x < E ? row_of(x) : 0u;
        const ulonglong2 rp = rptr[seg[j]];
        key[j] = x < E ? ss_key(ld_stream(reinterpret_cast<const CI*>(rp.x) + x)) : 0u;
        val[j] = x < E ? ld_stream(reinterpret_cast<const VT*>(rp.y) + x) : VT(0);
      }
      if constexpr (!in_place<Gs>::value) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) key[j] = gs.map(rows[seg[j]].mid, key[j]);
      }
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const int x = t + j * B;
        const SsRow r = rows[seg[j]];
        out[j] = r.rdel + x;
        if (key[j] > kmax) {  // a column outside [0, ncols)
          if (x < E) dev_fail(st, SP_ERR_INDEX_RANGE, base + out[j]);
          key[j] = kmax;
        }
        const uint32_t sl =
            x < E ? (r.ps_L & 0xFFFFu) + ss_bucket(key[j], r.scale, (r.ps_L >> 16) - 1u) : uint32_t(x);
        seg[j] = sl | (atomicAdd(&cnt[sl], 1u) << 16);
      }
    } else {
      const FinalEntry fe = pfe;
      if (nx < nitems) pfe = run_at(nx);
      base = fe.off;
      E = fe.len;
      if (fe.len < 0 || fe.len > CAP) {
        if (t == 0) dev_fail(st, SP_ERR_INTERNAL, -18);
        E = 0;
      }
      __syncthreads();  // the previous run's last reads of the staging arrays
      ss_clear<B, ITEMS>(cnt);
      // a single run (a row sorted alone or a key-range group of a long row): its
      // buckets span the run's own key range [min, max], found while loading
      uint32_t mn = 0xFFFFFFFFu, mx = 0u;
      auto load = [&](const auto* cp, const VT* vq) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
          const int x = t + j * B;
          key[j] = x < E ? ss_key(ld_stream(cp + x)) : 0u;
          val[j] = x < E ? ld_stream(vq + x) : VT(0);
        }
      };
      if (!in_place<Gs>::value && fe.buf == BUF_SRC) {
        GsView<CI, VT> gv = gs.view(gs.srcs()[fe.row], E);
        if (!gv.c) {
          if (t == 0) dev_fail(st, SP_ERR_INTERNAL, -13);
          gv = GsView<CI, VT>{out_col + base, out_val + base, 0u};
        }
        load(gv.c, gv.v);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) key[j] = gs.map(gv.mid, key[j]);
      } else if (fe.buf == BUF_TEMP) {
        load(tkey_g + base, tval_g + base);
      } else {
        load(out_col + base, out_val + base);
      }
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const bool ok = t + j * B < E;
        if (key[j] > kmax) {
          if (ok) dev_fail(st, SP_ERR_INDEX_RANGE, base + t + j * B);
          key[j] = kmax;
        }
        mn = ok && key[j] < mn ? key[j] : mn;
        mx = ok && key[j] > mx ? key[j] : mx;
      }
      mn = __reduce_min_sync(0xFFFFFFFFu, mn);
      mx = __reduce_max_sync(0xFFFFFFFFu, mx);
      if (lane == 0) {
        atomicMin(&s_min[par], mn);
        atomicMax(&s_max[par], mx);
      }
      __syncthreads();
      const uint32_t lo = s_min[par], w = s_max[par] > lo ? s_max[par] - lo : 0u;
      if (t == 0) {  // for the next run (its own pair was read a barrier ago)
        s_min[par ^ 1] = 0xFFFFFFFFu;
        s_max[par ^ 1] = 0u;
      }
      par ^= 1;
      const float sc = float(E) * ss_inv_root(w);
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const int x = t + j * B;
        const uint32_t sl = x < E ? ss_bucket(key[j] - lo, sc, uint32_t(E) - 1u) : uint32_t(x);
        seg[j] = sl | (atomicAdd(&cnt[sl], 1u) << 16);
      }
    }
    __syncthreads();
    ss_scan<B, ITEMS>(cnt, tmp32);
    bool hv = false;
    uint32_t open = 0;  // entries in a heavy bucket
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const uint32_t sc = cnt[seg[j] & 0xFFFFu], p = (sc & 0xFFFFu) + (seg[j] >> 16);
      skey[p] = key[j];
      if ((sc >> 16) > uint32_t(heavy)) {
        open |= 1u << j;
        hv = true;
        if constexpr (Cfg::kTiles) {  // left in bucket order, queued as a run
          if ((seg[j] >> 16) == 0u)
            queue_run(rl, FinalEntry{base + out[j] - uint32_t(t + j * B) + p, int(sc >> 16), BUF_OUT, 0}, st, -22);
          seg[j] = p;
          continue;
        }
      }
      seg[j] = sc;
    }
    if constexpr (Cfg::kTiles) {
      __syncthreads();
#pragma unroll
      for (int j = 0; j < ITEMS; ++j)
        if (!((open >> j) & 1u)) seg[j] = ss_rank(skey, seg[j] & 0xFFFFu, seg[j] >> 16, key[j]);
    } else {
      hv = __syncthreads_or(hv);
#pragma unroll
      for (int j = 0; j < ITEMS; ++j)
        if (!((open >> j) & 1u)) seg[j] = ss_rank(skey, seg[j] & 0xFFFFu, seg[j] >> 16, key[j]);
      for (int level = 1; hv; ++level) {
        // skewed keys: the entries of heavy buckets are bucketed again over their bucket's
        // own key range (found at the bucket's first two words); the others keep their
        // place through the scan
        __syncthreads();  // the bucket order has been read
        ss_clear<B, ITEMS>(cnt);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
          if ((open >> j) & 1u) {
            skey[seg[j] & 0xFFFFu] = 0xFFFFFFFFu;
            skey[(seg[j] & 0xFFFFu) + 1] = 0u;
          }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
          if ((open >> j) & 1u) {
            atomicMin(&skey[seg[j] & 0xFFFFu], key[j]);
            atomicMax(&skey[(seg[j] & 0xFFFFu) + 1], key[j]);
          }
        __syncthreads();
        uint32_t arr[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
          uint32_t sl = seg[j] & 0xFFFFu;
          if ((open >> j) & 1u) {
            const uint32_t lo = skey[sl], w = skey[sl + 1] - lo, nb = seg[j] >> 16;
            sl += ss_bucket(key[j] - lo, float(nb) * ss_inv_root(w), nb - 1);
          }
          arr[j] = sl | (atomicAdd(&cnt[sl], 1u) << 16);
        }
        __syncthreads();
        ss_scan<B, ITEMS>(cnt, tmp32);
        bool more = false;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
          if (!((open >> j) & 1u)) continue;
          seg[j] = cnt[arr[j] & 0xFFFFu];
          skey[(seg[j] & 0xFFFFu) + (arr[j] >> 16)] = key[j];
          more |= (seg[j] >> 16) > uint32_t(heavy);
        }
        hv = __syncthreads_or(more) && level < SS_LEVELS;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
          if (!((open >> j) & 1u) || (hv && (seg[j] >> 16) > uint32_t(heavy))) continue;
          seg[j] = ss_rank(skey, seg[j] & 0xFFFFu, seg[j] >> 16, key[j]);
          open &= ~(1u << j);
        }
      }
    }
    __syncthreads();  // the bucket order and the counters have been read
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      skey[seg[j]] = key[j];
      sval[seg[j]] = val[j];
    }
    __syncthreads();
    CI* const oc = out_col + base;
    VT* const ov = out_val + base;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const int x = t + j * B;
      if (x >= E) continue;
      const uint32_t g = Cfg::kTiles ? out[Cfg::kTiles ? j : 0] : uint32_t(x);
      st_stream(oc + g, CI(skey[x]));
      st_stream(ov + g, sval[x]);
    }
    if constexpr (Cfg::kTiles) {
      ra = rnext < nrow ? rnext : 0;
    } else {
      item = nx;
    }
  }
}

// Runs of at most SS_WARP_RUN entries (the first slice of the run lists: rows in the output
// arrays, the split's groups in either buffer), a warp each: every lane keeps four entries
// and counts the run's smaller keys, four at a time from shared memory (broadcast).
constexpr int WR_BLOCK = 256, WR_MINB = 4;
template <class CI, class VT>
__global__ void __launch_bounds__(WR_BLOCK, WR_MINB)
    k_sort_warp_runs(RunLists rl, const uint32_t* __restrict__ tkey, const VT* __restrict__ tval,
                     CI* __restrict__ out_col, VT* __restrict__ out_val, uint32_t kmax, DevStatus* st) {
  constexpr int NW = WR_BLOCK / 32, PER = SS_WARP_RUN / 32;
  __shared__ __align__(16) uint32_t s_key[NW][SS_WARP_RUN];
  const int lane = threadIdx.x & 31;
  uint32_t* wk = s_key[threadIdx.x >> 5];
  long long n = rl.n[0];
  if (n > rl.c0) n = rl.c0;
  const long long nw = (long long)gridDim.x * NW;
  for (long long i = (long long)blockIdx.x * NW + (threadIdx.x >> 5); i < n; i += nw) {
    const FinalEntry fe = rl.list[i];
    const int E = fe.len;
    if (E <= 0 || E > SS_WARP_RUN) {
      if (lane == 0) dev_fail(st, SP_ERR_INTERNAL, -20);
      continue;
    }
    CI* const oc = out_col + fe.off;
    VT* const ov = out_val + fe.off;
    uint32_t key[PER];
    VT val[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int x = lane + 32 * j;
      const bool tmp = fe.buf == BUF_TEMP;
      key[j] = x < E ? (tmp ? ld_stream(tkey + fe.off + x) : ss_key(ld_stream(oc + x))) : 0xFFFFFFFFu;
      val[j] = x < E ? ld_stream(tmp ? tval + fe.off + x : ov + x) : VT(0);
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (lane + 32 * j < E && key[j] > kmax) {
        dev_fail(st, SP_ERR_INDEX_RANGE, fe.off + lane + 32 * j);
        key[j] = kmax;
      }
      wk[lane + 32 * j] = key[j];  // (padding is below no key)
    }
    __syncwarp();
    int rank[PER] = {};
    const uint4* w4 = reinterpret_cast<const uint4*>(wk);
    const int nq = (E + 3) >> 2;
    auto count = [&](auto per) {
      constexpr int P = decltype(per)::value;
      for (int q = 0; q < nq; ++q) {
        const uint4 k = w4[q];
#pragma unroll
        for (int j = 0; j < P; ++j)
          rank[j] += int(k.x < key[j]) + int(k.y < key[j]) + int(k.z < key[j]) + int(k.w < key[j]);
      }
    };
    if (E <= 32) count(std::integral_constant<int, 1>{});
    else if (E <= 64) count(std::integral_constant<int, 2>{});
    else count(std::integral_constant<int, PER>{});
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (lane + 32 * j >= E) continue;
      st_stream(oc + rank[j], CI(key[j]));
      st_stream(ov + rank[j], val[j]);
    }
  }
}

// ---- host side --------------------------------------------------------------------------
struct RowsWs {
  long long ntiles_cap = 0, nchunks = 0, huge_cap = 0, lchunk_cap = 0, cur_cap = 0;
  long long run_cap[4] = {0, 0, 0, 0};
  long long* tile_first = nullptr;
  long long* chunk_first = nullptr;
  unsigned* counters = nullptr;  // [0..3] run list counts [4] fine split ticket [5] fine split list
                                 // [6] long chunks [7] long rows [8] RUNS_BAD
  FinalEntry* fin = nullptr;
  HugeEntry* huge = nullptr;
  HugeEntry* nxt = nullptr;      // oversized buckets (fine split); as many as long rows
  LongChunk* lchunk = nullptr;
  uint32_t* gstart = nullptr;    // long rows: the buckets that start a group, one bit each
  uint32_t* cursor = nullptr;    // long rows: next free place of each group
  uint32_t* tkey = nullptr;
  void* tval = nullptr;
  long long runs_total() const { return run_cap[0] + run_cap[1] + run_cap[2] + run_cap[3]; }
  RunLists runs() const { return RunLists{fin, counters, run_cap[0], run_cap[1], run_cap[2], run_cap[3]}; }
  SortLists lists() const {
    return SortLists{runs(), huge, counters + 7, huge_cap, lchunk, counters + 6, lchunk_cap};
  }
};

constexpr int kRowsSlots = 11;

// Workspace layout of the sort (sort = false: of the gather alone).  extra_runs: runs a
// caller queues itself (beyond the partition's and the split's).
inline RowsWs rows_caps(long long nrows, long long nnz, bool sort, long long extra_runs) {
  RowsWs w;
  w.nchunks = sort ? 0 : (nnz + GC_CH - 1) / GC_CH;
  if (!sort) return w;
  w.ntiles_cap = (nnz + SsTile::W * nrows) / SsTile::WIN + 1;
  // the split's groups (at most 3 L / GROUP_CAP + 1 of a row, and as many of the fine
  // split's buckets), the rows sorted alone, the tiles' heavy buckets (more than SS_HEAVY
  // entries each); the runs lie apart, so a slice for longer ones is bounded by their length
  const long long groups = nnz > SS_RUN_MAX ? 2 * (3 * (nnz / GROUP_CAP) + nnz / SS_RUN_MAX + 16) : 0;
  w.run_cap[0] = extra_runs > 0 ? groups + extra_runs : 0;
  w.run_cap[1] = groups + nnz / SS_HEAVY + 1;
  w.run_cap[2] = nnz / (SS_SMALL_RUN + 1) + 1;
  w.run_cap[3] = nnz / (SS_MID_RUN + 1) + 1;
  if (nnz > SS_RUN_MAX) {
    w.huge_cap = nnz / SS_RUN_MAX + 1;
    w.lchunk_cap = nnz / SL_CH + w.huge_cap;
    w.cur_cap = nnz / SL_GSLOT + 1;
  }
  return w;
}

inline void rows_reserve(Carver& cv, long long nrows, long long nnz, size_t vbytes, size_t* off,
                         bool sort = true, long long extra_runs = 0) {
  const RowsWs w = rows_caps(nrows, nnz, sort, extra_runs);
  const bool need_temp = sort && nnz > SS_RUN_MAX;
  off[0] = cv.reserve(size_t(w.ntiles_cap + 1) * 8);
  off[1] = cv.reserve(size_t(w.nchunks) * 8);
  off[2] = cv.reserve(16 * 4);
  off[3] = cv.reserve(size_t(w.runs_total()) * sizeof(FinalEntry));
  off[4] = cv.reserve(size_t(w.huge_cap) * sizeof(HugeEntry));
  off[5] = cv.reserve(size_t(w.huge_cap) * sizeof(HugeEntry));
  off[6] = cv.reserve(need_temp ? size_t(nnz) * 4 : 0);
  off[7] = cv.reserve(need_temp ? size_t(nnz) * vbytes : 0);
  off[8] = cv.reserve(size_t(w.lchunk_cap) * sizeof(LongChunk));
  off[9] = cv.reserve(size_t(w.huge_cap) * (SL_NB / 8));
  off[10] = cv.reserve(size_t(w.cur_cap) * 4);
}

inline RowsWs rows_bind(const Carver& cv, long long nrows, long long nnz, const size_t* off,
                        bool sort = true, long long extra_runs = 0) {
  RowsWs w = rows_caps(nrows, nnz, sort, extra_runs);
  w.tile_first = cv.at<long long>(off[0]);
  w.chunk_first = cv.at<long long>(off[1]);
  w.counters = cv.at<unsigned>(off[2]);
  w.fin = cv.at<FinalEntry>(off[3]);
  w.huge = cv.at<HugeEntry>(off[4]);
  w.nxt = cv.at<HugeEntry>(off[5]);
  w.tkey = cv.at<uint32_t>(off[6]);
  w.tval = cv.at<void>(off[7]);
  w.lchunk = cv.at<LongChunk>(off[8]);
  w.gstart = cv.at<uint32_t>(off[9]);
  w.cursor = cv.at<uint32_t>(off[10]);
  return w;
}

// Sorts in place the rows a caller queued itself in w.lists() (of nnz entries in all;
// w.counters zeroed before the caller queued them).  Defined and instantiated in rowsort.cu
// for the column and value words of the library, as sort_rows_in_place.
template <class CI, class VT>
sp_status sort_queued(sp_ctx* ctx, cudaStream_t s, const RowsWs& w, long long nnz, int key_bits, CI* out_col, VT* out_val);
// Sorts in place every row of the output arrays (row pointer vp).
template <class CI, class VT>
sp_status sort_rows_in_place(sp_ctx* ctx, cudaStream_t s, const long long* vp, long long nrows, long long nnz,
                             int key_bits, const RowsWs& w, CI* out_col, VT* out_val);

// Cuts the queued long rows (nnz > SS_RUN_MAX) into runs.
template <class Gs>
sp_status split_long(sp_ctx* ctx, cudaStream_t s, const RowsWs& w, int key_bits, const Gs& gs,
                     typename Gs::CI* out_col, typename Gs::VT* out_val) {
  using CI = typename Gs::CI;
  using VT = typename Gs::VT;
  const int nsm = ctx->num_sms;
  VT* tval = static_cast<VT*>(w.tval);
  const SortLists sl = w.lists();
  auto grid = [&](long long minb, long long cap) { return unsigned(cap < minb * nsm ? cap : minb * nsm); };
  {
    ::sp::PhaseScope ph(ctx, s, in_place<Gs>::value ? SP_PHASE_HUGE : SP_PHASE_GATHER);
    k_long_hist<Gs><<<grid(SL_HMINB, w.lchunk_cap), SL_HB, 0, s>>>(gs, sl, w.tkey, out_col, w.gstart, w.cursor, w.nxt,
                                                                  w.counters + 5, w.huge_cap, key_bits, ctx->dstatus);
  }
  SP_CUDA(cudaGetLastError());
  constexpr size_t ssm = long_scatter_smem<VT>();
  SP_CUDA(set_smem(k_long_scatter<Gs>, ssm));
  {
    SP_PHASE(SP_PHASE_HUGE);
    k_long_scatter<Gs><<<grid(sl_sminb<VT>(), w.lchunk_cap), SL_SB, ssm, s>>>(gs, sl, w.tkey, tval, out_col, out_val,
                                                                       w.gstart, w.cursor, key_bits);
  }
  SP_CUDA(cudaGetLastError());
  if (!fine_split_follows(key_bits)) return SP_OK;
  constexpr size_t fsm = split_fine_smem();
  SP_CUDA(set_smem(k_split_fine<CI, VT>, fsm));
  {
    SP_PHASE(SP_PHASE_HUGE);
    k_split_fine<CI, VT><<<grid(SF_MINB, w.huge_cap), SF_B, fsm, s>>>(w.nxt, w.counters + 5, w.huge_cap, w.counters + 4,
                                                                     w.tkey, tval, out_col, out_val, w.runs(),
                                                                     ctx->dstatus);
  }
  SP_CUDA(cudaGetLastError());
  return SP_OK;
}

// Sorts the queued runs; nnz bounds their length.
template <class Gs>
sp_status sort_runs(sp_ctx* ctx, cudaStream_t s, const RowsWs& w, long long nnz, int key_bits, const Gs& gs,
                    typename Gs::CI* out_col, typename Gs::VT* out_val) {
  using VT = typename Gs::VT;
  auto run = [&](auto cfg, int slice) -> sp_status {
    using Cfg = decltype(cfg);
    constexpr size_t sm = ss_smem_bytes<Cfg, VT>();
    SP_CUDA(set_smem(k_seg_sort<Cfg, Gs>, sm));
    SP_PHASE(SP_PHASE_LONG);
    const long long cap = (long long)ss_minb<Cfg, VT>() * ctx->num_sms, n = slice >= 0 ? w.run_cap[slice] : w.runs_total();
    k_seg_sort<Cfg, Gs><<<unsigned(n < cap ? n : cap), Cfg::B, sm, s>>>(gs, nullptr, 0, nullptr, 0, w.runs(), slice, w.tkey,
                                                        static_cast<const VT*>(w.tval), out_col, out_val, key_bits,
                                                        ctx->cur.heavy, ctx->dstatus);
    SP_CUDA(cudaGetLastError());
    return SP_OK;
  };
  // few runs in all: one launch whose CTAs take any of them (an empty launch costs 2 to 3 us;
  // the other two cost more than few small runs gain from small CTAs)
  if (nnz > SS_SMALL_RUN && nnz <= SS_ONE_LAUNCH) return run(SsRun{}, -1);
  SP_TRY(run(SsRunS{}, 1));
  if (nnz > SS_SMALL_RUN) SP_TRY(run(SsRunM{}, 2));
  if (nnz > SS_MID_RUN) SP_TRY(run(SsRun{}, 3));
  return SP_OK;
}

// The partition of a sort's rows (of nnz entries in all) with the kernel shapes of this call
// (context options or the tuning table); buf: where the rows' entries are.  It runs as part
// of the scan that makes the row pointer (StorePartition) or as a pass of its own; w.counters
// are cleared before.
inline RowsPartition sort_partition(sp_ctx* ctx, const RowsWs& w, long long nrows, long long nnz, int buf) {
  const bool large = ctx->cur.tile_shape == 1;
  const int wlog = large ? ceil_log2_u64(SsTileL::WIN) : ceil_log2_u64(SsTile::WIN);
  return RowsPartition{nrows, nnz, ((nnz + SsTile::W * nrows) >> wlog) + 1, w.tile_first, 0, nullptr, w.lists(), buf,
                       wlog, large ? SsTileL::TMAX : SsTile::TMAX, w.counters + RUNS_BAD, ctx->dstatus};
}
inline RowsPartition gather_partition(sp_ctx* ctx, const RowsWs& w, long long nrows, long long nnz) {
  RowsPartition part{};
  part.nrows = nrows;
  part.nnz = nnz;
  part.nchunks = w.nchunks;
  part.chunk_first = w.chunk_first;
  part.st = ctx->dstatus;
  return part;
}
inline sp_status launch_partition(sp_ctx* ctx, cudaStream_t s, const RowsPartition& part, const long long* vp) {
  {
    SP_PHASE(SP_PHASE_PARTITION);
    k_partition<0><<<grid_for(part.nrows, 256, ctx->num_sms * 16), 256, 0, s>>>(part, vp);
  }
  SP_CUDA(cudaGetLastError());
  return SP_OK;
}

// The output rows (row pointer vp, nnz entries, partitioned by sort_partition) from their
// source `gs`, sorted.
template <class Gs>
sp_status sort_rows_from(sp_ctx* ctx, cudaStream_t s, const long long* vp, long long nrows, long long nnz,
                         int key_bits, const RowsWs& w, const Gs& gs, typename Gs::CI* out_col,
                         typename Gs::VT* out_val) {
  using VT = typename Gs::VT;
  if (nrows == 0 || nnz == 0) return SP_OK;
  const int nsm = ctx->num_sms;
  const bool large_tiles = ctx->cur.tile_shape == 1;
  const long long ntiles = sort_partition(ctx, w, nrows, nnz, BUF_SRC).ntiles;
  // The rows longer than SS_RUN_MAX (cut by key range) and the tiles (rows of at most tmax)
  // are disjoint.  With the context's overlap on, the long rows run on the context's side
  // stream, whose higher priority dispatches their CTAs ahead of the tiles', while the
  // tiles run on `s`.  The runs, which the split queues, wait for both.
  const bool any_long = nnz > SS_RUN_MAX, fork = any_long && ctx->overlap && ctx->side;
  sp_status lst = SP_OK;
  if (any_long) {
    cudaStream_t ls = fork ? ctx->side : s;
    if (fork) {
      SP_CUDA(cudaEventRecord(ctx->fork_ev, s));
      SP_CUDA(cudaStreamWaitEvent(ls, ctx->fork_ev, 0));
    }
    lst = split_long(ctx, ls, w, key_bits, gs, out_col, out_val);
    if (fork) SP_CUDA(cudaEventRecord(ctx->join_ev, ls));
  }
  auto tiles = [&](auto cfg) -> sp_status {
    using Cfg = decltype(cfg);
    constexpr size_t sm = ss_smem_bytes<Cfg, VT>();
    SP_CUDA(set_smem(k_seg_sort<Cfg, Gs>, sm));
    SP_PHASE(SP_PHASE_TILE);
    const long long cap = (long long)ss_minb<Cfg, VT>() * nsm, g = ntiles < cap ? ntiles : cap;
    k_seg_sort<Cfg, Gs><<<unsigned(g), Cfg::B, sm, s>>>(gs, vp, nnz, w.tile_first, ntiles, w.runs(), 0, w.tkey,
                                                        static_cast<const VT*>(w.tval), out_col, out_val, key_bits,
                                                        ctx->cur.heavy, ctx->dstatus);
    SP_CUDA(cudaGetLastError());
    return SP_OK;
  };
  sp_status tst = ntiles > 0x7fffffffll ? SP_ERR_OVERFLOW : SP_OK;
  if (lst == SP_OK && tst == SP_OK) tst = large_tiles ? tiles(SsTileL{}) : tiles(SsTile{});
  if (fork) SP_CUDA(cudaStreamWaitEvent(s, ctx->join_ev, 0));
  SP_TRY(lst);
  SP_TRY(tst);
  return sort_runs(ctx, s, w, nnz, key_bits, gs, out_col, out_val);
}

// The output rows (partitioned by gather_partition) gathered from `gs` and relabelled, in
// source order (not if *bad; may be null).
template <class Gs>
sp_status gather_rows(sp_ctx* ctx, cudaStream_t s, const long long* vp, long long nrows, long long nnz,
                      const RowsWs& w, const unsigned* bad, const Gs& gs, typename Gs::CI* out_col,
                      typename Gs::VT* out_val) {
  if (nrows == 0 || nnz == 0) return SP_OK;
  if (w.nchunks > 0x7fffffffll) return SP_ERR_OVERFLOW;
  const int nsm = ctx->num_sms;
  {
    SP_PHASE(SP_PHASE_GATHER);
    const long long g = w.nchunks < (long long)GC_MINB * nsm ? w.nchunks : (long long)GC_MINB * nsm;  // persistent
    k_gather_chunks<Gs><<<unsigned(g), GC_BLOCK, 0, s>>>(gs, vp, nrows, nnz, w.chunk_first, w.nchunks, bad, out_col, out_val,
                                                         ctx->dstatus);
  }
  SP_CUDA(cudaGetLastError());
  return SP_OK;
}

}  // namespace sp
