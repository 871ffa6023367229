// Segment copy: an output assembled from contiguous pieces of one or two source arrays
// (the unchanged-row runs of an assignment, Sec. 2.3 / Algorithm 4's Add step, where rows
// outside I are A's rows verbatim).  Each segment j covers output positions
// [segs[j].dst, segs[j+1].dst) and reads consecutive positions from segs[j].src on (bit 62
// of src selects the second array).  A segment whose src is kSegSkip is left alone: its
// positions are written by another kernel, which may run at the same time.
//
// A warp takes SC_CH output positions at a time; its lanes hold the next 32 segments.  Inside
// a segment it moves sc_u() x 32 entries per step, all loads before any store: source and
// destination differ in alignment by an arbitrary number of entries, so words of one entry
// with sc_u() of each array in flight per lane keep more bytes on the way than 16-byte words
// realigned in registers, one group per thread behind a search for its segment.
//
// Where the held segments are short (less than 16 sc_u() entries each: rows of I side by side),
// one at a time would leave the warp waiting for a load per segment.  Then every lane takes
// positions of the whole window and finds each one's segment among the held ones with five
// shuffles.  An assignment (select-second) of 8371 consecutive rows of 4 entries, fp64, 1 M
// rows: 0.386 ms one at a time, 0.228 with this (16-byte words and a search each: 0.339); of
// 1 M random rows of 4 M, replaced: 0.817 -> 0.762.  Limits of 32 sc_u() entries, and 6 or 5
// CTAs per SM with four positions per lane, were within 3 % of it there and up to 4 %
// slower on 789 M entries in long segments.
#pragma once

#include "common.cuh"

namespace sp {

struct CopySeg {
  long long dst;  // first output position
  long long src;  // first source position; bit 62: the second array
};
constexpr long long kSegB = 1ll << 62;
constexpr long long kSegSkip = 1ll << 61;  // src of a segment another kernel writes: not copied
constexpr int SC_CHLOG = 11, SC_CH = 1 << SC_CHLOG;  // output positions per chunk
constexpr int SC_BLOCK = 256;
template <class CI, class VT>
constexpr int sc_u() { return sizeof(CI) + sizeof(VT) == 8 ? 4 : 2; }  // entries of each array in flight per lane
// Persistent grid, CTAs per SM: alone, and while the merge shares the SMs.  R-MAT scale 25,
// 789 M entries, whole assignment: 4 entries at 8 / 3 CTAs 4.62 ms, 8 at 5 / 3 4.69, 8 at 5 / 2
// 4.84, 6 at 6 / 2 5.12 (16-byte words realigned in registers: 5.28).
constexpr int SC_MINB = 8, SC_MINB_OVERLAP = 3;

// Which segment holds the first position of every chunk: the chunk's row (recorded by the
// scan that makes the row pointer) and the segment starts at or before that row, from the
// bitmap of I's rows and the number of starts before each of its words.
struct SegFinder {
  const long long* chunk_row;
  const long long* wseg;   // segments that start before word w's rows
  const uint32_t* ibits;
  long long m;
  bool each;               // every row of I is a segment of its own
  __device__ long long operator()(long long k) const;
};

// The segments are numbered by a scan; one that gave up waiting (SP_ERR_TIMEOUT) leaves a list
// whose starts do not ascend and whose closing entry another segment may have taken.  Every step
// below moves on in the chunk or in the list, or gives the chunk up, so the copy ends and stays in
// its chunk whatever the list holds.
//
// CI / VT: column / value words (uint32 or unsigned long long views of the arrays).
template <class CI, class VT>
__global__ void __launch_bounds__(SC_BLOCK, SC_MINB)
    k_seg_copy(const CopySeg* __restrict__ segs, const long long* __restrict__ nseg_p, long long total, SegFinder find,
               long long nchunks, const CI* __restrict__ ca, const VT* __restrict__ va, long long na,
               const CI* __restrict__ cb, const VT* __restrict__ vb, long long nb, CI* __restrict__ out_col,
               VT* __restrict__ out_val, DevStatus* st) {
  constexpr int SC_U = sc_u<CI, VT>();
  constexpr int SC_US = 2;  // positions in flight per lane among short segments (32 registers)
  const int lane = threadIdx.x & 31;
  const long long nseg = *nseg_p;
  const long long w0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long k = w0; k < nchunks; k += nw) {
    long long pos = k << SC_CHLOG;
    const long long c1 = pos + SC_CH < total ? pos + SC_CH : total;
    long long j0 = find(k);
    if (j0 < 0 || j0 >= nseg) {  // cannot happen for a consistent segment list
      if (lane == 0) dev_fail(st, SP_ERR_INTERNAL, -34);
      continue;
    }
    while (pos < c1) {
      if (j0 >= nseg) {  // cannot happen for a consistent segment list
        if (lane == 0) dev_fail(st, SP_ERR_INTERNAL, -35);
        break;
      }
      // segments j0 + lane (the list is closed by the total at nseg)
      const long long j = j0 + lane;
      const long long dst = segs[j < nseg ? j : nseg].dst, src = j < nseg ? segs[j].src : kSegSkip;
      const long long last = __shfl_sync(0xffffffffu, dst, 31), wend = last < c1 ? last : c1;
      const int below = __popc(__ballot_sync(0xffffffffu, dst <= pos));
      const int held = __popc(__ballot_sync(0xffffffffu, dst < wend)) - below + 1;  // that reach into [pos, wend)
      if (below > 0 && held > 2 && wend - pos < held * (16ll * SC_U)) {
        // start and source of each held segment, from pos on
        const long long d = dst - pos, w = wend - pos;
        const int rd = d <= 0 ? 0 : d < w ? int(d) : SC_CH;
        const long long so = src == kSegSkip || d >= 0 ? src : src - d;
        for (int x0 = 0; x0 < int(w); x0 += 32 * SC_US) {
          CI c[SC_US];
          VT v[SC_US];
          bool ok[SC_US];
#pragma unroll
          for (int u = 0; u < SC_US; ++u) {
            const int x = x0 + 32 * u + lane;
            int cur = 0;  // the last held segment that starts at or before x
#pragma unroll
            for (int step = 16; step; step >>= 1) {
              const int r = __shfl_sync(0xffffffffu, rd, cur + step);
              if (r <= x) cur += step;
            }
            const int first = __shfl_sync(0xffffffffu, rd, cur);
            const long long sc = __shfl_sync(0xffffffffu, so, cur), from = (sc & ~kSegB) + (x - first);
            const bool second = (sc & kSegB) != 0;
            ok[u] = x < int(w) && sc != kSegSkip;
            if (ok[u] && (from < 0 || from >= (second ? nb : na))) {
              dev_fail(st, SP_ERR_INTERNAL, -32);
              ok[u] = false;
            }
            c[u] = ok[u] ? __ldcs((second ? cb : ca) + from) : CI(0);
            v[u] = ok[u] ? __ldcs((second ? vb : va) + from) : VT(0);
          }
#pragma unroll
          for (int u = 0; u < SC_US; ++u) {
            const long long x = pos + x0 + 32 * u + lane;
            if (ok[u]) {
              __stcs(out_col + x, c[u]);
              __stcs(out_val + x, v[u]);
            }
          }
        }
        pos = wend;
        j0 += 31;
        continue;
      }
      for (;;) {
        // the last held segment that starts at or before pos; its end is the next one's start
        const int cur = __popc(__ballot_sync(0xffffffffu, dst <= pos)) - 1;
        if (cur < 0 || cur >= 31) {  // past the held ones (cur < 0 cannot happen)
          if (cur < 0) {
            if (lane == 0) dev_fail(st, SP_ERR_INTERNAL, -31);
            pos = c1;
          }
          j0 += 31;
          break;
        }
        const long long d0 = __shfl_sync(0xffffffffu, dst, cur), d1 = __shfl_sync(0xffffffffu, dst, cur + 1);
        const long long s = __shfl_sync(0xffffffffu, src, cur);
        const long long end = d1 < c1 ? d1 : c1;
        if (d0 > pos || end <= pos) {  // cannot happen for a consistent segment list
          if (lane == 0) dev_fail(st, SP_ERR_INTERNAL, -31);
          pos = c1;
          break;
        }
        if (s != kSegSkip) {
          const long long from = (s & ~kSegB) + (pos - d0);
          const bool second = (s & kSegB) != 0;
          int n = int(end - pos);
          if (from < 0 || from + n > (second ? nb : na)) {
            if (lane == 0) dev_fail(st, SP_ERR_INTERNAL, -32);
          } else {
            const CI* cs = (second ? cb : ca) + from + lane;
            const VT* vs = (second ? vb : va) + from + lane;
            CI* cd = out_col + pos + lane;
            VT* vd = out_val + pos + lane;
            n -= lane;  // entries from this lane's first on
            for (; __any_sync(0xffffffffu, n > 0); n -= 32 * SC_U, cs += 32 * SC_U, vs += 32 * SC_U, cd += 32 * SC_U,
                                                    vd += 32 * SC_U) {
              CI c[SC_U];
              VT v[SC_U];
#pragma unroll
              for (int u = 0; u < SC_U; ++u) c[u] = 32 * u < n ? __ldcs(cs + 32 * u) : CI(0);
#pragma unroll
              for (int u = 0; u < SC_U; ++u) v[u] = 32 * u < n ? __ldcs(vs + 32 * u) : VT(0);
#pragma unroll
              for (int u = 0; u < SC_U; ++u)
                if (32 * u < n) __stcs(cd + 32 * u, c[u]);
#pragma unroll
              for (int u = 0; u < SC_U; ++u)
                if (32 * u < n) __stcs(vd + 32 * u, v[u]);
            }
          }
        }
        pos = end;
        if (pos >= c1) break;
      }
    }
  }
}

}  // namespace sp
