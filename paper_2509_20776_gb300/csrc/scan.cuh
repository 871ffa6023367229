// The single-pass exclusive scan that turns per-row counts into row pointers (the
// proc_pointer of Algorithm 2), shared by every operation and exposed on its own.
#pragma once

#include "internal.h"

namespace sp {

// ------------------------------------------------------------------------------
// Decoupled look-back exclusive scan (Merrill & Garland, 2016).
// Each CTA takes a tile id from an atomic ticket, so a tile only ever waits for tiles
// that already started; every wait is bounded by ScanCtl::spin_limit polls and gives
// up with SP_ERR_TIMEOUT instead of hanging.  Status words pack a 2-bit flag with a
// 62-bit value so one relaxed 64-bit store publishes both.
// ------------------------------------------------------------------------------
constexpr unsigned long long kFlagAgg = 1ull << 62, kFlagInc = 2ull << 62,
                             kValMask = (1ull << 62) - 1;
constexpr int SCAN_BLOCK = 256, SCAN_ITEMS = 16, SCAN_TILE = SCAN_BLOCK * SCAN_ITEMS;
// Scans of at most SCAN_SMALL values take tiles of 4 values per thread: more CTAs, and a
// short chain of loads and stores per thread (a permutation's scan also partitions its rows,
// so each value's store is a chain of its own).
constexpr int SCAN_ITEMS_S = 4;
constexpr long long SCAN_SMALL = 1 << 17;

struct ScanCtl {
  unsigned long long* status;  // one word per tile, zeroed before the launch
  unsigned* ticket;            // zeroed before the launch
  unsigned* bad = nullptr;     // set where a wait gave up (may be null): the output does not ascend
  DevStatus* st;
  long long spin_limit;
  long long hold_tile;  // test hook: this tile never publishes (-1: off)
  long long n;
};

template <class Load, class Store, int IT = SCAN_ITEMS>
__global__ void __launch_bounds__(SCAN_BLOCK, 5) k_scan(Load load, Store store, ScanCtl c) {
  constexpr int B = SCAN_BLOCK, TILE = SCAN_BLOCK * IT;
  __shared__ long long buf[TILE + TILE / 16];
  __shared__ long long tmp[B / 32 + 1];
  __shared__ unsigned s_tile;
  __shared__ long long s_excl;
  const int t = threadIdx.x;
  if (t == 0) s_tile = atomicAdd(c.ticket, 1u);
  __syncthreads();
  const long long tile = s_tile;
  const long long base = tile * TILE;
#pragma unroll
  for (int j = 0; j < IT; ++j) {
    const int x = j * B + t;
    const long long i = base + x;
    buf[x + (x >> 4)] = i < c.n ? (long long)load(i) : 0;
  }
  __syncthreads();
  long long v[IT];
  long long sum = 0;
#pragma unroll
  for (int j = 0; j < IT; ++j) {
    const int x = t * IT + j;
    v[j] = buf[x + (x >> 4)];
    sum += v[j];
  }
  long long agg;
  const long long pre = block_excl_sum<B>(sum, tmp, &agg);
  if (tile == 0) {
    if (t == 0) {
      if (c.hold_tile != 0) st_relaxed_u64(&c.status[0], kFlagInc | (unsigned long long)agg);
      s_excl = 0;
    }
  } else {
    if (t == 0 && tile != c.hold_tile) st_relaxed_u64(&c.status[tile], kFlagAgg | (unsigned long long)agg);
    if (t < 32) {
      long long run = 0, pred = tile - 1;
      bool timeout = false;
      for (;;) {
        const long long idx = pred - t;
        unsigned long long w = kFlagInc;
        if (idx >= 0) {
          w = ld_relaxed_u64(&c.status[idx]);
          long long it = 0;
          while ((w >> 62) == 0) {
            if (++it > c.spin_limit) {
              timeout = true;
              w = kFlagInc;
              break;
            }
            __nanosleep(100);
            w = ld_relaxed_u64(&c.status[idx]);
          }
        }
        const unsigned incm = __ballot_sync(0xffffffffu, (w >> 62) == 2);
        const long long val = (long long)(w & kValMask);
        if (incm) {
          const int f = __ffs(incm) - 1;
          run += warp_sum(t <= f ? val : 0ll);
          break;
        }
        run += warp_sum(val);
        pred -= 32;
      }
      if (__any_sync(0xffffffffu, timeout) && t == 0) {
        dev_fail(c.st, SP_ERR_TIMEOUT, tile);
        if (c.bad) *c.bad = 1u;
      }
      if (t == 0) {
        s_excl = run;
        if (tile != c.hold_tile) st_relaxed_u64(&c.status[tile], kFlagInc | (unsigned long long)(run + agg));
      }
    }
  }
  __syncthreads();
  long long run = s_excl + pre;
#pragma unroll
  for (int j = 0; j < IT; ++j) {
    const int x = t * IT + j;
    buf[x + (x >> 4)] = run;
    run += v[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < IT; ++j) {
    const int x = j * B + t;
    const long long i = base + x;
    const int y = x + 1;
    if (i < c.n) store(i, buf[x + (x >> 4)], y < TILE ? buf[y + (y >> 4)] : s_excl + agg);
  }
  if (base + TILE >= c.n && t == 0) store(c.n, s_excl + agg, s_excl + agg);
}

// load functors
template <class T>
struct LoadArray {
  const T* a;
  __device__ long long operator()(long long i) const { return (long long)a[i]; }
};
// stores: (i, v, vn) with v the exclusive prefix of element i and vn that of i + 1 (i = n:
// the total, twice).  The int64 row pointer, optionally mirrored into a typed output array
template <class T>
struct StoreTyped {
  T* out;
  DevStatus* st;
  __device__ void operator()(long long i, long long v, long long) const {
    if (sizeof(T) == 4 && v > 0x7fffffffll) dev_fail(st, SP_ERR_OVERFLOW, i);
    out[i] = T(v);
  }
};
template <class T>
struct StoreDual {
  long long* vp;
  T* out;  // may be null
  DevStatus* st;
  __device__ void operator()(long long i, long long v, long long) const {
    vp[i] = v;
    if (out) {
      if (sizeof(T) == 4 && v > 0x7fffffffll) dev_fail(st, SP_ERR_OVERFLOW, i);
      out[i] = T(v);
    }
  }
};

inline long long scan_tiles(long long n) {
  const long long tile = n <= SCAN_SMALL ? SCAN_BLOCK * SCAN_ITEMS_S : SCAN_TILE;
  return n > 0 ? (n + tile - 1) / tile : 1;
}
// workspace of a scan of at most n values
inline size_t scan_ws_bytes(long long n) {
  const long long s = scan_tiles(n < SCAN_SMALL ? n : SCAN_SMALL), l = scan_tiles(n), tiles = s > l ? s : l;
  return align_up(size_t(tiles + 1) * 8) + kAlign;
}

// Exclusive scan of n values into n+1 outputs; `ws` must hold scan_ws_bytes(n) (`zeroed`: it
// is cleared already; `bad`: see ScanCtl).
template <class Load, class Store>
sp_status launch_scan(sp_ctx* ctx, cudaStream_t s, Load load, Store store, long long n, char* ws,
                      int phase = SP_PHASE_SCAN, bool zeroed = false, unsigned* bad = nullptr) {
  const long long tiles = scan_tiles(n);
  ScanCtl c;
  c.status = reinterpret_cast<unsigned long long*>(ws);
  c.ticket = reinterpret_cast<unsigned*>(ws + align_up(size_t(tiles + 1) * 8));
  c.bad = bad;
  c.st = ctx->dstatus;
  c.spin_limit = ctx->spin_limit;
  c.hold_tile = ctx->hold_tile;
  c.n = n;
  if (!zeroed) SP_CUDA(cudaMemsetAsync(ws, 0, scan_ws_bytes(n), s));
  if (tiles > 0x7fffffffll) return SP_ERR_OVERFLOW;
  {
    SP_PHASE(phase);
    if (n <= SCAN_SMALL) k_scan<Load, Store, SCAN_ITEMS_S><<<unsigned(tiles), SCAN_BLOCK, 0, s>>>(load, store, c);
    else k_scan<Load, Store><<<unsigned(tiles), SCAN_BLOCK, 0, s>>>(load, store, c);
  }
  SP_CUDA(cudaGetLastError());
  return SP_OK;
}

template <class K>
inline cudaError_t set_smem(K kernel, size_t bytes) {
  // set before every launch that needs it: a flag kept in an inline template is shared by
  // every translation unit of the library, but each one launches its own copy of a kernel.
  // Up to 40 KB beside the kernel's static arrays need no attribute.
  if (bytes <= 40 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
}

}  // namespace sp
