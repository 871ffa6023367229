// The row sort's launches (rowsort.cuh) that need no source, instantiated once for every
// column and value word of the library.
#include "rowsort.cuh"

namespace sp {

template <class CI, class VT>
sp_status sort_queued(sp_ctx* ctx, cudaStream_t s, const RowsWs& w, long long nnz, int key_bits, CI* out_col,
                      VT* out_val) {
  const RowsInPlace<CI, VT> gs{nullptr, out_col, out_val};
  if (nnz > SS_RUN_MAX) SP_TRY(split_long(ctx, s, w, key_bits, gs, out_col, out_val));
  if (w.run_cap[0] > 0) {
    SP_PHASE(SP_PHASE_LONG);
    const long long need = (w.run_cap[0] + 7) / 8, cap = (long long)WR_MINB * ctx->num_sms;
    k_sort_warp_runs<CI, VT><<<unsigned(need < cap ? need : cap), WR_BLOCK, 0, s>>>(
        w.runs(), w.tkey, static_cast<const VT*>(w.tval), out_col, out_val, key_bits >= 32 ? 0xFFFFFFFFu : (1u << key_bits) - 1u, ctx->dstatus);
    SP_CUDA(cudaGetLastError());
  }
  return sort_runs(ctx, s, w, nnz, key_bits, gs, out_col, out_val);
}

template <class CI, class VT>
sp_status sort_rows_in_place(sp_ctx* ctx, cudaStream_t s, const long long* vp, long long nrows, long long nnz,
                             int key_bits, const RowsWs& w, CI* out_col, VT* out_val) {
  if (nrows == 0 || nnz == 0) return SP_OK;
  SP_CUDA(cudaMemsetAsync(w.counters, 0, 16 * 4, s));
  SP_TRY(launch_partition(ctx, s, sort_partition(ctx, w, nrows, nnz, BUF_OUT), vp));
  return sort_rows_from(ctx, s, vp, nrows, nnz, key_bits, w, RowsInPlace<CI, VT>{vp, out_col, out_val}, out_col,
                        out_val);
}

#define SP_ROWSORT(CI, VT)                                                                                            \
  template sp_status sort_queued<CI, VT>(sp_ctx*, cudaStream_t, const RowsWs&, long long, int, CI*, VT*);             \
  template sp_status sort_rows_in_place<CI, VT>(sp_ctx*, cudaStream_t, const long long*, long long, long long, int,   \
                                                const RowsWs&, CI*, VT*);
SP_ROWSORT(int32_t, uint32_t)
SP_ROWSORT(int32_t, unsigned long long)
SP_ROWSORT(int64_t, uint32_t)
SP_ROWSORT(int64_t, unsigned long long)
SP_ROWSORT(uint32_t, uint32_t)

}  // namespace sp
