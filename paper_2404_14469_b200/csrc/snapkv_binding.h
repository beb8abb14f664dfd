/*
 * Entry points for the Python binding and the tests; not part of the interface in snapkv.h.  The ragged
 * calls with one argument more: with `fill`, rows behind a sequence's end are zeroed and positions set to -1,
 * so that the binding need not clear whole outputs first (two passes over them).
 */
#ifndef SNAPKV_BINDING_H_
#define SNAPKV_BINDING_H_

#include "../../include/snapkv.h"

#ifdef __cplusplus
extern "C" {
#endif

/* snapkv_schedule_items for a ragged batch (at most 32 lengths above W that share a launch): records
 * of eight int32, {unit, t0, t1, vote, slot, nseg, sequence, wave of the launch}. */
int snapkv_binding_ragged_items(const int32_t* seq_lens, int B, int Hq, int Hkv, int d, int W, int votes_only,
                                int grid, int cta, int32_t* out_items, int max_items);
/* Whether the scoring kernel of such a call (host_part: of a part of a call on host buffers) folds the
 * partial statistics with both of its book-keeping warps; -1: arguments not acceptable. */
int snapkv_binding_shared_fold(int B, int Hq, int Hkv, int L, int d, int W, int host_part);
snapkv_status_t snapkv_binding_varlen(const void* q_obs, const void* k, const void* v, const int64_t* k_strides,
                                      const int64_t* v_strides, const int64_t* k_seq_offsets,
                                      const int64_t* v_seq_offsets, const int32_t* seq_lens, const float* lse_obs,
                                      int B, int Hq, int Hkv, int Lmax, int d, int W, int pool_kernel, int pool_type,
                                      int budget, void* out_k, void* out_v, int32_t* out_idx, void* workspace,
                                      size_t workspace_bytes, void* stream, int fill);
snapkv_status_t snapkv_binding_paged(const void* q_obs, const void* k_pool, const void* v_pool,
                                     const int64_t* k_strides, const int64_t* v_strides, const int32_t* page_table,
                                     int pages_per_seq, int page_size, int num_pages, const int32_t* seq_lens,
                                     const float* lse_obs, int B, int Hq, int Hkv, int L, int d, int W,
                                     int pool_kernel, int pool_type, int budget, void* out_k, void* out_v,
                                     int32_t* out_idx, void* workspace, size_t workspace_bytes, void* stream,
                                     int fill);

#ifdef __cplusplus
}
#endif
#endif /* SNAPKV_BINDING_H_ */
