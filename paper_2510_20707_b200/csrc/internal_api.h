// Entry points the Python binding uses beside the public C ABI (include/mixkv.h): the same calls with a
// status word that the call itself sets to 0 first, so that a binding which hands out a new word per call
// need not enqueue a fill for it.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "mixkv.h"

#ifdef __cplusplus
extern "C" {
#endif

// mixkv_scores (static_scratch == 0) or mixkv_scores_static (workspace ignored).  The word is cleared
// by the first kernel right after its dependency wait; a kernel reports an expired wait two seconds later
// at the earliest.
int mixkv_internal_scores(const void* K, const void* V, const void* Qwin, const int32_t* cu_seqlens_host,
                          int32_t batch, int32_t L, const mixkv_params* p, int static_scratch,
                          void* workspace, size_t workspace_bytes, float* s_comp, float* s_ex_opt,
                          float* s_div_opt, float* rbar_opt, const float* rbar_in_opt, int32_t* status_dev,
                          void* stream);
int mixkv_internal_select(const float* scores, const int32_t* cu_seqlens_host, int32_t batch, int32_t L,
                          const mixkv_params* p, void* workspace, size_t workspace_bytes, int32_t* idx,
                          int32_t* counts, int32_t* idx_offsets, int32_t* status_dev, void* stream);

#ifdef __cplusplus
}
#endif
