// Entry points beside the public C ABI (include/mixkv.h): two the Python binding uses, and the launch rules for tests.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "mixkv.h"

#ifdef __cplusplus
extern "C" {
#endif

// The same calls as the public ones with a status word that the call itself sets to 0 first, so that a binding which
// hands out a new word per call need not enqueue a fill for it.
//
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

// The rules that split the work of a call over clusters, as functions of the sizes and of how many clusters of n CTAs a
// device holds at once (alone[n] with one CTA per SM, paired[n] with two, shared[n] with three, n = 1 .. 8).  No device is
// needed.  decode: CTAs per unit and the depth of their rings; tail, budget: CTAs per unit, per (sequence, layer) pair;
// adapt: threads of a CTA when the tail shares adaptive budgets out, 0: when it does not; gram: tiles of a map of `cells`
// cells a side (parts 2: of single rows, 3: of sums) that a CTA takes in a run, 0: one contiguous share.
void mixkv_internal_decode_shape(int64_t units, int32_t max_rows, int32_t even, int32_t sms, const int32_t* shared,
                                 const int32_t* alone, int32_t* ctas, int32_t* depth);
int mixkv_internal_tail_clusters(int64_t units, int32_t candidates, int32_t sms, const int32_t* alone);
int mixkv_internal_adapt_threads(int64_t sequences, int32_t heads, int32_t candidates, const int32_t* alone,
                                 const int32_t* paired);
int mixkv_internal_gram_run(int32_t heads, int32_t cells, int32_t parts, int32_t whole_sectors, int64_t l2_bytes);
int mixkv_internal_budget_clusters(int32_t pairs, int64_t keys_per_pair, const int32_t* alone);

// Rounds of a threshold search among keys lo .. hi that ends at `key` without listing any: keys [base, base + span] counted
// in bins of 2^shift.  Returns their number (three at most).
int mixkv_internal_search_rounds(uint32_t lo, uint32_t hi, uint32_t key, uint32_t* base, uint32_t* span, int32_t* shift);

// How `tiles` are split over at most `sms` CTAs (per_head: the tiles of every head, 0: heads differ): the number of CTAs;
// first[0 .. CTAs] their first tiles, owner[tiles] the CTA that pass 2 and the tail look for a tile's statistics at.
int mixkv_internal_split_tiles(int32_t tiles, int32_t per_head, int32_t sms, int32_t* first, int32_t* owner);

// Whether the spare warp of pass 2 folds normalisers: tiles of either pass (per_head as above), heads of the call, pass-1 tiles
// of its longest.
int mixkv_internal_pass2_spare(int32_t tiles1, int32_t per_head1, int32_t tiles2, int32_t per_head2, int32_t heads,
                               int32_t longest, int32_t sms);

// Table of 16 words that the warps of a pair of pass 2's epilogue hand their statistics of a CTA's segment over in.
int mixkv_internal_stats_table(int32_t segment, int32_t pair);

#ifdef __cplusplus
}
#endif
