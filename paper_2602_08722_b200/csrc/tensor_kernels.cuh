// Host-side entry points of the tcgen05 (5th-generation tensor core) kernels.
#pragma once

#include "common.cuh"

namespace quoka {

// Whether the tensor-core kernel covers this configuration (bf16, supported N / head_dim / layout).
bool score_keys_tc_supported(const quoka_params* p);
quoka_status launch_score_keys_tc(const quoka_params* p, const DevParams& P, const void* qbar, const void* k,
                                  float* scores, cudaStream_t st, bool chained);

// Grids that leave SMs idle, all the time or in their last wave: the key tiles of the lightest `split_rb` row blocks of
// every head are cut into `parts` parts, one CTA each (split_rb = 0: none).
// in_cluster: the parts of a row block are one cluster (and need no scratch)
// q_tiles: Q tiles of a CTA
struct AttnPlan { int split_rb = 0, parts = 1; bool in_cluster = false; int q_tiles = 2; };
constexpr size_t kMostAttnPartials = (size_t)128 << 20;     // what a grid of a wave or more may take, see attn_plan
AttnPlan attn_plan_sparse(const quoka_params* p, int budget_cap);
AttnPlan attn_plan_dense(const quoka_params* p);
// Scratch for the partial results
size_t attn_split_partial_bytes(const quoka_params* p, const AttnPlan& plan);
size_t attn_split_counter_bytes(const quoka_params* p, const AttnPlan& plan);
bool attn_tc_supported(const quoka_params* p);
// Whether the attention grid (256 query rows per CTA) has fewer CTAs than the GPU has SMs.
bool attn_below_a_wave(const quoka_params* p);
// Whether it is small enough for a plan with parts; chunk positions of the smallest row block that a plan may use
bool attn_may_have_parts(const quoka_params* p);
int attn_least_block(const quoka_params* p);
quoka_status launch_attn_tc(const quoka_params* p, const DevParams& P, const void* q, const void* k, const void* v,
                            const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st,
                            bool after_selection, const AttnPlan& plan);
// head_dim 128: two CTAs with neighbouring positions of a KV group work as a pair (cta_group::2)
quoka_status launch_attn_tc_pair(const quoka_params* p, const DevParams& P, const void* q, const void* k, const void* v,
                                 const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st,
                                 bool after_selection, const AttnPlan& plan);

}  // namespace quoka
