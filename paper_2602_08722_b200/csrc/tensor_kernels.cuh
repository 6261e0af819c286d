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
// q_tiles: Q tiles of a CTA; ctas: CTAs of a row block (2: a pair); pack: heads of a Q tile
struct AttnPlan { int split_rb = 0, parts = 1; bool in_cluster = false; int q_tiles = 2, ctas = 1, pack = 1; };
constexpr size_t kMostAttnPartials = (size_t)128 << 20;     // what a grid of a wave or more may take, see attn_plan
// room: the scratch there is; attn_plan_scratch_bytes: what a plan takes, counters and partial results in units of 256 bytes
AttnPlan attn_plan_sparse(const quoka_params* p, int budget_cap, size_t room = SIZE_MAX);
AttnPlan attn_plan_dense(const quoka_params* p, size_t room = SIZE_MAX);
size_t attn_plan_scratch_bytes(const quoka_params* p, const AttnPlan& plan);
size_t attn_split_partial_bytes(const quoka_params* p, const AttnPlan& plan);
size_t attn_split_counter_bytes(const quoka_params* p, const AttnPlan& plan);
bool attn_tc_supported(const quoka_params* p);
// Whether the attention grid (256 query rows per CTA) has fewer CTAs than the GPU has SMs.
bool attn_below_a_wave(const quoka_params* p);
// Whether it is small enough for a plan with parts
bool attn_may_have_parts(const quoka_params* p);
// The longest chunk that has the same plan as one of `chunk` positions
int attn_same_plan_up_to(const quoka_params* p, int chunk);
quoka_status launch_attn_tc(const quoka_params* p, const DevParams& P, const void* q, const void* k, const void* v,
                            const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st,
                            bool after_selection, const AttnPlan& plan);
// plan.ctas = 2: two CTAs with neighbouring positions of a KV group work as a pair (cta_group::2, head_dim 128)
quoka_status launch_attn_tc_pair(const quoka_params* p, const DevParams& P, const void* q, const void* k, const void* v,
                                 const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st,
                                 bool after_selection, const AttnPlan& plan);

}  // namespace quoka
