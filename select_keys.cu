// Top-B key selection (Algorithm 1: I = topk(S^, B_SA)).
//
// Scores are compared by order-preserving uint32 codes where it matters (the threshold and its ties).  The output pass walks
// the rows in position order and computes each selected row's slot with warp ballots and prefix sums, so the list comes out
// ascending and rows that tie at the threshold are taken lowest position first.
//
// select_keys_reg_kernel (the default): one CTA of 512 threads per (sequence, KV head), or a cluster
// of 2/4/8 CTAs, holds the whole row of scores IN REGISTERS (as bins, up to 64 per thread: the scores are
// read from memory once, coalesced); see select_row.cuh.
// select_keys_kernel (one CTA per head, a radix select: scores re-read from L2 every pass, 8-bit digits of the codes, most
// significant first) serves rows too long for that.
#include "select_row.cuh"

namespace quoka {

constexpr int kSelThreads = 1024;

__global__ void __launch_bounds__(kSelThreads) select_keys_kernel(DevParams P, const float* __restrict__ scores,
                                                                   int32_t* __restrict__ k_idx,
                                                                   int32_t* __restrict__ k_cnt) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_need;
  __shared__ uint32_t warp_tot[32];
  __shared__ uint32_t warp_off[33];

  grid_launch_dependents();     // the attention kernel may start now: it waits for this grid itself before it reads the list
  grid_dependency_wait();       // the scores come from the kernel before
  const int s = blockIdx.x / P.n_kv, kv = blockIdx.x % P.n_kv;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int T = __ldg(P.ctx_len + s);
  const int B = key_budget(T, P.kv_budget, P.budget_frac);
  const float* row = scores + ((int64_t)s * P.n_kv + kv) * P.max_ctx;
  int32_t* out = k_idx + ((int64_t)s * P.n_kv + kv) * P.budget_cap;
  if (kv == 0 && tid == 0) k_cnt[s] = B;
  for (int i = B + tid; i < P.budget_cap; i += kSelThreads) out[i] = -1;
  if (B <= 0) return;
  if (B >= T) {                              // budget covers the cache: identity
    for (int i = tid; i < T; i += kSelThreads) out[i] = i;
    return;
  }

  uint32_t prefix = 0, mask = 0, need = (uint32_t)B;
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    for (int t0 = 0; t0 < T; t0 += kSelThreads) {
      const int t = t0 + tid;
      const bool in = t < T;
      const uint32_t key = in ? float_order_key(__ldcg(row + t)) : 0u;
      const bool live = in && ((key & mask) == prefix);
      const uint32_t digit = live ? ((key >> shift) & 255u) : 256u + (uint32_t)lane;   // dead lanes match nobody
      const uint32_t peers = __match_any_sync(0xFFFFFFFFu, digit);
      if (live && lane == (__ffs(peers) - 1)) atomicAdd(&hist[digit], (uint32_t)__popc(peers));
    }
    __syncthreads();
    if (wid == 0) {
      // lane l owns bins 255-8l .. 248-8l (descending); find the bin where the running count reaches `need`
      uint32_t c[8], sum = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) { c[i] = hist[255 - 8 * lane - i]; sum += c[i]; }
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
      }
      const uint32_t excl = incl - sum;
      const uint32_t hit = __ballot_sync(0xFFFFFFFFu, incl >= need);
      if (lane == (__ffs(hit) - 1)) {
        uint32_t cum = excl;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (cum + c[i] >= need) {
            s_prefix = prefix | ((uint32_t)(255 - 8 * lane - i) << shift);
            s_need = need - cum;
            break;
          }
          cum += c[i];
        }
      }
    }
    __syncthreads();
    prefix = s_prefix;
    need = s_need;
    mask |= 255u << shift;
  }
  // prefix = code of the B-th largest score; take every row above it and the first `need` rows equal to it
  const uint32_t thr = prefix;
  uint32_t run_gt = 0, run_eq = 0;
  for (int t0 = 0; t0 < T; t0 += kSelThreads) {
    const int t = t0 + tid;
    const uint32_t key = (t < T) ? float_order_key(__ldcg(row + t)) : 0u;
    const bool gt = (t < T) && key > thr;
    const bool eq = (t < T) && key == thr;
    const uint32_t b_gt = __ballot_sync(0xFFFFFFFFu, gt);
    const uint32_t b_eq = __ballot_sync(0xFFFFFFFFu, eq);
    if (lane == 0) warp_tot[wid] = (uint32_t)__popc(b_gt) | ((uint32_t)__popc(b_eq) << 16);
    __syncthreads();
    if (wid == 0) {
      const uint32_t v = warp_tot[lane];
      uint32_t incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += u;
      }
      warp_off[lane] = incl - v;
      if (lane == 31) warp_off[32] = incl;
    }
    __syncthreads();
    const uint32_t off = warp_off[wid], tot = warp_off[32];
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t gt_before = run_gt + (off & 0xFFFFu) + (uint32_t)__popc(b_gt & lt);
    const uint32_t eq_before = run_eq + (off >> 16) + (uint32_t)__popc(b_eq & lt);
    if (gt || (eq && eq_before < need)) out[gt_before + min(eq_before, need)] = t;
    run_gt += tot & 0xFFFFu;
    run_eq += tot >> 16;
  }
}


template <int ITEMS, int CL>
__global__ void __launch_bounds__(kRegThreads) select_keys_reg_kernel(DevParams P, const float* __restrict__ scores,
                                                                       int32_t* __restrict__ k_idx,
                                                                       int32_t* __restrict__ k_cnt) {
  __shared__ SelectSmem<ITEMS, CL> sm;
  grid_launch_dependents();     // the attention kernel may start now: it waits for this grid itself before it reads the list
  const int rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const int head = blockIdx.x / CL;
  const int s = head / P.n_kv, kv = head % P.n_kv;
  const int tid = threadIdx.x;
  const int T = __ldg(P.ctx_len + s);
  const int B = key_budget(T, P.kv_budget, P.budget_frac);
  const float* row = scores + (long long)head * P.max_ctx;
  int32_t* out = k_idx + (long long)head * P.budget_cap;
  const int gtid = rank * kRegThreads + tid;
  constexpr int kAll = CL * kRegThreads;
  if (kv == 0 && gtid == 0) k_cnt[s] = B;
  for (int i = B + gtid; i < P.budget_cap; i += kAll) out[i] = -1;
  // Every exit path waits for the kernel before this one: the kernels of a fused call are ordered as a chain, and
  // "the last kernel has completed" implies "all of them have" only if no link finishes without having waited.
  if (B <= 0) { grid_dependency_wait(); return; }      // uniform over the cluster
  if (B >= T) {                                 // budget covers the cache: identity
    for (int i = gtid; i < T; i += kAll) out[i] = i;
    grid_dependency_wait();
    return;
  }
  const Selected sel = select_row<ITEMS, CL, 8>(P, row, T, B, rank, sm, out);
  if (sel.mine <= (uint32_t)kHistWords) {       // copied out with full-width stores
    __syncthreads();
    for (uint32_t i = tid; i < sel.mine && sel.before + i < (uint32_t)B; i += kRegThreads) out[sel.before + i] = (int32_t)sm.hist_all[i];
  }
}

template <int ITEMS, int CL>
static cudaError_t launch_reg(const DevParams& P, const float* scores, int32_t* k_idx, int32_t* k_cnt, cudaStream_t st,
                              bool chained) {
  return launch_kernel("select_keys_reg", select_keys_reg_kernel<ITEMS, CL>, dim3(P.batch * P.n_kv * CL), dim3(kRegThreads), 0, st, CL, chained,
                       P, scores, k_idx, k_cnt);
}

template <int CL>
static cudaError_t launch_cl(const DevParams& P, const float* scores, int32_t* k_idx, int32_t* k_cnt, cudaStream_t st,
                             bool chained) {
  const int per_thread = (P.max_ctx + CL * kRegThreads - 1) / (CL * kRegThreads);
  if (per_thread <= 8) return launch_reg<8, CL>(P, scores, k_idx, k_cnt, st, chained);
  if (per_thread <= 16) return launch_reg<16, CL>(P, scores, k_idx, k_cnt, st, chained);
  if (per_thread <= 32) return launch_reg<32, CL>(P, scores, k_idx, k_cnt, st, chained);
  return launch_reg<64, CL>(P, scores, k_idx, k_cnt, st, chained);
}

cudaError_t launch_select_keys(const DevParams& P, const float* scores, int32_t* k_idx, int32_t* k_cnt,
                               cudaStream_t st, bool chained) {
  const int per_thread = (P.max_ctx + kRegThreads - 1) / kRegThreads;    // items per thread with one CTA per row
  const int rows = P.batch * P.n_kv;
  // Cluster width.  Clusters pay while all of them are resident together, about one CTA per SM (14 of eight CTAs, 32 of
  // four, 72 of two; beyond that the time doubles), and for rows long enough to cut the loops by more than the two
  // cluster barriers cost.  Stand-alone launches of 8 rows with 1 / 2 / 4 / 8 CTAs each: 8192 scores 6.0 / 6.4 / 6.3 /
  // 6.6 us, 16384 scores 8.3 / 7.2 / 6.5 / 6.8, 32768 scores 13.2 / 10.1 / 7.7 / 7.0; 128 rows of 32768: 13.8 / 20.0 /
  // 18.7 / 30.5.
  int cl = 1;
  if (per_thread > 32 && rows <= 14) cl = 8;
  else if (per_thread > 16 && rows <= 32) cl = 4;
  else if (per_thread > 16 && rows <= 72) cl = 2;
  while (cl * 64 < per_thread && cl < 8) cl *= 2;
  cudaError_t e;
  if (per_thread > 8 * 64) e = launch_kernel("select_keys", select_keys_kernel, dim3(P.batch * P.n_kv), dim3(kSelThreads), 0, st, 1, chained, P, scores, k_idx, k_cnt);
  else if (cl == 8) e = launch_cl<8>(P, scores, k_idx, k_cnt, st, chained);
  else if (cl == 4) e = launch_cl<4>(P, scores, k_idx, k_cnt, st, chained);
  else if (cl == 2) e = launch_cl<2>(P, scores, k_idx, k_cnt, st, chained);
  else e = launch_cl<1>(P, scores, k_idx, k_cnt, st, chained);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace quoka
