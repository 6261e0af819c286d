// Key selection and attention of a generation step in one launch (Algorithm 1: I = topk(S^, B_SA); Algorithm 2's attention
// line for a chunk of one query), for problems whose (sequence, KV head) rows number about as many as the GPU has room for
// clusters.
//
// What bounds it: latency.  As two kernels the list went through memory, and the second one's start, its read of the list
// and the first one's end were on the path.  Here a cluster of eight CTAs selects from a row of scores (select_row.cuh), and
// every CTA goes on with the rows of its own eighth of the cache, straight from its list in shared memory; the parts are
// added up through distributed shared memory, in rank order.  Append and step in a graph, one sequence, 8 KV heads of 4, 256
// listed rows, two launches / one: 4003 cached rows 18.4 / 17.5 us, 16384 23.3 / 21.4, 100000 60.5 / 57.0; 2000 listed rows of
// 16384 28.6 / 25.6.  (The parts are as uneven as the selection: a list that lies in one eighth of the cache is gathered by
// one CTA.)
#include "decode_tiles.cuh"
#include "select_row.cuh"

namespace quoka {

constexpr int kFuseCl = 8;
constexpr int kFuseShort = kFuseCl * kRegThreads * 8;        // rows that fit 8 items per thread

template <typename T, int D, int GH, int ITEMS>
__global__ void __launch_bounds__(kRegThreads, 1) decode_select_attn_kernel(DevParams P, const T* __restrict__ q,
                                                                             const T* __restrict__ k, const T* __restrict__ v,
                                                                             const float* __restrict__ scores,
                                                                             int32_t* __restrict__ k_idx,
                                                                             int32_t* __restrict__ k_cnt, T* __restrict__ out) {
  __shared__ union Smem {
    SelectSmem<ITEMS, kFuseCl> sel;
    DecodeWarps<D, GH, kRegWarps> w;                 // once the list has been read
  } sm;
  __shared__ DecodePart<D, GH> mine;
  grid_launch_dependents();                          // the next call's first kernel, which waits for this grid's end
  const int rank = (int)cg::this_cluster().block_rank(), tid = threadIdx.x;
  const int blocks = (P.group + GH - 1) / GH, unit = blockIdx.x / kFuseCl, head = unit / blocks;
  const int s = head / P.n_kv, kv = head % P.n_kv, g0 = (unit % blocks) * GH, h0 = kv * P.group + g0;
  const int n_heads = min(GH, P.group - g0);
  const int T_s = __ldg(P.ctx_len + s);
  const int B = key_budget(T_s, P.kv_budget, P.budget_frac);
  float qv[GH][VecOf<T>::N];
  decode_load_q<T, D, GH>(P, q, s, h0, n_heads, (tid & 31) % (D / VecOf<T>::N), qv);
  int32_t* list = k_idx != nullptr && g0 == 0 ? k_idx + (long long)head * P.budget_cap : nullptr;
  if (k_cnt != nullptr && kv == 0 && g0 == 0 && rank == 0 && tid == 0) k_cnt[s] = B;
  if (list != nullptr)
    for (int i = B + rank * kRegThreads + tid; i < P.budget_cap; i += kFuseCl * kRegThreads) list[i] = -1;
  const bool all = B >= T_s;                         // the budget covers the cache (an empty one too)
  int first = (int)((long long)rank * T_s / kFuseCl), n = (int)((long long)(rank + 1) * T_s / kFuseCl) - first;
  if (all) {
    grid_dependency_wait();
  } else if (B > 0) {
    const Selected sel = select_row<ITEMS, kFuseCl, ITEMS == 8 ? 1 : 8>(P, scores + (long long)head * P.max_ctx, T_s, B, rank, sm.sel, nullptr);
    first = (int)sel.before;
    n = (int)sel.mine;
    __syncthreads();
  } else {
    grid_dependency_wait();
    n = 0;
  }
  if (list != nullptr)
    for (int i = tid; i < n; i += kRegThreads) list[first + i] = all ? first + i : (int)sm.sel.hist_all[i];
  // the last CTA takes the query's own row as well
  decode_attend<T, D, GH, kRegWarps>(P, k, v, s, kv, qv, 0, n + (rank == kFuseCl - 1 ? 1 : 0),
                                     [&](int u) { return u >= n ? T_s : (all ? first + u : (int)sm.sel.hist_all[u]); }, sm.w, mine);
  decode_merge<T, D, GH, kRegWarps>(P, mine, rank, kFuseCl, s, h0, n_heads, out, nullptr);
}

// The attention of the staged call on the same problems: the list is cut at the same cache positions and added up in the
// same order, so that the staged calls give the fused one's bits.
template <typename T, int D, int GH>
__global__ void __launch_bounds__(kRegThreads, 1) decode_listed_attn_kernel(DevParams P, const T* __restrict__ q,
                                                                             const T* __restrict__ k, const T* __restrict__ v,
                                                                             const int32_t* __restrict__ k_idx,
                                                                             const int32_t* __restrict__ k_cnt,
                                                                             T* __restrict__ out, float* __restrict__ lse) {
  __shared__ DecodeWarps<D, GH, kRegWarps> w;
  __shared__ DecodePart<D, GH> mine;
  __shared__ int s_lo, s_hi;
  const int rank = (int)cg::this_cluster().block_rank(), tid = threadIdx.x;
  const int blocks = (P.group + GH - 1) / GH, unit = blockIdx.x / kFuseCl, head = unit / blocks;
  const int s = head / P.n_kv, kv = head % P.n_kv, g0 = (unit % blocks) * GH, h0 = kv * P.group + g0;
  const int n_heads = min(GH, P.group - g0);
  const int T_s = __ldg(P.ctx_len + s), cnt = __ldg(k_cnt + s);
  const int32_t* idx = k_idx + (long long)head * P.budget_cap;
  float qv[GH][VecOf<T>::N];
  decode_load_q<T, D, GH>(P, q, s, h0, n_heads, (tid & 31) % (D / VecOf<T>::N), qv);
  if (tid == 0) { s_lo = 0; s_hi = 0; }
  __syncthreads();
  int lo = (int)((long long)rank * cnt / kFuseCl), hi = (int)((long long)(rank + 1) * cnt / kFuseCl);    // (cnt >= T_s: all)
  if (cnt < T_s) {                                   // entries below the first position of this CTA, and of the next
    const int piece = P.max_ctx <= kFuseShort ? select_piece<kFuseCl, 1>(T_s) : select_piece<kFuseCl, 8>(T_s);
    int a = 0, b = 0;
    for (int i = tid; i < cnt; i += kRegThreads) {
      const int t = __ldg(idx + i);
      a += t < rank * piece ? 1 : 0;
      b += t < (rank + 1) * piece ? 1 : 0;
    }
    a = __reduce_add_sync(0xFFFFFFFFu, a);
    b = __reduce_add_sync(0xFFFFFFFFu, b);
    if ((tid & 31) == 0) { atomicAdd(&s_lo, a); atomicAdd(&s_hi, b); }
    __syncthreads();
    lo = s_lo; hi = s_hi;
  }
  const int n = hi - lo;
  decode_attend<T, D, GH, kRegWarps>(P, k, v, s, kv, qv, 0, n + (rank == kFuseCl - 1 ? 1 : 0),
                                     [&](int u) { return u >= n ? T_s : __ldg(idx + lo + u); }, w, mine);
  decode_merge<T, D, GH, kRegWarps>(P, mine, rank, kFuseCl, s, h0, n_heads, out, lse);
}

// Up to 14 clusters of eight CTAs, one CTA per SM, are resident together on a B200; the list of a CTA has to fit its shared
// memory, the row its registers.  Below 2K rows a single CTA selects faster than a cluster's barriers take (append and step,
// 8 KV heads, 256 listed: 1000 rows 15.7 us in two launches, 17.7 in one; 2048: 16.2 / 16.5).
bool decode_select_attn_applies(const DevParams& P) {
  const long long units = (long long)P.batch * P.n_kv * ((P.group + 3) / 4);
  return P.chunk == 1 && P.max_ctx > 2048 && units <= 14 && P.budget_cap <= kHistWords && P.max_ctx <= kFuseCl * kRegThreads * 32;
}

// CALL(T, D, GH) for the problem's data type, head_dim and group
#define QUOKA_DECODE_DISPATCH(CALL)                                                        \
  do {                                                                                     \
    if (dtype == QUOKA_BF16) {                                                             \
      if (P.d == 128) QUOKA_DECODE_GROUP(CALL, __nv_bfloat16, 128); else QUOKA_DECODE_GROUP(CALL, __nv_bfloat16, 64); \
    } else {                                                                               \
      if (P.d == 128) QUOKA_DECODE_GROUP(CALL, float, 128); else QUOKA_DECODE_GROUP(CALL, float, 64); \
    }                                                                                      \
  } while (0)
#define QUOKA_DECODE_GROUP(CALL, T_, D_) \
  do { if (P.group == 1) CALL(T_, D_, 1); else if (P.group == 2) CALL(T_, D_, 2); else CALL(T_, D_, 4); } while (0)

// k_idx and k_cnt may be null.  The kernel before it on the stream is the scoring kernel of the same call.
cudaError_t launch_decode_select_attn(const DevParams& P, int dtype, const void* q, const void* k, const void* v,
                                      const float* scores, int32_t* k_idx, int32_t* k_cnt, void* out, cudaStream_t st) {
  cudaError_t e;
#define QUOKA_CALL(T_, D_, GH_)                                                                                                \
  e = launch_kernel("decode_select_attn", P.max_ctx <= kFuseShort ? decode_select_attn_kernel<T_, D_, GH_, 8>                  \
                                                                  : decode_select_attn_kernel<T_, D_, GH_, 32>,                \
                    dim3((unsigned)(P.batch * P.n_kv * ((P.group + GH_ - 1) / GH_) * kFuseCl)), dim3(kRegThreads), 0, st,      \
                    kFuseCl, /*chained=*/true, P, (const T_*)q, (const T_*)k, (const T_*)v, scores, k_idx, k_cnt, (T_*)out)
  QUOKA_DECODE_DISPATCH(QUOKA_CALL);
#undef QUOKA_CALL
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_decode_listed_attn(const DevParams& P, int dtype, const void* q, const void* k, const void* v,
                                      const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st) {
  cudaError_t e;
#define QUOKA_CALL(T_, D_, GH_)                                                                                                \
  e = launch_kernel("decode_listed_attn", decode_listed_attn_kernel<T_, D_, GH_>,                                              \
                    dim3((unsigned)(P.batch * P.n_kv * ((P.group + GH_ - 1) / GH_) * kFuseCl)), dim3(kRegThreads), 0, st,      \
                    kFuseCl, /*chained=*/false, P, (const T_*)q, (const T_*)k, (const T_*)v, k_idx, k_cnt, (T_*)out, lse)
  QUOKA_DECODE_DISPATCH(QUOKA_CALL);
#undef QUOKA_CALL
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace quoka
