// Generation phase (a chunk of ONE query per sequence; Section 4.4, Appendix B): Algorithm 1 skips the query
// sub-selection, Q-bar is one vector per KV head, and the two contraction steps lose their matrix shape:
//   scoring    S^_t = (Qbar . k_t) / |k_t|  is a matrix-vector product that reads every cached key once:
//              HBM-bound, 2 flops per 2 bytes.  score_keys_gemv_kernel streams the keys through a ring per warp.
//   attention  each query head attends B + 1 rows.  decode_attn_kernel gathers them once per KV group, a few rows per
//              warp with an online softmax of its own, the keys cut into parts over a cluster.
// The tensor-core kernels would spend a 128-row MMA tile on one query.  Everything is fp32 arithmetic on the
// stored values; the softmax weights are not rounded to bf16 here.
#include "decode_tiles.cuh"
#include "qbar.cuh"
#include "sm100_ptx.cuh"

namespace quoka {

constexpr int kDecodeAttnThreads = 256;

// ------------------------------------------------------------------------------------------ scoring (N = 1)
// Persistent warps, each with an equal contiguous share of the valid units of 4 KB (kUnr rows per lane group) of the
// (sequence, KV head, row) list.  LPR lanes share a row, the words c and c + LPR of 16 bytes
// each (a warp's copies then ask for every 32-byte sector once: with adjacent words, which asked twice, 3.3 TB/s).
//
// What bounds it: HBM for long caches, one DRAM round trip for short ones.  Every warp keeps kGemvStages units in
// flight in a ring of its own, filled with cp.async (the lane that copies a word is the lane that reads it: no barrier
// anywhere); page numbers are fetched one unit ahead.  8 x 32768 rows of 128 bf16: 16.7 -> 14.7 us stand-alone; 16 sequences
// of them 190 -> 169 us (6.4 TB/s); 16 paged ones of 8K to 32K rows with cached norms 147 -> 115 us (a grid of 512-row CTAs,
// empty ones among them, before).
//
// In a fused call (`q` given) the kernel forms Q-bar itself, under the first keys' flight: the group's G queries are 1 KB,
// and one launch less is worth more than the work of doing it once per warp.  Same arithmetic and rounding as
// aggregate_queries_kernel.
constexpr int kGemvThreads = 384;
constexpr int kGemvStages = 3;
constexpr int kGemvUnr = 4;
constexpr int kGemvUnitBytes = 32 * 32 * kGemvUnr;
constexpr size_t kGemvSmem = (size_t)(kGemvThreads / 32) * kGemvStages * (kGemvUnitBytes + 128);

template <typename T, int D>
constexpr int gemv_unit_rows() { return kGemvUnitBytes / (D * (int)sizeof(T)); }

// Position in the list of units: the u-th unit of (sequence s, KV head kv), `left` units before the warp's share ends; T rows
// in the sequence.
struct UnitWalk {
  int s, kv, u, units_s, left, T;
  __device__ __forceinline__ void next(const DevParams& P, int unit_rows) {
    --left;
    if (++u < units_s || left <= 0) return;
    u = 0;
    if (++kv < P.n_kv) return;
    kv = 0;
    do { T = load_input<true>(P.ctx_len + ++s); units_s = (T + unit_rows - 1) / unit_rows; } while (units_s == 0);
  }
};

template <typename T, int D>
__global__ void __launch_bounds__(kGemvThreads, 1) score_keys_gemv_kernel(DevParams P, const T* __restrict__ q,
                                                                           const T* __restrict__ qbar,
                                                                           const T* __restrict__ k,
                                                                           float* __restrict__ scores) {
  constexpr int NE = VecOf<T>::N;                    // elements per 16-byte word
  constexpr int LPR = D / (2 * NE);                  // lanes per row
  constexpr int RPW = 32 / LPR;                      // rows per warp instruction
  constexpr int ROWS = RPW * kGemvUnr;               // rows per unit: a divisor of the page size
  constexpr int kRep = LPR / kGemvUnr;               // lanes that hold the same row's sum
  static_assert(ROWS * D * (int)sizeof(T) == kGemvUnitBytes && kPage % ROWS == 0 && LPR >= kGemvUnr, "unit");
  extern __shared__ __align__(16) unsigned char gemv_smem[];
  grid_dependency_wait();                            // the inputs, and in a staged call Q-bar, come from the kernels before
  grid_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = lane % LPR, rsub = lane / LPR;
  uint4* ring = reinterpret_cast<uint4*>(gemv_smem + (size_t)warp * kGemvStages * kGemvUnitBytes) + lane;   // [stage][8][32]
  float* norms = reinterpret_cast<float*>(gemv_smem + (size_t)(kGemvThreads / 32) * kGemvStages * kGemvUnitBytes) +
                 warp * kGemvStages * 32 + lane;                                                           // [stage][32]
  // ---- this warp's share
  UnitWalk w;
  {
    int total = 0;
    for (int s0 = 0; s0 < P.batch; s0 += 32) {
      const int T_l = s0 + lane < P.batch ? load_input<true>(P.ctx_len + s0 + lane) : 0;
      total += __reduce_add_sync(0xFFFFFFFFu, (T_l + ROWS - 1) / ROWS * P.n_kv);
    }
    const int n_warps = gridDim.x * (kGemvThreads / 32), id = blockIdx.x + gridDim.x * warp;   // (a short list: all SMs)
    int lo = (int)((long long)total * id / n_warps);
    w.left = (int)((long long)total * (id + 1) / n_warps) - lo;
    if (w.left == 0) return;
    for (int s0 = 0;; s0 += 32) {
      const int T_l = s0 + lane < P.batch ? load_input<true>(P.ctx_len + s0 + lane) : 0;
      const int u_l = (T_l + ROWS - 1) / ROWS, n_l = u_l * P.n_kv;
      int incl = n_l;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
      }
      const uint32_t hit = __ballot_sync(0xFFFFFFFFu, incl > lo);
      if (hit != 0) {
        const int src = __ffs(hit) - 1;
        lo -= __shfl_sync(0xFFFFFFFFu, incl - n_l, src);
        w.s = s0 + src;
        w.units_s = __shfl_sync(0xFFFFFFFFu, u_l, src);
        w.T = __shfl_sync(0xFFFFFFFFu, T_l, src);
        w.kv = lo / w.units_s;
        w.u = lo % w.units_s;
        break;
      }
      lo -= __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
  }
  const bool cosine = !P.score_dot;
  const bool cached = cosine && P.k_inv_norm != nullptr;
  const int my_row = c / kRep * RPW + rsub;          // the row of a unit whose score this lane ends up with
  // ---- filling the ring: one group per unit, empty past the share
  UnitWalk in = w;
  const auto page_of = [&](const UnitWalk& at) {
    return P.page_size != 0 && at.left > 0 ? load_input<true>(P.block_table + (long long)at.s * P.max_pages + at.u * ROWS / kPage) : 0;
  };
  int page = page_of(in);
  const auto fill = [&](int stage) {
    if (in.left > 0) {
      const int t0 = in.u * ROWS, T_s = in.T;
      const T* base = P.page_size == 0 ? k + (long long)in.s * P.kv_sb + (long long)in.kv * P.kv_sh + (long long)t0 * P.kv_st
                                       : k + (long long)page * P.kv_sb + (long long)in.kv * P.kv_sh + (long long)(t0 & (kPage - 1)) * P.kv_st;
#pragma unroll
      for (int j = 0; j < kGemvUnr; ++j) {
        const uint4* src = reinterpret_cast<const uint4*>(base + (long long)min(j * RPW + rsub, T_s - 1 - t0) * P.kv_st) + c;
        ptx::cp_async_16(ptx::smem_u32(ring + (stage * 8 + 2 * j) * 32), src, true);
        ptx::cp_async_16(ptx::smem_u32(ring + (stage * 8 + 2 * j + 1) * 32), src + LPR, true);
      }
      if (cached) {
        const int r = min(my_row, T_s - 1 - t0);
        const float* src = P.k_inv_norm + (P.page_size == 0 ? ((long long)in.s * P.n_kv + in.kv) * P.kv_rows + t0 + r
                                                            : ((long long)page * P.n_kv + in.kv) * kPage + (t0 & (kPage - 1)) + r);
        ptx::cp_async_4(ptx::smem_u32(norms + stage * 32), src);
      }
      in.next(P, ROWS);
      page = page_of(in);
    }
    ptx::cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < kGemvStages; ++i) fill(i);
  uint64_t qv[NE];                                   // this lane's 2 NE elements of Q-bar, in pairs
  int s_cur = -1, kv_cur = -1;
  for (int stage = 0; w.left > 0; w.next(P, ROWS)) {
    if (w.s != s_cur || w.kv != kv_cur) {
      s_cur = w.s; kv_cur = w.kv;
      float qf[2 * NE];
      if (q == nullptr) {
        const uint4* qp = reinterpret_cast<const uint4*>(qbar + ((long long)s_cur * P.n_kv + kv_cur) * D) + c;
        word_to_f32<T>(__ldcg(qp), qf);
        word_to_f32<T>(__ldcg(qp + LPR), qf + NE);
      } else {
        constexpr int E = D / 32;                    // elements of a query per lane
        float mean[E];
        mean_normalised_query<T, E>(P, q, s_cur, kv_cur, lane, [](int) { return 0; }, mean);
#pragma unroll
        for (int i = 0; i < E; ++i) mean[i] = to_f32(from_f32<T>(mean[i]));
#pragma unroll
        for (int i = 0; i < 2 * NE; ++i) {
          const int e = (i / NE * LPR + c) * NE + i % NE;          // this lane's i-th element
          qf[i] = __shfl_sync(0xFFFFFFFFu, mean[i % E], e / E);
        }
      }
#pragma unroll
      for (int i = 0; i < NE; ++i) qv[i] = ptx::pack2(qf[2 * i], qf[2 * i + 1]);
    }
    ptx::cp_async_wait<kGemvStages - 1>();
    float dot[kGemvUnr], nn[kGemvUnr];
#pragma unroll
    for (int j = 0; j < kGemvUnr; ++j) {
      const uint4 w0 = ring[(stage * 8 + 2 * j) * 32], w1 = ring[(stage * 8 + 2 * j + 1) * 32];
      float x[2 * NE];
      word_to_f32<T>(w0, x);
      word_to_f32<T>(w1, x + NE);
      uint64_t d2[2] = {0ull, 0ull}, n2[2] = {0ull, 0ull};
#pragma unroll
      for (int i = 0; i < NE; ++i) {
        const uint64_t x2 = ptx::pack2(x[2 * i], x[2 * i + 1]);
        d2[i & 1] = ptx::fma2(x2, qv[i], d2[i & 1]);
        if (cosine && !cached) n2[i & 1] = ptx::fma2(x2, x2, n2[i & 1]);
      }
      float a, b;
      ptx::unpack2(ptx::add2(d2[0], d2[1]), a, b);
      dot[j] = a + b;
      ptx::unpack2(ptx::add2(n2[0], n2[1]), a, b);
      nn[j] = a + b;
    }
    transposing_sum<kGemvUnr, LPR>(dot, c);
    float val = dot[0];
    if (cached) {
      val *= norms[stage * 32];
    } else if (cosine) {
      transposing_sum<kGemvUnr, LPR>(nn, c);
      val /= fmaxf(sqrtf(nn[0]), kNormEps);
    }
    const int t = w.u * ROWS + my_row;
    if (c % kRep == 0 && t < w.T) scores[((long long)s_cur * P.n_kv + kv_cur) * P.max_ctx + t] = val;
    fill(stage);
    if (++stage == kGemvStages) stage = 0;
  }
  ptx::cp_async_wait_all();                          // nothing of this thread is in flight at exit
}

// ------------------------------------------------------------------------------------------ attention (C = 1)
// A CTA takes GH query heads of one KV group and one part of the keys (the listed cached rows, then the query's own row
// T_s); the parts of a group are a cluster and are added up through distributed shared memory, in part order.
//
// What bounds it: latency (a list of 256 rows is 0.13 MB of K and V per KV head), and in a batch the reads.  So a warp
// fetches its list entries, then K AND V of its rows together: two memory round trips for up to 64 rows per CTA; the
// heads of a group share the rows; and each warp keeps its own running maximum, so that nothing but the final sum
// crosses warps (decode_tiles.cuh).
//   One sequence, 8 KV heads of 4, listed rows 256 / 4000 / 16000: 9.7 / 82 / 221 -> 6.8 / 17.5 / 56 us (one CTA per query
//   head, logits in shared memory, K and V one after the other, before); 16 sequences, 256 / 4000 rows: 19.5 / 251 ->
//   11.1 / 93 us; without a list, 32768 rows: 405 -> 134 us (a 128-row tensor-core tile for one query, before).
template <typename T, int D, int GH>
__global__ void __launch_bounds__(kDecodeAttnThreads, 2) decode_attn_kernel(DevParams P, const T* __restrict__ q,
                                                                          const T* __restrict__ k,
                                                                          const T* __restrict__ v,
                                                                          const int32_t* __restrict__ k_idx,
                                                                          const int32_t* __restrict__ k_cnt,
                                                                          T* __restrict__ out, float* __restrict__ lse,
                                                                          int parts) {
  constexpr int kWarps = kDecodeAttnThreads / 32;
  __shared__ DecodeWarps<D, GH, kWarps> w;
  __shared__ DecodePart<D, GH> mine;
  grid_launch_dependents();                          // the next call's first kernel, which waits for this grid's end
  const int part = blockIdx.x % parts, unit = blockIdx.x / parts, s = blockIdx.y;
  const int blocks = (P.group + GH - 1) / GH;        // CTAs per KV group (more than one for groups beyond 4 heads:
                                                     // eight heads per CTA take 230 registers and a second wave)
  const int kv = unit / blocks, g0 = (unit % blocks) * GH, h0 = kv * P.group + g0;
  const int n_heads = min(GH, P.group - g0);
  const int T_s = __ldg(P.ctx_len + s);
  float qv[GH][VecOf<T>::N];
  decode_load_q<T, D, GH>(P, q, s, h0, n_heads, (threadIdx.x & 31) % (D / VecOf<T>::N), qv);
  grid_dependency_wait();                            // the list comes from the kernel before
  const int cnt = k_idx ? __ldcg(k_cnt + s) : T_s;   // without a list: every cached row (Eq. 2)
  const int32_t* idx = k_idx ? k_idx + ((long long)s * P.n_kv + kv) * P.budget_cap : nullptr;
  const int n_keys = cnt + 1;
  const int u_lo = (int)((long long)part * n_keys / parts), u_hi = (int)((long long)(part + 1) * n_keys / parts);
  decode_attend<T, D, GH, kWarps>(P, k, v, s, kv, qv, u_lo, u_hi,
                                  [&](int u) { return u < cnt ? (idx ? __ldcg(idx + u) : u) : T_s; }, w, mine);
  decode_merge<T, D, GH, kWarps>(P, mine, part, parts, s, h0, n_heads, out, lse);
}

// ---------------------------------------------------------------------------------------------- host
bool decode_path_applies(const DevParams& P) {
  return P.chunk == 1 && P.n_sel == 1;
}

template <typename T, int D>
static cudaError_t launch_gemv_t(const DevParams& P, const void* q, const void* qbar, const void* k, float* scores,
                                 cudaStream_t st, bool chained) {
  const int sms = device_sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  const long long units = (long long)P.batch * P.n_kv * ((P.max_ctx + gemv_unit_rows<T, D>() - 1) / gemv_unit_rows<T, D>());
  const long long ctas = (units + kGemvThreads / 32 - 1) / (kGemvThreads / 32);
  cudaError_t e = cudaFuncSetAttribute(score_keys_gemv_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemvSmem);
  if (e != cudaSuccess) return e;
  return launch_kernel("score_keys_gemv", score_keys_gemv_kernel<T, D>, dim3((unsigned)(ctas < sms ? ctas : sms)), dim3(kGemvThreads),
                       kGemvSmem, st, 1, chained, P, (const T*)q, (const T*)qbar, (const T*)k, scores);
}

// q != nullptr: Q-bar is formed from the queries in the kernel, `qbar` is not read.
cudaError_t launch_score_keys_gemv(const DevParams& P, int dtype, const void* q, const void* qbar, const void* k,
                                   float* scores, cudaStream_t st, bool chained) {
  if (P.max_ctx <= 0) return cudaSuccess;
  cudaError_t e;
  if (dtype == QUOKA_BF16) e = P.d == 128 ? launch_gemv_t<__nv_bfloat16, 128>(P, q, qbar, k, scores, st, chained) : launch_gemv_t<__nv_bfloat16, 64>(P, q, qbar, k, scores, st, chained);
  else e = P.d == 128 ? launch_gemv_t<float, 128>(P, q, qbar, k, scores, st, chained) : launch_gemv_t<float, 64>(P, q, qbar, k, scores, st, chained);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

template <typename T, int D, int GH>
static cudaError_t launch_decode_attn_t(const DevParams& P, const void* q, const void* k, const void* v, const int32_t* k_idx,
                                        const int32_t* k_cnt, void* out, float* lse, cudaStream_t st, bool chained) {
  // Parts: one trip of every warp where the SMs have room for them (two CTAs each), at most a portable cluster.
  const long long keys = (k_idx ? (long long)P.budget_cap : (long long)P.max_ctx) + 1;
  const int rows = 32 / (D / VecOf<T>::N) * kDecodeUnroll * (kDecodeAttnThreads / 32);
  const long long units = (long long)P.batch * P.n_kv * ((P.group + GH - 1) / GH), room = 2ll * device_sm_count() / units;
  long long parts = (keys + rows - 1) / rows;
  if (parts > room) parts = room;
  if (parts > 8) parts = 8;
  if (parts < 1) parts = 1;
  const dim3 grid((unsigned)(units / P.batch * parts), P.batch), block(kDecodeAttnThreads);
  return launch_kernel("decode_attn", decode_attn_kernel<T, D, GH>, grid, block, 0, st, (int)parts, chained, P, (const T*)q,
                       (const T*)k, (const T*)v, k_idx, k_cnt, (T*)out, lse, (int)parts);
}

cudaError_t launch_decode_attn(const DevParams& P, int dtype, const void* q, const void* k, const void* v,
                               const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st,
                               bool chained) {
  cudaError_t e;
#define QUOKA_DECODE_ATTN(T_, D_)                                                                            \
  do {                                                                                                       \
    if (P.group == 1) e = launch_decode_attn_t<T_, D_, 1>(P, q, k, v, k_idx, k_cnt, out, lse, st, chained);  \
    else if (P.group == 2) e = launch_decode_attn_t<T_, D_, 2>(P, q, k, v, k_idx, k_cnt, out, lse, st, chained); \
    else e = launch_decode_attn_t<T_, D_, 4>(P, q, k, v, k_idx, k_cnt, out, lse, st, chained);               \
  } while (0)
  if (dtype == QUOKA_BF16) {
    if (P.d == 128) QUOKA_DECODE_ATTN(__nv_bfloat16, 128); else QUOKA_DECODE_ATTN(__nv_bfloat16, 64);
  } else {
    if (P.d == 128) QUOKA_DECODE_ATTN(float, 128); else QUOKA_DECODE_ATTN(float, 64);
  }
#undef QUOKA_DECODE_ATTN
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace quoka
