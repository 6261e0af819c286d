// Generation phase (a chunk of ONE query per sequence; Section 4.4, Appendix B): Algorithm 1 skips the query
// sub-selection, Q-bar is one vector per KV head, and the two contraction steps lose their matrix shape:
//   scoring    S^_t = (Qbar . k_t) / |k_t|  is a matrix-vector product that reads every cached key once:
//              HBM-bound, 2 flops per 2 bytes.  score_keys_gemv_kernel streams the keys with 16-byte loads,
//              32 bytes of a row per lane, four rows in flight per lane.
//   attention  each query head attends B + 1 rows.  decode_attn_kernel gathers them once per KV group, a few rows per
//              warp with an online softmax of its own, the keys cut into parts over a cluster.
// The tensor-core kernels would spend a 128-row MMA tile on one query.  Everything is fp32 arithmetic on the
// stored values; the softmax weights are not rounded to bf16 here.
#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace quoka {

constexpr int kGemvThreads = 256;
constexpr int kGemvRowsPerCta = 512;
constexpr int kDecodeAttnThreads = 256;

// 8 consecutive elements as floats from one 16-byte word (bf16) or two (f32 uses 4 per word: see LPR below).
template <typename T> struct VecOf;
template <> struct VecOf<__nv_bfloat16> { static constexpr int N = 8; };
template <> struct VecOf<float> { static constexpr int N = 4; };

template <typename T>
__device__ __forceinline__ void word_to_f32(const uint4& w, float* x) {
  if constexpr (sizeof(T) == 2) {
    const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) { x[2 * j] = __uint_as_float(v[j] << 16); x[2 * j + 1] = __uint_as_float(v[j] & 0xFFFF0000u); }
  } else {
    x[0] = __uint_as_float(w.x); x[1] = __uint_as_float(w.y); x[2] = __uint_as_float(w.z); x[3] = __uint_as_float(w.w);
  }
}

// ------------------------------------------------------------------------------------------ scoring (N = 1)
// grid = (row slices, KV heads, sequences); a CTA scores kGemvRowsPerCta consecutive cached rows of one
// (sequence, KV head).  LPR lanes share a row, 32 bytes (two 16-byte words, one DRAM sector) each; a warp covers
// 32 / LPR rows per trip and keeps UNR trips (2 * UNR loads per lane) in flight.
template <typename T, int D>
__global__ void __launch_bounds__(kGemvThreads) score_keys_gemv_kernel(DevParams P, const T* __restrict__ qbar,
                                                                        const T* __restrict__ k,
                                                                        float* __restrict__ scores) {
  constexpr int NE = VecOf<T>::N;                    // elements per 16-byte word
  constexpr int LPR = D / (2 * NE);                  // lanes per row
  constexpr int RPW = 32 / LPR;                      // rows per warp trip
  constexpr int UNR = 4;
  grid_launch_dependents();
  const int s = blockIdx.z, kv = blockIdx.y;
  const int T_s = __ldg(P.ctx_len + s);
  const int row0 = blockIdx.x * kGemvRowsPerCta;
  if (row0 >= T_s) { grid_dependency_wait(); return; }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = lane % LPR, rsub = lane / LPR;
  grid_dependency_wait();                            // Q-bar comes from the kernel before
  float qv[2 * NE];
  {
    const uint4* qp = reinterpret_cast<const uint4*>(qbar + ((long long)s * P.n_kv + kv) * D) + 2 * c;
    word_to_f32<T>(__ldcg(qp), qv);
    word_to_f32<T>(__ldcg(qp + 1), qv + NE);
  }
  const bool cosine = !P.score_dot;
  const bool cached = cosine && P.k_inv_norm != nullptr;
  float* out = scores + ((long long)s * P.n_kv + kv) * P.max_ctx;
  const int row_end = min(T_s, row0 + kGemvRowsPerCta);
  constexpr int kWarps = kGemvThreads / 32;
  for (int r = row0 + warp * RPW * UNR; r < row_end; r += kWarps * RPW * UNR) {
    uint4 w[UNR][2];
    int t[UNR];
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      t[u] = r + u * RPW + rsub;
      const int tc = min(t[u], row_end - 1);         // clamped: no branch around the loads
      const uint4* kp = reinterpret_cast<const uint4*>(k + kv_row_offset(P, s, kv, tc)) + 2 * c;
      w[u][0] = __ldg(kp);
      w[u][1] = __ldg(kp + 1);
    }
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      float x[2 * NE];
      word_to_f32<T>(w[u][0], x);
      word_to_f32<T>(w[u][1], x + NE);
      float dot = 0.f, dot1 = 0.f, nn = 0.f, nn1 = 0.f;
#pragma unroll
      for (int i = 0; i < NE; ++i) {
        dot = fmaf(x[i], qv[i], dot); nn = fmaf(x[i], x[i], nn);
        dot1 = fmaf(x[NE + i], qv[NE + i], dot1); nn1 = fmaf(x[NE + i], x[NE + i], nn1);
      }
      dot += dot1; nn += nn1;
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) {
        dot += __shfl_xor_sync(0xFFFFFFFFu, dot, o);
        nn += __shfl_xor_sync(0xFFFFFFFFu, nn, o);
      }
      if (c == 0 && t[u] < row_end) {
        float val = dot;
        if (cached) val = dot * __ldg(P.k_inv_norm + kv_norm_index(P, s, kv, t[u]));
        else if (cosine) val = dot / fmaxf(sqrtf(nn), kNormEps);
        out[t[u]] = val;
      }
    }
  }
}

// ------------------------------------------------------------------------------------------ attention (C = 1)
// A CTA takes GH query heads of one KV group and one part of the keys (the listed cached rows, then the query's own row
// T_s); the parts of a group are a cluster and are added up through distributed shared memory, in part order.
//
// What bounds it: latency (a list of 256 rows is 0.13 MB of K and V per KV head), and in a batch the reads.  So a warp
// fetches its list entries, then K AND V of its rows together: two memory round trips for up to 64 rows per CTA; the
// heads of a group share the rows; and each warp keeps its own running maximum, so that nothing but the final sum
// crosses warps.  LPR lanes share a row; the UNR x GH partial products of a lane are summed over those lanes by a
// transposing butterfly that leaves one logit per lane, where its exponential is taken once.
//   One sequence, 8 KV heads of 4, listed rows 256 / 4000 / 16000: 9.7 / 82 / 221 -> 6.8 / 17.5 / 56 us (one CTA per query
//   head, logits in shared memory, K and V one after the other, before); 16 sequences, 256 / 4000 rows: 19.5 / 251 ->
//   11.1 / 93 us; without a list, 32768 rows: 405 -> 134 us (a 128-row tensor-core tile for one query, before).
constexpr int kDecodeUnroll = 4;

// v[0 .. NV) summed over the LPR lanes of a row; afterwards lane c of them holds the values c * NV / LPR + i (NV >= LPR)
// or the one value c / (LPR / NV) (NV < LPR).
template <int NV, int LPR>
__device__ __forceinline__ void transposing_sum(float (&v)[NV], int c) {
  int n = NV;
#pragma unroll
  for (int o = LPR / 2; o > 0; o >>= 1) {
    if (n > 1) {
      n /= 2;
      const bool up = (c & o) != 0;
#pragma unroll
      for (int i = 0; i < NV / 2; ++i)
        if (i < n) {
          const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
          v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
        }
    } else {
      v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
    }
  }
}

template <typename T, int D, int GH>
__global__ void __launch_bounds__(kDecodeAttnThreads, 2) decode_attn_kernel(DevParams P, const T* __restrict__ q,
                                                                          const T* __restrict__ k,
                                                                          const T* __restrict__ v,
                                                                          const int32_t* __restrict__ k_idx,
                                                                          const int32_t* __restrict__ k_cnt,
                                                                          T* __restrict__ out, float* __restrict__ lse,
                                                                          int parts) {
  constexpr int NE = VecOf<T>::N;
  constexpr int LPR = D / NE;                        // lanes per row
  constexpr int RPW = 32 / LPR;                      // rows per warp instruction
  constexpr int UNR = kDecodeUnroll;
  constexpr int kRows = RPW * UNR;                   // rows per warp and trip
  constexpr int kWarps = kDecodeAttnThreads / 32;
  constexpr int NV = UNR * GH;
  constexpr int PER = NV >= LPR ? NV / LPR : 1;      // logits a lane holds after the transposing sum
  constexpr int kRep = NV < LPR ? LPR / NV : 1;      // lanes that hold the same one
  __shared__ float w_m[kWarps][GH], w_l[kWarps][GH];
  __shared__ __align__(16) float w_o[kWarps][GH][D];
  __shared__ __align__(16) float part_o[GH][D];
  __shared__ float part_m[GH], part_l[GH];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = lane % LPR, rsub = lane / LPR;
  const int part = blockIdx.x % parts, unit = blockIdx.x / parts, s = blockIdx.y;
  const int blocks = (P.group + GH - 1) / GH;        // CTAs per KV group (more than one for groups beyond 4 heads:
                                                     // eight heads per CTA take 230 registers and a second wave)
  const int kv = unit / blocks, g0 = (unit % blocks) * GH, h0 = kv * P.group + g0;
  const int n_heads = min(GH, P.group - g0);
  const int T_s = __ldg(P.ctx_len + s);
  float qv[GH][NE];
#pragma unroll
  for (int g = 0; g < GH; ++g) {
    const int h = h0 + min(g, n_heads - 1);          // a head past the group's end repeats the last one, unused
    const uint4 w = __ldg(reinterpret_cast<const uint4*>(q + (long long)s * P.q_sb + (long long)h * P.q_sh) + c);
    word_to_f32<T>(w, qv[g]);
#pragma unroll
    for (int i = 0; i < NE; ++i) qv[g][i] *= P.scale;
  }
  grid_dependency_wait();                            // the list comes from the kernel before
  const int cnt = k_idx ? __ldcg(k_cnt + s) : T_s;   // without a list: every cached row (Eq. 2)
  const int32_t* idx = k_idx ? k_idx + ((long long)s * P.n_kv + kv) * P.budget_cap : nullptr;
  const int n_keys = cnt + 1;
  const int u_lo = (int)((long long)part * n_keys / parts), u_hi = (int)((long long)(part + 1) * n_keys / parts);
  const auto row_of = [&](int u) { return u < cnt ? (idx ? __ldcg(idx + u) : u) : T_s; };
  float m[PER], l[PER], acc[GH][NE];                 // m, l: of the head this lane's logits belong to
#pragma unroll
  for (int i = 0; i < PER; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
#pragma unroll
  for (int g = 0; g < GH; ++g)
#pragma unroll
    for (int i = 0; i < NE; ++i) acc[g][i] = 0.f;
  for (int u0 = u_lo + warp * kRows; u0 < u_hi; u0 += kWarps * kRows) {
    int t[UNR];
#pragma unroll
    for (int j = 0; j < UNR; ++j) t[j] = row_of(min(u0 + j * RPW + rsub, u_hi - 1));
    uint4 kw[UNR], vw[UNR];
#pragma unroll
    for (int j = 0; j < UNR; ++j) {
      const long long off = kv_row_offset(P, s, kv, t[j]);
      kw[j] = __ldg(reinterpret_cast<const uint4*>(k + off) + c);
      vw[j] = __ldg(reinterpret_cast<const uint4*>(v + off) + c);
    }
    float lg[NV];                                    // index j * GH + g
#pragma unroll
    for (int j = 0; j < UNR; ++j) {
      float x[NE];
      word_to_f32<T>(kw[j], x);
#pragma unroll
      for (int g = 0; g < GH; ++g) {
        float dot = 0.f;
#pragma unroll
        for (int i = 0; i < NE; ++i) dot = fmaf(x[i], qv[g][i], dot);
        lg[j * GH + g] = dot;
      }
    }
    transposing_sum<NV, LPR>(lg, c);
    float alpha[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int id = NV >= LPR ? c * PER + i : c / kRep, j = id / GH;
      const float x = u0 + j * RPW + rsub < u_hi ? lg[i] : -INFINITY;
      float mx = fmaxf(m[i], x);
#pragma unroll
      for (int o = LPR / UNR; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));   // rows of the same head
      alpha[i] = __expf(m[i] - mx);                  // (0 on the first trip: m is -inf, mx is not, every warp has a row)
      m[i] = mx;
      lg[i] = __expf(x - mx);
      l[i] = fmaf(l[i], alpha[i], lg[i]);
    }
    if (u0 >= u_lo + kWarps * kRows) {               // not the warp's first trip
#pragma unroll
      for (int g = 0; g < GH; ++g) {
        const float a = __shfl_sync(0xFFFFFFFFu, alpha[g % PER], g / PER * kRep, LPR);
#pragma unroll
        for (int i = 0; i < NE; ++i) acc[g][i] *= a;
      }
    }
#pragma unroll
    for (int j = 0; j < UNR; ++j) {
      float x[NE];
      word_to_f32<T>(vw[j], x);
#pragma unroll
      for (int g = 0; g < GH; ++g) {
        const int id = j * GH + g;
        const float p = __shfl_sync(0xFFFFFFFFu, lg[id % PER], id / PER * kRep, LPR);
#pragma unroll
        for (int i = 0; i < NE; ++i) acc[g][i] = fmaf(p, x[i], acc[g][i]);
      }
    }
  }
  // ---- the warp's result: lanes that hold the same word of different rows, and the sums of the weights
#pragma unroll
  for (int o = LPR; o < 32; o <<= 1) {
#pragma unroll
    for (int g = 0; g < GH; ++g)
#pragma unroll
      for (int i = 0; i < NE; ++i) acc[g][i] += __shfl_xor_sync(0xFFFFFFFFu, acc[g][i], o);
  }
#pragma unroll
  for (int i = 0; i < PER; ++i) {
#pragma unroll
    for (int o = LPR / UNR; o < 32; o <<= 1) l[i] += __shfl_xor_sync(0xFFFFFFFFu, l[i], o);
    const int id = NV >= LPR ? c * PER + i : c / kRep;
    if (rsub == 0 && id < GH && c % kRep == 0) { w_m[warp][id] = m[i]; w_l[warp][id] = l[i]; }
  }
  if (rsub == 0) {
#pragma unroll
    for (int g = 0; g < GH; ++g)
#pragma unroll
      for (int i = 0; i < NE; i += 4)
        *reinterpret_cast<float4*>(&w_o[warp][g][c * NE + i]) = make_float4(acc[g][i], acc[g][i + 1], acc[g][i + 2], acc[g][i + 3]);
  }
  __syncthreads();
  // ---- the CTA's (a warp without rows left m = -inf, l = 0)
  const auto finish = [&](int g, int x, float o, float l_sum) {
    if (g < n_heads) out[(long long)s * P.o_sb + (long long)(h0 + g) * P.o_sh + x] = from_f32<T>(o / l_sum);
  };
  for (int e = tid; e < GH * D; e += kDecodeAttnThreads) {
    const int g = e / D, x = e % D;
    float M = -INFINITY, L = 0.f, o = 0.f;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) M = fmaxf(M, w_m[i][g]);
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
      const float wgt = w_m[i][g] == -INFINITY ? 0.f : __expf(w_m[i][g] - M);
      L = fmaf(wgt, w_l[i][g], L);
      o = fmaf(wgt, w_o[i][g][x], o);
    }
    if (parts == 1) {
      finish(g, x, o, L);
      if (lse && x == 0 && g < n_heads) lse[(long long)s * P.n_q + h0 + g] = M + logf(L);
    } else {
      part_o[g][x] = o;
      if (x == 0) { part_m[g] = M; part_l[g] = L; }
    }
  }
  if (parts == 1) return;
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();
  for (int e = tid * parts + part; e < GH * D; e += kDecodeAttnThreads * parts) {
    const int g = e / D, x = e % D;
    float pm[8], pl[8], po[8], M = -INFINITY, L = 0.f, o = 0.f;
#pragma unroll
    for (int p = 0; p < 8; ++p) {                    // (independent remote reads, all in flight together)
      pm[p] = p < parts ? *cluster.map_shared_rank(&part_m[g], p) : -INFINITY;
      pl[p] = p < parts ? *cluster.map_shared_rank(&part_l[g], p) : 0.f;
      po[p] = p < parts ? *cluster.map_shared_rank(&part_o[g][x], p) : 0.f;
    }
#pragma unroll
    for (int p = 0; p < 8; ++p) M = fmaxf(M, pm[p]);
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const float wgt = pm[p] == -INFINITY ? 0.f : __expf(pm[p] - M);
      L = fmaf(wgt, pl[p], L);
      o = fmaf(wgt, po[p], o);
    }
    finish(g, x, o, L);
    if (lse && x == 0 && g < n_heads) lse[(long long)s * P.n_q + h0 + g] = M + logf(L);
  }
  cluster.sync();                                    // my part stays mapped until every peer has read it
}

// ---------------------------------------------------------------------------------------------- host
bool decode_path_applies(const DevParams& P) {
  return P.chunk == 1 && P.n_sel == 1;
}

cudaError_t launch_score_keys_gemv(const DevParams& P, int dtype, const void* qbar, const void* k, float* scores,
                                   cudaStream_t st, bool chained) {
  if (P.max_ctx <= 0) return cudaSuccess;
  const dim3 grid((P.max_ctx + kGemvRowsPerCta - 1) / kGemvRowsPerCta, P.n_kv, P.batch), block(kGemvThreads);
  cudaError_t e;
  if (dtype == QUOKA_BF16) {
    if (P.d == 128) e = launch_kernel("score_keys_gemv", score_keys_gemv_kernel<__nv_bfloat16, 128>, grid, block, 0, st, 1, chained, P, (const __nv_bfloat16*)qbar, (const __nv_bfloat16*)k, scores);
    else e = launch_kernel("score_keys_gemv", score_keys_gemv_kernel<__nv_bfloat16, 64>, grid, block, 0, st, 1, chained, P, (const __nv_bfloat16*)qbar, (const __nv_bfloat16*)k, scores);
  } else {
    if (P.d == 128) e = launch_kernel("score_keys_gemv", score_keys_gemv_kernel<float, 128>, grid, block, 0, st, 1, chained, P, (const float*)qbar, (const float*)k, scores);
    else e = launch_kernel("score_keys_gemv", score_keys_gemv_kernel<float, 64>, grid, block, 0, st, 1, chained, P, (const float*)qbar, (const float*)k, scores);
  }
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
