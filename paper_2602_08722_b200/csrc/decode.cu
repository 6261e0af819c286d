// Generation phase (a chunk of ONE query per sequence; Section 4.4, Appendix B): Algorithm 1 skips the query
// sub-selection, Q-bar is one vector per KV head, and the two contraction steps lose their matrix shape:
//   scoring    S^_t = (Qbar . k_t) / |k_t|  is a matrix-vector product that reads every cached key once:
//              HBM-bound, 2 flops per 2 bytes.  score_keys_gemv_kernel streams the keys through a ring per warp.
//   attention  each query head attends B + 1 rows.  decode_attn_kernel gathers them once per KV group, a few rows per
//              warp with an online softmax of its own, the keys cut into parts over a cluster.
// The tensor-core kernels would spend a 128-row MMA tile on one query.  Everything is fp32 arithmetic on the
// stored values; the softmax weights are not rounded to bf16 here.
#include <cooperative_groups.h>

#include "common.cuh"
#include "qbar.cuh"
#include "sm100_ptx.cuh"

namespace cg = cooperative_groups;

namespace quoka {

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

// Position in the list of units: the u-th unit of (sequence s, KV head kv), `left` units before the warp's share ends.
struct UnitWalk {
  int s, kv, u, units_s, left;
  __device__ __forceinline__ void next(const DevParams& P, int unit_rows) {
    --left;
    if (++u < units_s || left <= 0) return;
    u = 0;
    if (++kv < P.n_kv) return;
    kv = 0;
    do { units_s = (__ldg(P.ctx_len + ++s) + unit_rows - 1) / unit_rows; } while (units_s == 0);
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
      const int T_l = s0 + lane < P.batch ? __ldg(P.ctx_len + s0 + lane) : 0;
      total += __reduce_add_sync(0xFFFFFFFFu, (T_l + ROWS - 1) / ROWS * P.n_kv);
    }
    const int n_warps = gridDim.x * (kGemvThreads / 32), id = blockIdx.x + gridDim.x * warp;   // (a short list: all SMs)
    int lo = (int)((long long)total * id / n_warps);
    w.left = (int)((long long)total * (id + 1) / n_warps) - lo;
    if (w.left == 0) return;
    for (int s0 = 0;; s0 += 32) {
      const int T_l = s0 + lane < P.batch ? __ldg(P.ctx_len + s0 + lane) : 0;
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
    return P.page_size != 0 && at.left > 0 ? __ldg(P.block_table + (long long)at.s * P.max_pages + at.u * ROWS / kPage) : 0;
  };
  int page = page_of(in);
  const auto fill = [&](int stage) {
    if (in.left > 0) {
      const int t0 = in.u * ROWS, T_s = __ldg(P.ctx_len + in.s);
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
    if (c % kRep == 0 && t < __ldg(P.ctx_len + s_cur)) scores[((long long)s_cur * P.n_kv + kv_cur) * P.max_ctx + t] = val;
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
// crosses warps.  LPR lanes share a row; the UNR x GH partial products of a lane are summed over those lanes by a
// transposing butterfly that leaves one logit per lane, where its exponential is taken once.
//   One sequence, 8 KV heads of 4, listed rows 256 / 4000 / 16000: 9.7 / 82 / 221 -> 6.8 / 17.5 / 56 us (one CTA per query
//   head, logits in shared memory, K and V one after the other, before); 16 sequences, 256 / 4000 rows: 19.5 / 251 ->
//   11.1 / 93 us; without a list, 32768 rows: 405 -> 134 us (a 128-row tensor-core tile for one query, before).
constexpr int kDecodeUnroll = 4;

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
  grid_launch_dependents();                          // the next call's first kernel, which waits for this grid's end
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
