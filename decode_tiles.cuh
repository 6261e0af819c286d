// Attention of one query per sequence over a handful of rows, shared by the generation-step kernels.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace quoka {

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

constexpr int kDecodeUnroll = 4;

// f32: the library's exp and compensated sums, as in the f32 attention of longer chunks (attn_f32.cu): a lane adds up thousands
// of weights, and those below half an ulp of its sum must not vanish one by one.  bf16: the outputs are rounded to 8 bits.
template <typename T>
__device__ __forceinline__ float decode_exp(float x) {
  if constexpr (sizeof(T) == 4) return expf(x); else return __expf(x);
}
// s += x; c: what the sum has lost so far, added once at the end (and left out where the sum has become infinite)
__device__ __forceinline__ void add_compensated(float& s, float& c, float x) {
  const float z = s + x;
  c += (s - z) + x;
  s = z;
}
__device__ __forceinline__ float compensated(float s, float c) { return c == c ? s + c : s; }

// What the warps of a CTA leave for its sum, and what a CTA leaves for its cluster's: per head the reference point, the
// sum of the weights and the un-normalised output.
template <int D, int GH, int WARPS>
struct DecodeWarps { float m[WARPS][GH], l[WARPS][GH]; __align__(16) float o[WARPS][GH][D]; };
template <int D, int GH>
struct DecodePart { float m[GH], l[GH]; __align__(16) float o[GH][D]; };

// This lane's words of GH queries, times the softmax scale; a head past the group's end repeats the last one, unused.
template <typename T, int D, int GH>
__device__ __forceinline__ void decode_load_q(const DevParams& P, const T* __restrict__ q, int s, int h0, int n_heads, int c,
                                              float (&qv)[GH][VecOf<T>::N]) {
#pragma unroll
  for (int g = 0; g < GH; ++g) {
    const int h = h0 + min(g, n_heads - 1);
    const uint4 w = __ldg(reinterpret_cast<const uint4*>(q + (long long)s * P.q_sb + (long long)h * P.q_sh) + c);
    word_to_f32<T>(w, qv[g]);
#pragma unroll
    for (int i = 0; i < VecOf<T>::N; ++i) qv[g][i] *= P.scale;
  }
}

// GH heads of (sequence s, KV head kv) over the cache rows row_of(u), u_lo <= u < u_hi.  A warp fetches its rows' numbers,
// then K AND V of the rows together; LPR lanes share a row; the UNR x GH partial products of a lane are summed over those
// lanes by a transposing butterfly that leaves one logit per lane, where its exponential is taken once; each warp keeps its
// own running maximum.  Leaves the CTA's result in `part` (m = -inf, l = 0 without rows), without a barrier behind it;
// row_of is not used after the first barrier (so that `w` may lie over what it reads).
template <typename T, int D, int GH, int WARPS, typename RowOf>
__device__ __forceinline__ void decode_attend(const DevParams& P, const T* __restrict__ k, const T* __restrict__ v, int s, int kv,
                                              const float (&qv)[GH][VecOf<T>::N], int u_lo, int u_hi, RowOf&& row_of,
                                              DecodeWarps<D, GH, WARPS>& w, DecodePart<D, GH>& part) {
  constexpr int NE = VecOf<T>::N;
  constexpr int LPR = D / NE;                        // lanes per row
  constexpr int RPW = 32 / LPR;                      // rows per warp instruction
  constexpr int UNR = kDecodeUnroll;
  constexpr int kRows = RPW * UNR;                   // rows per warp and trip
  constexpr int kWarps = WARPS;
  constexpr int NV = UNR * GH;
  constexpr int PER = NV >= LPR ? NV / LPR : 1;      // logits a lane holds after the transposing sum
  constexpr int kRep = NV < LPR ? LPR / NV : 1;      // lanes that hold the same one
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = lane % LPR, rsub = lane / LPR;
  constexpr bool kComp = sizeof(T) == 4;
  float m[PER], l[PER], acc[GH][NE];                 // m, l: of the head this lane's logits belong to
  float cl[kComp ? PER : 1], cacc[kComp ? GH : 1][NE];
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    m[i] = -INFINITY; l[i] = 0.f;
    if constexpr (kComp) cl[i] = 0.f;
  }
#pragma unroll
  for (int g = 0; g < GH; ++g)
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      acc[g][i] = 0.f;
      if constexpr (kComp) cacc[g][i] = 0.f;
    }
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
      const float ref = mx == -INFINITY ? 0.f : mx;  // (logits of -infinity alone: weights of 0)
      alpha[i] = decode_exp<T>(m[i] - ref);          // (0 on the first trip: m is -inf, ref is not)
      m[i] = mx;
      lg[i] = decode_exp<T>(x - ref);
      if constexpr (kComp) {
        l[i] *= alpha[i]; cl[i] *= alpha[i];
        add_compensated(l[i], cl[i], lg[i]);
      } else {
        l[i] = fmaf(l[i], alpha[i], lg[i]);
      }
    }
    if (u0 >= u_lo + kWarps * kRows) {               // not the warp's first trip
#pragma unroll
      for (int g = 0; g < GH; ++g) {
        const float a = __shfl_sync(0xFFFFFFFFu, alpha[g % PER], g / PER * kRep, LPR);
#pragma unroll
        for (int i = 0; i < NE; ++i) {
          acc[g][i] *= a;
          if constexpr (kComp) cacc[g][i] *= a;
        }
      }
    }
    if constexpr (kComp) {
#pragma unroll
      for (int g = 0; g < GH; ++g) {                 // the trip's rows first, then to the running sum
        float pv[NE];
#pragma unroll
        for (int j = 0; j < UNR; ++j) {
          const int id = j * GH + g;
          const float p = __shfl_sync(0xFFFFFFFFu, lg[id % PER], id / PER * kRep, LPR);
          float x[NE];
          word_to_f32<T>(vw[j], x);
#pragma unroll
          for (int i = 0; i < NE; ++i) pv[i] = j == 0 ? p * x[i] : fmaf(p, x[i], pv[i]);
        }
#pragma unroll
        for (int i = 0; i < NE; ++i) add_compensated(acc[g][i], cacc[g][i], pv[i]);
      }
    } else {
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
  }
  if constexpr (kComp) {
#pragma unroll
    for (int i = 0; i < PER; ++i) l[i] = compensated(l[i], cl[i]);
#pragma unroll
    for (int g = 0; g < GH; ++g)
#pragma unroll
      for (int i = 0; i < NE; ++i) acc[g][i] = compensated(acc[g][i], cacc[g][i]);
  }
  __syncthreads();
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
    if (rsub == 0 && id < GH && c % kRep == 0) { w.m[warp][id] = m[i]; w.l[warp][id] = l[i]; }
  }
  if (rsub == 0) {
#pragma unroll
    for (int g = 0; g < GH; ++g)
#pragma unroll
      for (int i = 0; i < NE; i += 4)
        *reinterpret_cast<float4*>(&w.o[warp][g][c * NE + i]) = make_float4(acc[g][i], acc[g][i + 1], acc[g][i + 2], acc[g][i + 3]);
  }
  __syncthreads();
  for (int e = tid; e < GH * D; e += kWarps * 32) {
    const int g = e / D, x = e % D;
    float M = -INFINITY, L = 0.f, o = 0.f;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) M = fmaxf(M, w.m[i][g]);
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
      const float wgt = w.m[i][g] == -INFINITY ? 0.f : decode_exp<T>(w.m[i][g] - M);
      L = fmaf(wgt, w.l[i][g], L);
      o = fmaf(wgt, w.o[i][g][x], o);
    }
    part.o[g][x] = o;
    if (x == 0) { part.m[g] = M; part.l[g] = L; }
  }
}

// Adds up the parts of a cluster (or the one part of a CTA), in rank order, and stores the outputs of heads h0 ..
template <typename T, int D, int GH, int WARPS>
__device__ __forceinline__ void decode_merge(const DevParams& P, DecodePart<D, GH>& part, int rank, int parts, int s, int h0,
                                             int n_heads, T* __restrict__ out, float* __restrict__ lse) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  if (parts > 1) cluster.sync(); else __syncthreads();
  for (int e = threadIdx.x * parts + rank; e < GH * D; e += WARPS * 32 * parts) {
    const int g = e / D, x = e % D;
    float pm[8], pl[8], po[8], M = -INFINITY, L = 0.f, o = 0.f;
#pragma unroll
    for (int p = 0; p < 8; ++p) {                    // (independent remote reads, all in flight together)
      pm[p] = p < parts ? *cluster.map_shared_rank(&part.m[g], p) : -INFINITY;
      pl[p] = p < parts ? *cluster.map_shared_rank(&part.l[g], p) : 0.f;
      po[p] = p < parts ? *cluster.map_shared_rank(&part.o[g][x], p) : 0.f;
    }
#pragma unroll
    for (int p = 0; p < 8; ++p) M = fmaxf(M, pm[p]);
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const float wgt = pm[p] == -INFINITY ? 0.f : decode_exp<T>(pm[p] - M);
      L = fmaf(wgt, pl[p], L);
      o = fmaf(wgt, po[p], o);
    }
    if (g < n_heads) out[(long long)s * P.o_sb + (long long)(h0 + g) * P.o_sh + x] = from_f32<T>(o / L);
    if (lse && x == 0 && g < n_heads) lse[(long long)s * P.n_q + h0 + g] = M + logf(L);
  }
  if (parts > 1) cluster.sync();                     // my part stays mapped until every peer has read it
}

}  // namespace quoka
