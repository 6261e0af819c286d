// One row of Q-bar (Algorithm 1, normalisation and mean over the heads of a KV group), for the kernels that need it.
#pragma once

#include "common.cuh"

namespace quoka {

// acc = the NE = head_dim / 32 elements at lane * NE of the mean over the group's heads of q[h][rank of h] / |q[h][rank of h]|,
// in fp32; a warp works on it together.  row_of(g): the chunk row of head g of the group, for lane g % 32 (heads g0 .. g0 + 31
// are asked for together).
template <typename T, int NE, typename RowOf>
__device__ __forceinline__ void mean_normalised_query(const DevParams& P, const T* __restrict__ q, int s, int kv, int lane,
                                                      RowOf&& row_of, float (&acc)[NE]) {
#pragma unroll
  for (int i = 0; i < NE; ++i) acc[i] = 0.f;
  for (int g0 = 0; g0 < P.group; g0 += 32) {
    // the group's ranks in one load, then the rows four at a time so their loads overlap
    const int r_lane = g0 + lane < P.group ? row_of(g0 + lane) : 0;
    const int g_end = min(32, P.group - g0);
    for (int g4 = 0; g4 < g_end; g4 += 4) {
      float x[4][NE];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int g = g4 + u;
        const int r = __shfl_sync(0xFFFFFFFFu, r_lane, g & 31);
        if (g < g_end) {
          const int h = kv * P.group + g0 + g;
          load_vec<T, NE, /*FIRST=*/true>(q + (int64_t)s * P.q_sb + (int64_t)h * P.q_sh + (int64_t)r * P.q_st + lane * NE, x[u]);
        } else {
#pragma unroll
          for (int i = 0; i < NE; ++i) x[u][i] = 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float nn = 0.f;
#pragma unroll
        for (int i = 0; i < NE; ++i) nn += x[u][i] * x[u][i];
        nn = warp_sum(nn);
        const float norm = P.score_dot ? 1.f : fmaxf(sqrtf(nn), kNormEps);
        if (g4 + u < g_end) {
#pragma unroll
          for (int i = 0; i < NE; ++i) acc[i] += x[u][i] / norm;
        }
      }
    }
  }
  const float inv_g = 1.f / (float)P.group;
#pragma unroll
  for (int i = 0; i < NE; ++i) acc[i] *= inv_g;
}

}  // namespace quoka
