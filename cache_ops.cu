// Appending a chunk's keys and values to the cache (Algorithm 2, "append K_i, V_i to the cache").
//
// The chunk's K_i, V_i arrive dense, [b][n_KV][C][d]; row r of (sequence s, KV head h) goes to cache row
// T_s + r, whose address comes from the strides or, in a paged cache, from the block table.  T_s is read on
// the device, so a loop over chunks needs no host round trip.  One thread moves 16 bytes of K and the same 16
// bytes of V; a warp covers whole rows, so both the reads and the writes are full-width.  HBM-bound:
// 2 * b * n_KV * C * d * es bytes read and as many written; a generation step's single rows are launch latency, so the
// inverse norms are taken in the same pass (a launch of 2.5 us less) and the launch overlaps its neighbours.
#include "common.cuh"

namespace quoka {

template <typename E, int D>
__global__ void __launch_bounds__(256) append_kv_kernel(DevParams P, const uint4* __restrict__ k_new,
                                                         const uint4* __restrict__ v_new, uint4* __restrict__ k_cache,
                                                         uint4* __restrict__ v_cache, float* __restrict__ k_inv_norm) {
  constexpr int ES = (int)sizeof(E);
  grid_dependency_wait();
  grid_launch_dependents();
  constexpr int wpr = D * ES / 16;                                   // 16-byte words per row: 8, 16 or 32
  const int64_t total = (int64_t)P.batch * P.n_kv * P.chunk * wpr;
  const int lane = threadIdx.x & 31;
  for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; e0 < total; e0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = e0 + lane;
    const bool live = e < total;
    const int w = (int)(e % wpr);
    const int64_t row = live ? e / wpr : 0;
    const int r = (int)(row % P.chunk);
    const int h = (int)((row / P.chunk) % P.n_kv);
    const int s = (int)(row / ((int64_t)P.chunk * P.n_kv));
    uint4 kw = make_uint4(0, 0, 0, 0);
    int t = 0;
    if (live) {
      kw = load_input<true>(k_new + e);
      const uint4 vw = load_input<true>(v_new + e);
      t = load_input<true>(P.ctx_len + s) + r;
      const int64_t dst = kv_row_offset<true>(P, s, h, t) * ES / 16 + w;   // strides are multiples of 8 elements
      k_cache[dst] = kw;
      v_cache[dst] = vw;
    }
    if (k_inv_norm != nullptr) {
      // The sum of squares in key_norms_kernel's order, for its bits: D / 32 elements in a row, then the 32 such pieces of the
      // row by a butterfly from the far halves to the neighbours.  A word holds kPieces of them, next to each other.
      constexpr int NE = D / 32, kPieces = 16 / ES / NE;
      const uint32_t v[4] = {kw.x, kw.y, kw.z, kw.w};
      float nn[kPieces];
#pragma unroll
      for (int i = 0; i < kPieces; ++i) {
        nn[i] = 0.f;
#pragma unroll
        for (int j = i * NE; j < (i + 1) * NE; ++j) {
          const uint32_t w32 = v[j * ES / 4];
          const float x = ES == 4 ? __uint_as_float(w32) : __uint_as_float(j % 2 ? w32 & 0xFFFF0000u : w32 << 16);
          nn[i] = fmaf(x, x, nn[i]);
        }
      }
#pragma unroll
      for (int o = wpr / 2; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < kPieces; ++i) nn[i] += __shfl_xor_sync(0xFFFFFFFFu, nn[i], o);
#pragma unroll
      for (int o = kPieces / 2; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) nn[i] += nn[i + o];
      if (live && w == 0) k_inv_norm[kv_norm_index<true>(P, s, h, t)] = 1.f / fmaxf(sqrtf(nn[0]), kNormEps);
    }
  }
}

cudaError_t launch_append_kv(const DevParams& P, int dtype, const void* k_new, const void* v_new, void* k_cache,
                             void* v_cache, float* k_inv_norm, cudaStream_t st) {
  const int es = dtype == QUOKA_BF16 ? 2 : 4;
  const int64_t total = (int64_t)P.batch * P.n_kv * P.chunk * (P.d * es / 16);
  if (total <= 0) return cudaSuccess;
  int64_t blocks = (total + 255) / 256;
  const int64_t most = 16ll * device_sm_count();                     // two waves of eight CTAs per SM; longer appends loop
  if (blocks > most && most > 0) blocks = most;
  const dim3 grid((unsigned)blocks), block(256);
  cudaError_t e;
#define QUOKA_APPEND(E_, D_)                                                                                        \
  e = launch_kernel("append_kv", append_kv_kernel<E_, D_>, grid, block, 0, st, 1, true, P, (const uint4*)k_new,     \
                    (const uint4*)v_new, (uint4*)k_cache, (uint4*)v_cache, k_inv_norm)
  if (es == 2) { if (P.d == 128) QUOKA_APPEND(__nv_bfloat16, 128); else QUOKA_APPEND(__nv_bfloat16, 64); }
  else { if (P.d == 128) QUOKA_APPEND(float, 128); else QUOKA_APPEND(float, 64); }
#undef QUOKA_APPEND
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace quoka
