// Register-tiled fp32 products for the f32 kernels: 256 threads = 16 x 16, thread (ty, tx) owns rows 4 ty .. 4 ty + 3 and
// columns tx, tx + 16, ... of a 64-row tile.  Rows are padded by 16 bytes, so that 16 lanes reading the same 16-byte
// piece of 16 consecutive rows touch every bank once per phase.
#pragma once

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace quoka {

constexpr int kF32Threads = 256;
constexpr int kF32Tile = 64;

template <int D> __host__ __device__ constexpr int f32_pitch() { return D + 4; }      // floats

// acc[i][j] = A[4 ty + i] . B[tx + 16 j] over D elements; fp32 FMAs, even and odd elements in the halves of a pair
// (16 J FMAs for 4 + J shared-memory reads of 16 bytes).  Summed in chains over BLOCK elements, those in blocks of 32: chains
// of 64 FMAs doubled the rounding error of the attention output, chains over 32 elements leave a tenth more than over 8.
template <int D, int J, int BLOCK>
__device__ __forceinline__ void f32_dot_tile(const float* __restrict__ A, const float* __restrict__ B, int ty, int tx,
                                             float (&acc)[4][J]) {
  constexpr int LD = f32_pitch<D>();
  uint64_t a2[4][J];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < J; ++j) a2[i][j] = 0ull;
  const float* ap = A + 4 * ty * LD;
  const float* bp = B + tx * LD;
#pragma unroll 1
  for (int c0 = 0; c0 < D; c0 += 32) {
    uint64_t u2[4][J];
#pragma unroll
    for (int c1 = 0; c1 < 32; c1 += BLOCK) {
      uint64_t t2[4][J];
#pragma unroll
      for (int c = c0 + c1; c < c0 + c1 + BLOCK; c += 4) {
        ulonglong2 a[4], b[J];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(ap + i * LD + c);
#pragma unroll
        for (int j = 0; j < J; ++j) b[j] = *reinterpret_cast<const ulonglong2*>(bp + 16 * j * LD + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < J; ++j)
            t2[i][j] = ptx::fma2(a[i].y, b[j].y, ptx::fma2(a[i].x, b[j].x, c == c0 + c1 ? 0ull : t2[i][j]));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < J; ++j) u2[i][j] = c1 == 0 ? t2[i][j] : ptx::add2(u2[i][j], t2[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < J; ++j) a2[i][j] = ptx::add2(a2[i][j], u2[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < J; ++j) {
      float lo, hi;
      ptx::unpack2(a2[i][j], lo, hi);
      acc[i][j] = lo + hi;
    }
}

// Sum / maximum over the 16 lanes that share a row.
__device__ __forceinline__ float half_warp_sum(float x) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}
__device__ __forceinline__ float half_warp_max(float x) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xFFFFFFFFu, x, o));
  return x;
}

}  // namespace quoka
