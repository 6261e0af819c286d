// Attention for the f32 dtype over [selected cached rows | the chunk's own causal rows] (Algorithm 2's attention line;
// Eq. 1 / Eq. 2), fp32 FMAs throughout.  Without an index list every cached row is visited (Eq. 2).
//
// What bounds it: the FMA pipes (a tile of 64 queries x 64 keys is 2 * 64 * 64 * D FMAs = 8192 cycles of an SM at D = 128)
// and, on small problems, how many SMs have a tile.  A CTA of 256 threads owns 64 query rows of one head; scores are
// 4 x 4 per thread, the output 4 x D/16 per thread, so that a 16-byte shared-memory read feeds 8 to 11 FMAs.  A problem
// with fewer row blocks than SMs has every row block's keys cut into up to 8 parts, one CTA of a cluster each; the parts
// are added up through distributed shared memory, in part order.
//   8 heads x 256 queries over 512 listed rows + the chunk: 353 -> 37 us (one warp per query row, key by key, before).
// K of the next tile is in flight under this tile's softmax and PV, V of the next one under the next scores: one buffer
// of each.  Half a tile's PV sum is formed in fresh accumulators and added to the running output with compensation:
// thousands of weights below half an ulp of a sum that one key dominates must not vanish one by one.
// Error against 64 bits (relative, 2-norm, 60 problems of 300 to 16000 keys): 2.9e-7; 3.4e-7 with dot products in chains over 32
// elements and the last sums in 32 bits (for 3 % less time), 2.6e-7 in the scalar kernel, whose every sum is compensated.
// Quarters of a tile instead of halves 2.8e-7 and 8 % more time.
#include <cooperative_groups.h>

#include <type_traits>

#include "f32_tiles.cuh"

namespace cg = cooperative_groups;

namespace quoka {

using namespace ptx;

constexpr int kPPitch = kF32Tile + 4;

__device__ __forceinline__ uint64_t neg2(uint64_t a) { return a ^ 0x8000000080000000ull; }      // of a pair of floats
// 1 / x beyond fp32: what all elements of a row are multiplied with should not round them all alike.
__device__ __forceinline__ double inverse(double x) {
  const double r = (double)(1.f / (float)x);
  return isfinite(r) ? r * (2. - x * r) : r;
}

template <int D>
constexpr size_t attn_f32_smem() {
  return ((size_t)2 * kF32Tile * f32_pitch<D>() + (size_t)kF32Tile * D + (size_t)kF32Tile * kPPitch) * sizeof(float);
}

template <int D>
__global__ void __launch_bounds__(kF32Threads, 1)
attn_f32_kernel(DevParams P, const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                const int32_t* __restrict__ k_idx, const int32_t* __restrict__ k_cnt, float* __restrict__ out,
                float* __restrict__ lse, int parts) {
  constexpr int LD = f32_pitch<D>();
  constexpr int W = D / 4;                       // 16-byte words per row
  constexpr int RPI = 32 / W;                    // rows per warp copy instruction
  constexpr int RPW = kF32Tile / (kF32Threads / 32);   // rows of a tile per warp
  constexpr int NC = D / 64;                     // float4 column groups of the output per thread
  extern __shared__ __align__(16) float smf[];
  float* qs = smf;                               // [64][LD]
  float* ks = qs + kF32Tile * LD;                // [64][LD]
  float* vs = ks + kF32Tile * LD;                // [64][D]
  float* ps = vs + kF32Tile * D;                 // [64][kPPitch]
  __shared__ float part_m[kF32Tile], part_l[kF32Tile];
  grid_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = tid & 15, ty = tid >> 4;
  const int part = blockIdx.x % parts, h = blockIdx.x / parts, s = blockIdx.z, kv = h / P.group;
  const int r0 = (int)(gridDim.y - 1 - blockIdx.y) * kF32Tile;       // heaviest first
  const int T = __ldg(P.ctx_len + s), C = P.chunk;
  const int c = lane % W, rsub = lane / W;
  {
    const float* qh = q + (long long)s * P.q_sb + (long long)h * P.q_sh;
#pragma unroll
    for (int i = 0; i < RPW / RPI; ++i) {
      const int r = warp * RPW + i * RPI + rsub;
      cp_async_16(smem_u32(qs + r * LD + 4 * c), qh + (long long)min(r0 + r, C - 1) * P.q_st + 4 * c, r0 + r < C);
    }
    cp_async_commit();
  }
  grid_dependency_wait();                        // the list comes from the kernel before
  const int cnt = k_idx ? __ldcg(k_cnt + s) : T;
  const int32_t* idx = k_idx ? k_idx + ((long long)s * P.n_kv + kv) * P.budget_cap : nullptr;
  const int n_keys = cnt + min(C, r0 + kF32Tile);                    // keys any row of the block sees
  const int n_tiles = (n_keys + kF32Tile - 1) / kF32Tile;
  const int t_lo = (int)((long long)part * n_tiles / parts), t_hi = (int)((long long)(part + 1) * n_tiles / parts);
  // Cache rows of this warp's RPW rows of a tile: lane l < RPW fetches row l's number.
  const auto rows_of = [&](int t) -> int {
    const int u = t * kF32Tile + warp * RPW + (lane & (RPW - 1));
    if (u >= n_keys || t >= t_hi) return -1;
    return u < cnt ? (idx ? __ldcg(idx + u) : u) : T + (u - cnt);
  };
  const auto fetch = [&](const float* src, float* dst, int ld, int rows) {
#pragma unroll
    for (int i = 0; i < RPW / RPI; ++i) {
      const int row = __shfl_sync(0xFFFFFFFFu, rows, i * RPI + rsub);
      cp_async_16(smem_u32(dst + (warp * RPW + i * RPI + rsub) * ld + 4 * c), src + kv_row_offset(P, s, kv, max(row, 0)) + 4 * c, row >= 0);
    }
    cp_async_commit();
  };
  float m[4], l[4], cl[4];                       // cl, co: what the sums have gained too much so far
  uint64_t o[4][2 * NC], co[4][2 * NC];          // in pairs
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = -INFINITY; l[i] = 0.f; cl[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 2 * NC; ++j) { o[i][j] = 0ull; co[i][j] = 0ull; }
  }
  int rows = rows_of(t_lo);
  fetch(k, ks, LD, rows);
  fetch(v, vs, D, rows);
  for (int t = t_lo; t < t_hi; ++t) {
    const int next = rows_of(t + 1);
    cp_async_wait<1>();                          // Q and K have landed, V may still be in flight
    if (t == t_lo) {                             // the softmax scale goes into the queries (every thread its own words): a
#pragma unroll                                   // product may overflow where the logit would not
      for (int i = 0; i < RPW / RPI; ++i) {
        float4* w = reinterpret_cast<float4*>(qs + (warp * RPW + i * RPI + rsub) * LD + 4 * c);
        *w = make_float4(w->x * P.scale, w->y * P.scale, w->z * P.scale, w->w * P.scale);
      }
    }
    __syncthreads();
    float sc[4][4];
    f32_dot_tile<D, 4, 8>(qs, ks, ty, tx, sc);
    __syncthreads();                             // K may be overwritten
    fetch(k, ks, LD, next);
    // ---- softmax of the tile; row 4 ty + i is shared by the 16 lanes of a half warp
    float alpha[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + 4 * ty + i, lim = cnt + r + 1 - t * kF32Tile;      // row r sees columns [0, lim)
      float mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sc[i][j] = tx + 16 * j < lim && r < C ? sc[i][j] : -INFINITY;
        mx = fmaxf(mx, sc[i][j]);
      }
      const float m_new = fmaxf(m[i], half_warp_max(mx));
      alpha[i] = m[i] == -INFINITY ? 0.f : expf(m[i] - m_new);
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = m_new == -INFINITY ? 0.f : expf(sc[i][j] - m_new);
        ps[(4 * ty + i) * kPPitch + tx + 16 * j] = p;
        sum += p;
      }
      l[i] *= alpha[i]; cl[i] *= alpha[i];
      const float y = sum - cl[i], z = l[i] + y;
      cl[i] = (z - l[i]) - y;
      l[i] = z;
      m[i] = m_new;
    }
    cp_async_wait<1>();                          // V has landed, the next K may still be in flight
    __syncthreads();                             // (and P is written: its rows are read by the same half warp only)
    // (in halves of 32 keys, each added to the running output with compensation)
    const int seen = cnt + r0 + 1 - t * kF32Tile;               // columns that every row of the block sees
#pragma unroll 1
    for (int u0 = 0; u0 < kF32Tile; u0 += kF32Tile / 2) {
      uint64_t pv[4][2 * NC];
      const auto sum_half = [&](auto leave_out) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 2 * NC; ++j) pv[i][j] = 0ull;
#pragma unroll 2
        for (int u = u0; u < u0 + kF32Tile / 2; u += 4) {
          float4 p[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4*>(ps + (4 * ty + i) * kPPitch + u);
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            ulonglong2 vv[NC];
#pragma unroll
            for (int g = 0; g < NC; ++g) vv[g] = *reinterpret_cast<const ulonglong2*>(vs + (u + w) * D + 64 * g + 4 * tx);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if constexpr (decltype(leave_out)::value) {
                if (u + w >= seen + 4 * ty + i) continue;       // row r0 + 4 ty + i does not see this key
              }
              const float pw = w == 0 ? p[i].x : (w == 1 ? p[i].y : (w == 2 ? p[i].z : p[i].w));
              const uint64_t p2 = pack2(pw, pw);
#pragma unroll
              for (int g = 0; g < NC; ++g) {
                pv[i][2 * g] = fma2(p2, vv[g].x, pv[i][2 * g]);
                pv[i][2 * g + 1] = fma2(p2, vv[g].y, pv[i][2 * g + 1]);
              }
            }
          }
        }
      };
      sum_half(std::false_type{});
      if (seen < kF32Tile) {
        // Rows of the chunk that some of these query rows do not see.  Their weights are 0, and 0 times a value that is
        // not finite is NaN: then once more without them.
        uint64_t all = 0ull;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 2 * NC; ++j) all = fma2(pv[i][j], 0ull, all);
        float x[2];
        unpack2(all, x[0], x[1]);
        if (!(x[0] + x[1] == 0.f)) sum_half(std::true_type{});
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float f = u0 == 0 ? alpha[i] : 1.f;
        const uint64_t f2 = pack2(f, f);
#pragma unroll
        for (int j = 0; j < 2 * NC; ++j) {
          const uint64_t oo = fma2(o[i][j], f2, 0ull), y = fma2(neg2(co[i][j]), f2, pv[i][j]), z = add2(oo, y);
          co[i][j] = add2(add2(z, neg2(oo)), neg2(y));
          o[i][j] = z;
        }
      }
    }
    __syncthreads();                             // V may be overwritten
    fetch(v, vs, D, next);
  }
  cp_async_wait_all();
  // What is left is in 64 bits: a handful of sums and one product per element, whose roundings would add up to those above.
  double ld[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    ld[i] = (double)l[i] - (double)cl[i];
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) ld[i] += __shfl_xor_sync(0xFFFFFFFFu, ld[i], off);
  }
  float* oh = out + (long long)s * P.o_sb + (long long)h * P.o_sh;
  if (parts == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + 4 * ty + i;
      if (r >= C) continue;
      const double inv = inverse(ld[i]);
#pragma unroll
      for (int g = 0; g < NC; ++g) {
        float x[4], c4[4];
#pragma unroll
        for (int j = 0; j < 2; ++j) { unpack2(o[i][2 * g + j], x[2 * j], x[2 * j + 1]); unpack2(co[i][2 * g + j], c4[2 * j], c4[2 * j + 1]); }
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = (float)(((double)x[j] - (double)c4[j]) * inv);
        *reinterpret_cast<float4*>(oh + (long long)r * P.o_st + 64 * g + 4 * tx) = make_float4(x[0], x[1], x[2], x[3]);
      }
      if (lse && tx == 0) lse[((long long)s * P.n_q + h) * C + r] = m[i] + logf((float)ld[i]);
    }
    return;
  }
  // ---- the parts' results side by side in shared memory (over V); CTA `part` adds up rows part, part + parts, ...
  cg::cluster_group cluster = cg::this_cluster();
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int g = 0; g < NC; ++g)
      *reinterpret_cast<ulonglong2*>(vs + (4 * ty + i) * D + 64 * g + 4 * tx) = make_ulonglong2(o[i][2 * g], o[i][2 * g + 1]);
    if (tx == 0) { part_m[4 * ty + i] = m[i]; part_l[4 * ty + i] = (float)ld[i]; }
  }
  cluster.sync();
  for (int e = tid; e < (kF32Tile / parts + 1) * W; e += kF32Threads) {
    const int lr = (e / W) * parts + part, w = e % W;
    if (lr >= kF32Tile || r0 + lr >= C) continue;
    float pm[8], M = -INFINITY;
    double L = 0., acc[4] = {0., 0., 0., 0.};
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      pm[p] = p < parts ? *cluster.map_shared_rank(part_m + lr, p) : -INFINITY;
      M = fmaxf(M, pm[p]);
    }
#pragma unroll
    for (int p = 0; p < 8; ++p)
      if (p < parts && pm[p] != -INFINITY) {
        const double wgt = (double)expf(pm[p] - M);
        L += wgt * (double)*cluster.map_shared_rank(part_l + lr, p);
        const float4 x = *cluster.map_shared_rank(reinterpret_cast<const float4*>(vs + lr * D + 4 * w), p);
        acc[0] += wgt * (double)x.x; acc[1] += wgt * (double)x.y; acc[2] += wgt * (double)x.z; acc[3] += wgt * (double)x.w;
      }
    const double inv = inverse(L);
    *reinterpret_cast<float4*>(oh + (long long)(r0 + lr) * P.o_st + 4 * w) =
        make_float4((float)(acc[0] * inv), (float)(acc[1] * inv), (float)(acc[2] * inv), (float)(acc[3] * inv));
    if (lse && w == 0) lse[((long long)s * P.n_q + h) * C + r0 + lr] = M + logf((float)L);
  }
  cluster.sync();                                // my part stays mapped until every peer has read it
}

cudaError_t launch_attn_f32(const DevParams& P, const float* q, const float* k, const float* v, const int32_t* k_idx,
                            const int32_t* k_cnt, float* out, float* lse, cudaStream_t st, bool chained) {
  const int rb = (P.chunk + kF32Tile - 1) / kF32Tile;
  const long long jobs = (long long)P.n_q * rb * P.batch, sms = device_sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  // Parts: as many as leave every CTA resident at once, at least two tiles each (a part costs about a tile's time of
  // start-up and merge).
  const int tiles = ((k_idx ? P.budget_cap : P.max_ctx) + (P.chunk + 1) / 2) / kF32Tile;
  int parts = (int)(sms / jobs);
  parts = parts > 8 ? 8 : parts;
  parts = parts > tiles / 2 ? tiles / 2 : parts;
  if (parts < 1 || P.attn_one_part) parts = 1;
  const dim3 grid((unsigned)(P.n_q * parts), (unsigned)rb, (unsigned)P.batch), block(kF32Threads);
  cudaError_t e;
#define QUOKA_ATTN_F32(D_)                                                                                                \
  do {                                                                                                                    \
    e = cudaFuncSetAttribute(attn_f32_kernel<D_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attn_f32_smem<D_>()); \
    if (e != cudaSuccess) return e;                                                                                       \
    e = launch_kernel("attn_f32", attn_f32_kernel<D_>, grid, block, attn_f32_smem<D_>(), st, parts, chained, P, q, k, v,  \
                      k_idx, k_cnt, out, lse, parts);                                                                     \
  } while (0)
  if (P.d == 128) QUOKA_ATTN_F32(128); else QUOKA_ATTN_F32(64);
#undef QUOKA_ATTN_F32
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace quoka
