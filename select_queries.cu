// Query sub-selection, normalisation and GQA pre-aggregation (Algorithm 1, first two blocks).
//
// rank_queries : a thread-block cluster of 2 / 4 / 8 CTAs (slices of 64 to 512 rows, `launch_rank_d`) per
//                (sequence, query head); each CTA owns a contiguous slice of the head's C query rows.
//                Pass 1 brings the slice into shared memory with 16-byte cp.async in eight groups and sums
//                the columns group by group as they land (of a longer slice the first rows; the rest is summed
//                from registers); the CTAs' shares of the mean query are added across the cluster
//                through distributed shared memory in a fixed order.  Pass 2 computes CosSim(q_r, M) for
//                every row of the slice (two lanes per two rows; the rows that were not kept come again from L2,
//                a block of rows at a time) as an order code, and puts the slice in order: up to 256 rows by
//                counting, for every row, the rows before it; more by 32-key runs sorted in registers
//                (bitonic network over shuffles) and merged by branch-free binary searches.  Each CTA
//                then copies the first codes of its peers' sorted slices into local shared memory and
//                places each of its N smallest by global rank: own rank + number of smaller codes in
//                every peer.  The N lowest cosines come out in ascending order, equal cosines by position.
//                Bound by latency (a CTA's slice takes 2 us to arrive, four cluster barriers and the steps between
//                them another 4) and, with two CTAs per SM, by shared memory and instruction issue.  Against every
//                slice sorted in runs, M read once per row and long slices read again a row per lane pair, ranking and
//                aggregation took before / now: 8 heads x 256 rows 12.4 / 10.3 us (f32 13.1 / 10.8), 32 x 512
//                14.4 / 12.7, 32 x 2048 20.5 / 19.1, 256 x 1024 54.2 / 49.4, 32 x 4096 34.9 / 28.9, all with the
//                same slices; `launch_rank_d` has what their length is worth.
// aggregate    : one warp per (sequence, KV head, rank j): mean over the G heads of the group of
//                their j-th retained query, each divided by its own norm; one rounding to dtype.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "qbar.cuh"

namespace cg = cooperative_groups;

namespace quoka {

constexpr int kRankThreads = 512;
constexpr int kRankCluster = 8;
// Shared memory of a CTA, where its sort leaves room for any rows at all: two CTAs must fit an SM (with 128 KB slices,
// chunk 4096, one CTA per SM meant two waves of the grid and a fifth more time).
constexpr size_t kRankSmem = 112 * 1024;
// Slices up to this many rows are ordered by counting: quadratic, but with a handful of dependent steps (runs and
// merge / counting, cycles of a CTA with two on the SM: 256 rows 5300 / 4000; alone on it, 128 rows 2700 / 1300).  512 rows
// would count four times as long, the runs and their merge take 8500.
constexpr int kRankCount = 256;

template <typename T> struct Raw8;                // 8 consecutive elements as 16-byte words
template <> struct Raw8<__nv_bfloat16> { uint4 w[1]; };
template <> struct Raw8<float> { uint4 w[2]; };

template <typename T>
__device__ __forceinline__ void raw_to_f32(const Raw8<T>& r, float (&x)[8]) {
  if constexpr (sizeof(T) == 2) {
    const uint32_t w[4] = {r.w[0].x, r.w[0].y, r.w[0].z, r.w[0].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[2 * j] = __uint_as_float(w[j] << 16);
      x[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
    }
  } else {
    x[0] = __uint_as_float(r.w[0].x); x[1] = __uint_as_float(r.w[0].y);
    x[2] = __uint_as_float(r.w[0].z); x[3] = __uint_as_float(r.w[0].w);
    x[4] = __uint_as_float(r.w[1].x); x[5] = __uint_as_float(r.w[1].y);
    x[6] = __uint_as_float(r.w[1].z); x[7] = __uint_as_float(r.w[1].w);
  }
}

template <typename T, int D, int CL>
__global__ void __launch_bounds__(kRankThreads, 2) rank_queries_kernel(DevParams P, const T* __restrict__ q,
                                                                     int32_t* __restrict__ q_idx, int rpc, int n_sort,
                                                                     int n_stage, int m_peer) {
  // The first kernel of a fused call is launched early as well (its launch runs under the tail of whatever is before it on
  // the stream); nothing is read or written, and no later kernel of the call starts, before that has completed.
  grid_dependency_wait();
  grid_launch_dependents();                 // the aggregation kernel may become resident; it waits for this grid itself
  constexpr int LG = D / 8;                 // lanes per row, 8 elements each
  constexpr int RPI = kRankThreads / LG;    // rows per iteration
  constexpr int NW = sizeof(T) * 8 / 16;    // 16-byte words per lane
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // dynamic shared memory: sort keys | reduction buffer | peer codes | staged rows
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem_raw);               // [n_sort] 32-key sorted runs
  unsigned long long* sorted = keys + n_sort;                                               // [n_sort] the sorted slice
  float* red = reinterpret_cast<float*>(smem_raw + (size_t)n_sort * 16);                    // [RPI][D]
  unsigned long long* peer_keys = reinterpret_cast<unsigned long long*>(red + RPI * D);     // [CL - 1][m_peer]
  uint4* rows = reinterpret_cast<uint4*>(peer_keys + (((size_t)(CL - 1) * m_peer + 1) & ~(size_t)1));   // [n_stage][LG][NW]
  __shared__ float part[D];                 // this CTA's share of the column sums
  __shared__ __align__(16) float M[D + 4];  // the second half 16 bytes on: the halves of a row read different banks

  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int head = blockIdx.x / CL;
  const int s = head / P.n_q, h = head % P.n_q;
  const int C = P.chunk, N = P.n_sel;
  int32_t* out = q_idx + (long long)head * N;
  const int tid = threadIdx.x;

  // (C <= N_Q, where every query is kept, never reaches this kernel: the aggregation kernel writes those ranks)
  const T* qh = q + (long long)s * P.q_sb + (long long)h * P.q_sh;
  const int lane_in_row = tid % LG;
  const int row_slot = tid / LG;
  const int lo = min(C, rank * rpc), hi = min(C, lo + rpc);
  const int n_loc = hi - lo;

  constexpr int WPR = LG * NW;                               // 16-byte words per row
  constexpr int EPW = 16 / (int)sizeof(T);                   // elements per word
  constexpr int HW = WPR / 2;                                // words per half row
  // word c of row r lives in slot c ^ (r & 7): both passes then read shared memory without bank conflicts
  const auto slot = [](int r, int c) { return r * WPR + (c ^ (r & 7)); };
  const uint32_t rows_s = (uint32_t)__cvta_generic_to_shared(rows);
  const auto copy_rows = [&](int first, int r_lo, int r_hi) {     // rows [r_lo, r_hi) of the buffer, which starts at row `first`
    for (int w = r_lo * WPR + tid; w < r_hi * WPR; w += kRankThreads) {
      const int r = w / WPR, c = w % WPR;
      const T* src = qh + (long long)(lo + first + r) * P.q_st + c * EPW;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(rows_s + (uint32_t)slot(r, c) * 16u), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // ---- pass 1: the slice's first n_stage rows go to shared memory with every 16-byte copy in flight at once, committed
  // in 8 groups of rows; the column sums are taken group by group as the copies land, so the arithmetic runs under
  // the HBM transfer
  const int n_kept = min(n_loc, n_stage);
  const int n_iter = (n_kept + RPI - 1) / RPI;               // 32/64-row trips over the kept rows
  const int grp_rows = ((n_iter + 7) / 8) * RPI;             // rows per copy group
#pragma unroll 1
  for (int gi = 0; gi < 8; ++gi) copy_rows(0, min(n_kept, gi * grp_rows), min(n_kept, (gi + 1) * grp_rows));
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
  const auto add_row = [&](const Raw8<T>& raw, bool live) {
    float x[8];
    raw_to_f32<T>(raw, x);
    const float f = live ? 1.f : 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = fmaf(x[i], f, acc[i]);
  };
#pragma unroll
  for (int gi = 0; gi < 8; ++gi) {
    const int g_lo = gi * grp_rows, g_hi = min(n_kept, (gi + 1) * grp_rows);
    if (g_lo >= n_kept) break;
    switch (gi) {                                            // all but the 7 - gi newest groups have landed
      case 0: asm volatile("cp.async.wait_group 7;" ::: "memory"); break;
      case 1: asm volatile("cp.async.wait_group 6;" ::: "memory"); break;
      case 2: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
      case 3: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
      case 4: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
      case 5: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
      case 6: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
      default: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    }
    __syncthreads();
    for (int r0 = g_lo; r0 < g_hi; r0 += RPI) {
      const int r = r0 + row_slot, rc = min(r, n_kept - 1);  // clamped: no branch around the loads
      Raw8<T> raw;
#pragma unroll
      for (int w = 0; w < NW; ++w) raw.w[w] = rows[slot(rc, lane_in_row * NW + w)];
      add_row(raw, r < n_kept);
    }
  }
  // (n_stage is a multiple of RPI where it is less than the slice: the sums are in row order either way)
#pragma unroll 4
  for (int r0 = n_stage; r0 < n_loc; r0 += RPI) {
    const int r = r0 + row_slot, rc = min(r, n_loc - 1);
    const uint4* src = reinterpret_cast<const uint4*>(qh + (long long)(lo + rc) * P.q_st + lane_in_row * 8);
    Raw8<T> raw;
#pragma unroll
    for (int w = 0; w < NW; ++w) raw.w[w] = load_input<true>(src + w);
    add_row(raw, r < n_loc);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) red[row_slot * D + lane_in_row * 8 + i] = acc[i];
  __syncthreads();
  if (tid < D) {
    float sum = 0.f;
    for (int r = 0; r < RPI; ++r) sum += red[r * D + tid];
    part[tid] = sum;
  }
  cluster.sync();
  if (tid < D) {
    float sum = 0.f;
#pragma unroll
    for (int r = 0; r < CL; ++r) sum += cluster.map_shared_rank(part, r)[tid];   // fixed order
    M[tid + (tid >= D / 2 ? 4 : 0)] = sum / (float)C;
  }
  __syncthreads();
  const int lane = tid & 31, wid = tid >> 5;
  float mn = 0.f;                                            // |M|, in every warp
  for (int x = lane; x < D; x += 32) { const float m = M[x + (x >= D / 2 ? 4 : 0)]; mn += m * m; }
  mn = fmaxf(sqrtf(warp_sum(mn)), kNormEps);

  // ---- pass 2: cosine of every row of the slice to M as an order code.  A warp takes 32 rows, lanes l and l + 16 the
  // halves of rows l and l + 16 (the rows' norms and dot products with M in the same sweep, M read from shared memory as a
  // broadcast, which is two thirds of the words read with one row at a time); one shuffle joins the halves.
  const bool count = n_sort <= kRankCount;
  uint32_t* codes = reinterpret_cast<uint32_t*>(keys);       // [n_sort], with the counts [n_sort] behind them
  uint32_t* counts = codes + n_sort;
  const int half = lane >> 4;
  for (int first = 0; first == 0 || first < n_loc; first += n_stage) {
    if (first > 0) {                                         // the next rows, from L2
      __syncthreads();
      copy_rows(first, 0, min(n_loc - first, n_stage));
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
    }
    // (the last block also writes the padding up to n_sort)
    const int end = first + n_stage < n_loc ? first + n_stage : n_sort;
    for (int r0 = first + wid * 32; r0 < end; r0 += kRankThreads) {
      const uint4* row[2];
      int x7[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {                          // clamped (an empty slice reads what is there)
        const int rc = max(min(r0 + 16 * u + (lane & 15) - first, min(n_loc - first, n_stage) - 1), 0);
        row[u] = rows + rc * WPR;
        x7[u] = rc & 7;
      }
      float dot[2] = {0.f, 0.f}, nn[2] = {0.f, 0.f};
#pragma unroll 2
      for (int i = 0; i < HW; ++i) {
        const int c = half * HW + i;
        uint4 wv[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) wv[u] = row[u][c ^ x7[u]];
#pragma unroll
        for (int j = 0; j < EPW; j += 4) {
          const float4 mv = *reinterpret_cast<const float4*>(&M[half * (D / 2 + 4) + i * EPW + j]);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            float x[4];
            if constexpr (sizeof(T) == 2) {
              const uint32_t w0 = j ? wv[u].z : wv[u].x, w1 = j ? wv[u].w : wv[u].y;
              x[0] = __uint_as_float(w0 << 16); x[1] = __uint_as_float(w0 & 0xFFFF0000u);
              x[2] = __uint_as_float(w1 << 16); x[3] = __uint_as_float(w1 & 0xFFFF0000u);
            } else {
              x[0] = __uint_as_float(wv[u].x); x[1] = __uint_as_float(wv[u].y); x[2] = __uint_as_float(wv[u].z); x[3] = __uint_as_float(wv[u].w);
            }
            dot[u] = fmaf(x[0], mv.x, dot[u]); dot[u] = fmaf(x[1], mv.y, dot[u]);
            dot[u] = fmaf(x[2], mv.z, dot[u]); dot[u] = fmaf(x[3], mv.w, dot[u]);
            nn[u] = fmaf(x[0], x[0], nn[u]); nn[u] = fmaf(x[1], x[1], nn[u]);
            nn[u] = fmaf(x[2], x[2], nn[u]); nn[u] = fmaf(x[3], x[3], nn[u]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        dot[u] += __shfl_xor_sync(0xFFFFFFFFu, dot[u], 16);
        nn[u] += __shfl_xor_sync(0xFFFFFFFFu, nn[u], 16);
      }
      // the first half's lanes write the first 16 rows, the second half's the others
      const int r = r0 + lane;
      const float d = half ? dot[1] : dot[0], n = half ? nn[1] : nn[0];
      if (r < end) {
        const uint32_t code = r < n_loc ? float_order_key(d / (fmaxf(sqrtf(n), kNormEps) * mn)) : 0xFFFFFFFFu;
        if (count) { codes[r] = code; counts[r] = 0; }
        else keys[r] = r < n_loc ? ((unsigned long long)code << 32) | (unsigned)(lo + r) : ~0ull;    // padding sorts last
      }
    }
  }
  __syncthreads();

  // ---- sort of the slice, ascending, equal codes by position.
  if (count) {
    // A warp holds 32 rows, one per lane, and counts those of 32 other rows (read as a broadcast) that come before each:
    // two instructions a pair, the borrow of (other - mine) taken off the count.
    const int log_blk = __popc(n_sort - 1) - 5, n_blk = (n_loc + 31) >> 5;
    for (int e = wid; e < 1 << (2 * log_blk); e += kRankThreads / 32) {
      const int mine = e & ((1 << log_blk) - 1), other = e >> log_blk;
      if (max(mine, other) >= n_blk) continue;
      const uint32_t code = codes[mine * 32 + lane];
      const uint4* oc = reinterpret_cast<const uint4*>(codes + other * 32);
      uint32_t n0 = 0, n1 = 0;                               // minus the number of smaller codes
      const auto below = [](uint32_t& n, uint32_t a, uint32_t b) {   // n -= a < b
        uint32_t t;
        asm("sub.cc.u32 %0, %2, %3;\n\tsubc.u32 %1, %1, 0;" : "=r"(t), "+r"(n) : "r"(a), "r"(b));
      };
      if (other < mine) {                                    // rows before mine: n = 32 - those with a larger code
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint4 o = oc[j];
          below(n0, code, o.x); below(n1, code, o.y); below(n0, code, o.z); below(n1, code, o.w);
        }
        n0 = 32u + (n0 + n1);
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint4 o = oc[j];
          below(n0, o.x, code); below(n1, o.y, code); below(n0, o.z, code); below(n1, o.w, code);
        }
        n0 = 0u - (n0 + n1);
        if (other == mine && __reduce_add_sync(0xFFFFFFFFu, n0) != 32 * 31 / 2)      // not all different
          n0 += __popc(__match_any_sync(0xFFFFFFFFu, code) & ((1u << lane) - 1));    // the equal ones before
      }
      atomicAdd(&counts[mine * 32 + lane], n0);
    }
    __syncthreads();
    for (int i = tid; i < n_sort; i += kRankThreads)
      sorted[i < n_loc ? counts[i] : i] = i < n_loc ? ((unsigned long long)codes[i] << 32) | (unsigned)(lo + i) : ~0ull;
  } else {
    // Each warp sorts 32-key runs in registers (no block barriers); then every key finds its place by counting the smaller
    // keys of the other runs with branch-free binary searches (keys are unique) and is scattered to `sorted`.
    const int n_runs = n_sort >> 5;
    for (int run = wid; run < n_runs; run += kRankThreads / 32) {
      unsigned long long v = keys[run * 32 + lane];
#pragma unroll
      for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
          const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, v, j);
          const bool up = (lane & k) == 0, lower = (lane & j) == 0;
          const bool take_min = up == lower;
          v = take_min ? (v < o ? v : o) : (v < o ? o : v);
        }
      }
      keys[run * 32 + lane] = v;
    }
    for (int i = tid; i < n_sort; i += kRankThreads) sorted[i] = ~0ull;   // slots the padding keys do not reach
    __syncthreads();
    for (int i = tid; i < n_sort; i += kRankThreads) {
      const unsigned long long key = keys[i];
      const int my_run = i >> 5;
      int rk = i & 31;
#pragma unroll 1
      for (int run0 = 0; run0 < n_runs; run0 += 8) {        // eight searches side by side: their loads overlap
        int pos[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) pos[u] = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int run = min(run0 + u, n_runs - 1);
            pos[u] += keys[run * 32 + pos[u] + step - 1] < key ? step : 0;
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int run = min(run0 + u, n_runs - 1);
          pos[u] += keys[run * 32 + pos[u]] < key ? 1 : 0;
          rk += (run0 + u < n_runs && run != my_run) ? pos[u] : 0;
        }
      }
      sorted[rk] = key;                                     // padding keys are equal: they may collide, all ~0
    }
  }
  cluster.sync();                                         // every slice is sorted

  // ---- global rank of my N smallest: own rank + number of smaller codes in each peer's slice.  Only a
  // peer's first m_peer codes matter (m_peer = a power of two >= min(n_sort, N): more smaller ones than N
  // already push the rank past N); they are copied into local shared memory first, because a chain of
  // dependent remote reads is slow.
  for (int e = tid; e < (CL - 1) * m_peer; e += kRankThreads) {
    const int pr = e / m_peer, j = e % m_peer;
    const int r = pr + (pr >= rank ? 1 : 0);
    peer_keys[e] = cluster.map_shared_rank(sorted, r)[j];
  }
  cluster.barrier_arrive();                               // done with the peers' shared memory
  __syncthreads();
  const int n_cand = min(N, n_loc);
  for (int li = tid; li < n_cand; li += kRankThreads) {
    const unsigned long long key = sorted[li];
    int rk = li;
    int pos[CL - 1];                            // number of each peer's codes below key; the
#pragma unroll                                            // branch-free searches run side by side
    for (int pr = 0; pr < CL - 1; ++pr) pos[pr] = 0;
    for (int step = m_peer >> 1; step > 0; step >>= 1) {
#pragma unroll
      for (int pr = 0; pr < CL - 1; ++pr)
        pos[pr] += peer_keys[(size_t)pr * m_peer + pos[pr] + step - 1] < key ? step : 0;
    }
#pragma unroll
    for (int pr = 0; pr < CL - 1; ++pr) {
      pos[pr] += peer_keys[(size_t)pr * m_peer + pos[pr]] < key ? 1 : 0;
      rk += pos[pr];
    }
    if (rk < N) out[rk] = (int32_t)(key & 0xFFFFFFFFull);
  }
  cluster.barrier_wait();                                 // my keys stay mapped until every peer is done
}

template <typename T, int D>
__global__ void __launch_bounds__(256) aggregate_queries_kernel(DevParams P, const T* __restrict__ q,
                                                                 int32_t* __restrict__ q_idx,
                                                                 T* __restrict__ qbar) {
  // a chunk no longer than the number of retained queries keeps every query, in position order (Alg. 1's `if`):
  // no ranking kernel runs then, and this kernel writes the identity ranks itself
  const bool identity = P.chunk <= P.n_retain;
  if (!identity) grid_launch_dependents();
  grid_dependency_wait();                   // the ranks come from the kernel before
  if (identity) grid_launch_dependents();   // the call's first kernel: nothing of it starts before the inputs are there
  if (P.attn_counters) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    for (int e = i; e < P.n_attn_counters; e += step) P.attn_counters[e] = 0;
  }
  constexpr int NE = D / 32;
  const int N = P.n_sel;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t total = (int64_t)P.batch * P.n_kv * N;
  if (warp >= total) return;
  const int j = (int)(warp % N);
  const int kv = (int)((warp / N) % P.n_kv);
  const int s = (int)(warp / ((int64_t)N * P.n_kv));
  float acc[NE];
  mean_normalised_query<T, NE>(P, q, s, kv, lane, [&](int g) {
    int32_t* slot = q_idx + ((int64_t)s * P.n_q + kv * P.group + g) * N + j;
    if (!identity) return (int)__ldcg(slot);
    *slot = j;
    return j;
  }, acc);
  store_vec<T, NE>(qbar + warp * D + lane * NE, acc);
}

template <typename T, int D, int CL>
static cudaError_t launch_rank_t(const DevParams& P, const void* q, int32_t* q_idx, cudaStream_t st, bool chained) {
  constexpr int LG = D / 8, RPI = kRankThreads / LG;
  int rpc = (P.chunk + CL - 1) / CL;
  int n_sort = 32;
  while (n_sort < rpc) n_sort <<= 1;
  int m_peer = 1;
  while (m_peer < P.n_sel && m_peer < n_sort) m_peer <<= 1;
  const size_t row_bytes = (size_t)D * sizeof(T);
  const size_t fixed = (size_t)n_sort * 16 + (size_t)RPI * D * 4 + (((size_t)(CL - 1) * m_peer + 1) & ~(size_t)1) * 8;
  // the rows that stay in shared memory: all, or as many whole sweeps of pass 2 (of pass 1) as there is room for
  int n_stage = fixed < kRankSmem ? (int)((kRankSmem - fixed) / row_bytes) : 0;
  if (n_stage >= rpc) n_stage = rpc;
  else if (n_stage >= kRankThreads / 2) n_stage -= n_stage % (kRankThreads / 2);
  else n_stage = std::max(n_stage - n_stage % RPI, RPI);
  const size_t smem = fixed + (size_t)n_stage * row_bytes;
  cudaError_t e = cudaFuncSetAttribute(rank_queries_kernel<T, D, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_kernel("rank_queries", rank_queries_kernel<T, D, CL>, dim3(P.batch * P.n_q * CL), dim3(kRankThreads), smem, st, CL, chained, P,
                       (const T*)q, q_idx, rpc, n_sort, n_stage, m_peer);
}

// A cluster per (sequence, head).  While every CTA has an SM of its own, shorter slices end sooner, down to 64 rows (8 heads x
// 256 rows, f32, 2 / 4 CTAs per head: 10.8 / 9.6 us with the aggregation; 32 x 512 12.8 / 11.6); with two CTAs per SM slices
// of 256 rows (32 x 777, 4 / 8 CTAs: 12.4 / 14.3; 32 x 2048 the same 19); and in grids of several waves the costs of a CTA
// (barriers, order, merge) weigh more than the second read of what a slice of 512 rows cannot keep (256 x 1024, 4 / 2 CTAs:
// 48.7 / 43.0).
template <typename T, int D>
static cudaError_t launch_rank_d(const DevParams& P, const void* q, int32_t* q_idx, cudaStream_t st, bool chained) {
  const long long heads = P.rank_heads, sms = device_sm_count();
  int cl = 2;
  while (cl < kRankCluster) {
    const int rows = (P.chunk + cl - 1) / cl;
    const long long ctas = 2 * heads * cl;                  // after doubling
    if (!(rows > 512 || (rows > 256 && ctas <= 2 * sms) || (rows > 64 && ctas <= sms))) break;
    cl *= 2;
  }
  if (cl == 2) return launch_rank_t<T, D, 2>(P, q, q_idx, st, chained);
  if (cl == 4) return launch_rank_t<T, D, 4>(P, q, q_idx, st, chained);
  return launch_rank_t<T, D, kRankCluster>(P, q, q_idx, st, chained);
}

cudaError_t launch_rank_queries(const DevParams& P, int dtype, const void* q, int32_t* q_idx, cudaStream_t st, bool chained) {
  if (P.chunk <= P.n_retain) return cudaSuccess;      // every query is kept: the aggregation kernel writes the ranks
  cudaError_t e;
  if (dtype == QUOKA_BF16) e = P.d == 128 ? launch_rank_d<__nv_bfloat16, 128>(P, q, q_idx, st, chained) : launch_rank_d<__nv_bfloat16, 64>(P, q, q_idx, st, chained);
  else e = P.d == 128 ? launch_rank_d<float, 128>(P, q, q_idx, st, chained) : launch_rank_d<float, 64>(P, q, q_idx, st, chained);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_aggregate_queries(const DevParams& P, int dtype, const void* q, int32_t* q_idx, void* qbar,
                                     cudaStream_t st, bool chained) {
  const int64_t warps = (int64_t)P.batch * P.n_kv * P.n_sel;
  const dim3 grid((unsigned)((warps * 32 + 255) / 256)), block(256);
  cudaError_t e;
  if (dtype == QUOKA_BF16) {
    if (P.d == 128) e = launch_kernel("aggregate_queries", aggregate_queries_kernel<__nv_bfloat16, 128>, grid, block, 0, st, 1, chained, P, (const __nv_bfloat16*)q, q_idx, (__nv_bfloat16*)qbar);
    else e = launch_kernel("aggregate_queries", aggregate_queries_kernel<__nv_bfloat16, 64>, grid, block, 0, st, 1, chained, P, (const __nv_bfloat16*)q, q_idx, (__nv_bfloat16*)qbar);
  } else {
    if (P.d == 128) e = launch_kernel("aggregate_queries", aggregate_queries_kernel<float, 128>, grid, block, 0, st, 1, chained, P, (const float*)q, q_idx, (float*)qbar);
    else e = launch_kernel("aggregate_queries", aggregate_queries_kernel<float, 64>, grid, block, 0, st, 1, chained, P, (const float*)q, q_idx, (float*)qbar);
  }
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace quoka
