// Selection of the B largest of a row of scores by a CTA or a cluster of CTAs (Algorithm 1: I = topk(S^, B_SA)), for the
// selection kernel and the fused selection + attention kernel of a generation step.
//
// One histogram over bins linear in the score, the bin of the B-th largest, and that bin's few rows ranked against each other.
// Where that bin is crowded (equal scores, or scores in a narrow band): histograms over the row's order codes, each over the
// bin of the one before, until a bin is a single code.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace quoka {

namespace cg = cooperative_groups;

// Cluster barrier in two halves (release / acquire): what a thread wrote into its peers' shared memory before the
// arrive is there for everyone after the wait.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

constexpr int kRegThreads = 512, kRegWarps = kRegThreads / 32;
constexpr int kLinBits = 13, kLinBins = 1 << kLinBits;
constexpr int kHistWords = kLinBins + 256;
constexpr int kCoarse = 256;              // sums of 32 consecutive bins
constexpr int kCandMax = 512;             // rows of the threshold's bin that are ranked against each other, all CTAs

template <int ITEMS, int CL>
struct SelectSmem {
  static constexpr int kSeg = kCandMax / CL;    // listed rows per CTA
  static_assert(kRegThreads * ITEMS < 65536, "a CTA's sums are kept in 16 bits");
  __align__(16) uint32_t hist_all[kHistWords];  // the histogram, then the list
  __align__(16) uint16_t coarse[kCoarse];       // this CTA's sums, and every CTA's (pushed by the peers)
  __align__(16) uint16_t coarse_in[CL][kCoarse];
  __align__(16) uint32_t sel_bits[kRegWarps * ITEMS];   // of the listed rows, the ones that are taken: bit = lane, word = item
  unsigned long long cand_in[CL][kSeg];         // every CTA's rows of the threshold's bin, (order code, ~position)
  uint32_t list_pos[kSeg];                      // this CTA's
  uint32_t cnt_in[CL][2];                       // every CTA's counts
  uint32_t mm_in[CL][2];                        // every CTA's smallest / largest code
  uint32_t s_bin, s_need, s_cand, s_n;
  int s_cut;
  uint32_t warp_val[32];
  uint32_t warp_off[33];
};

// The row is cut into as many equal pieces as the cluster has warps, 32 * n_it positions each (n_it <= ITEMS, by the row's
// own length, a multiple of GRAN: 8 lets the compiler work on eight items at a time, 1 spreads a short row over every CTA,
// which is what the attention behind the selection wants); lane l of a warp holds positions i*32 + l of its piece.
//
// What bounds it: latency in a cluster, instruction issue where one CTA has a long row (16 warps x 64 x 32 rows).  So
// every row's bin is computed once and kept in a register; a row is then placed by comparing its bin, and only the few
// rows of the threshold's own bin are looked at again.  A row of 32K scores in a cluster of eight CTAs takes 7.0 us as a
// stand-alone launch (one CTA that histogrammed it between its own extremes: 15.0), eight rows of 128K 39.6 -> 10.7, 64
// rows of 64K 41.4 -> 16.1, 128 rows of 32K 14.7 -> 13.7.  The CTAs exchange two sets of pushes (posted stores into the peers'
// shared memory, 16 bytes per lane: four-byte ones took 2000 cycles) and one remote read, with two cluster barriers: 256
// sums of 32 bins each, the 32 bins of the sum in which the B-th largest lies (read by one warp), then every row of
// that one bin.
// Positions per CTA: kRegThreads times a multiple of GRAN.
template <int CL, int GRAN>
__device__ __forceinline__ int select_piece(int T) {
  constexpr int kStep = CL * kRegThreads * GRAN;
  return (T + kStep - 1) / kStep * GRAN * kRegThreads;
}

// Returns this CTA's share of the selection of a row of T scores, B of them (0 < B < T): its number of rows, and how many
// the CTAs before it have.  The rows are left in sm.hist_all, ascending, without a barrier, if they fit there; else they are
// written to `out` (the row's list).  Waits for the kernel before this one ahead of its first look at the scores.
struct Selected { uint32_t before, mine; };
template <int ITEMS, int CL, int GRAN>
__device__ __forceinline__ Selected select_row(const DevParams& P, const float* __restrict__ row, int T, int B, int rank,
                                               SelectSmem<ITEMS, CL>& sm, int32_t* __restrict__ out) {
  constexpr int kSeg = kCandMax / CL;
  typedef unsigned long long key64;             // (order code of the score, ~position): larger = taken earlier
  auto& hist_all = sm.hist_all;
  auto& coarse = sm.coarse;
  auto& coarse_in = sm.coarse_in;
  auto& list_pos = sm.list_pos;
  auto& cand_in = sm.cand_in;
  auto& sel_bits = sm.sel_bits;
  auto& cnt_in = sm.cnt_in;
  auto& mm_in = sm.mm_in;
  auto& warp_val = sm.warp_val;
  auto& warp_off = sm.warp_off;
  uint32_t &s_bin = sm.s_bin, &s_need = sm.s_need, &s_cand = sm.s_cand, &s_n = sm.s_n;
  int& s_cut = sm.s_cut;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int n_it = select_piece<CL, GRAN>(T) / kRegThreads;
  const int base = (rank * kRegThreads + wid * 32) * n_it + lane;       // position of item i: base + 32 i
  for (int i = tid; i < kHistWords / 4; i += kRegThreads) reinterpret_cast<uint4*>(hist_all)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < kRegWarps * ITEMS; i += kRegThreads) sel_bits[i] = 0;
  if (tid == 0) s_n = 0;
  __syncthreads();
  if (CL > 1) cluster_arrive();                 // awaited before the first push: every CTA of the cluster runs by then
  // Everything above needs nothing from the kernel before this one (launched early, it has run under that kernel's
  // tail); the scores do.
  grid_dependency_wait();

  const auto peer = [&](auto* mine, int r) { return CL > 1 ? cluster.map_shared_rank(mine, r) : mine; };
  const auto sync_all = [&]() { if (CL > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads(); };
  const auto warp_scan = [&](uint32_t v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, v, o);
      if (lane >= o) v += u;
    }
    return v;
  };
  // f(position, order code, is it a row) for this thread's rows, read again a few at a time: the loads of a batch overlap.
  // (Kept small: unrolled further, this code costs the fused kernel 6 us that never runs it.)
  const auto each_code = [&](auto&& f) {
    constexpr int kBatch = ITEMS == 64 ? 8 : 4;
#pragma unroll 1
    for (int i = 0; i < n_it; i += kBatch) {
      float v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) v[u] = __ldcg(row + min(base + 32 * (i + u), T - 1));
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        f(base + 32 * (i + u), float_order_key(v[u]), base + 32 * (i + u) < T && (GRAN % kBatch == 0 || i + u < n_it));
    }
  };
  uint32_t cmin = 0u, cmax = 0xFFFFFFFFu;       // smallest and largest code of the row, where they are needed
  const auto row_range = [&]() {
    cmin = 0xFFFFFFFFu; cmax = 0u;
    each_code([&](int, uint32_t c, bool) { cmin = min(cmin, c); cmax = max(cmax, c); });       // (rows read past the end repeat the last)
    cmin = __reduce_min_sync(0xFFFFFFFFu, cmin);
    cmax = __reduce_max_sync(0xFFFFFFFFu, cmax);
    if (lane == 0) { warp_val[wid] = cmin; warp_off[wid] = cmax; }
    __syncthreads();
    cmin = __reduce_min_sync(0xFFFFFFFFu, warp_val[lane % kRegWarps]);
    cmax = __reduce_max_sync(0xFFFFFFFFu, warp_off[lane % kRegWarps]);
    if (CL > 1 && tid < CL) { uint32_t* d = peer(mm_in[rank], tid); d[0] = cmin; d[1] = cmax; }
    sync_all();
    if (CL > 1) {
#pragma unroll
      for (int r = 0; r < CL; ++r) { cmin = min(cmin, mm_in[r][0]); cmax = max(cmax, mm_in[r][1]); }
    }
  };

  // The bin of the histogram, over all CTAs, in which the running count from the top reaches `count`, + 1 (s_bin); what is
  // still needed inside it (s_need); its size (s_cand).
  const auto find_bin = [&](uint32_t count) {
    {
      // sums of 32 bins (two threads each), then to every CTA of the cluster, warp r to CTA r
      static_assert(kRegThreads == 2 * kCoarse && kLinBins == 32 * kCoarse, "16 bins per thread");
      uint32_t c = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {                       // (rotated: the two threads of a sum stay off each other's banks)
        const uint4 h = reinterpret_cast<const uint4*>(hist_all)[4 * tid + ((j + (tid >> 1)) & 3)];
        c += (h.x + h.y) + (h.z + h.w);
      }
      c += __shfl_xor_sync(0xFFFFFFFFu, c, 1);
      const int cb = kCoarse - 1 - (tid >> 1);            // counted from the top
      if ((tid & 1) == 0) (CL > 1 ? coarse : coarse_in[0])[cb] = (uint16_t)c;
      if (CL > 1) {
        __syncthreads();
        if (wid < CL)
          reinterpret_cast<uint4*>(peer(coarse_in[rank], wid))[lane] = reinterpret_cast<const uint4*>(coarse)[lane];
      }
    }
    sync_all();
    if (wid == 0) {
      // the sum, then the bin, in which the running count from the top reaches `count`; lane l owns sums 8l .. 8l + 7
      uint32_t c[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) c[j] = 0;
#pragma unroll
      for (int r = 0; r < CL; ++r) {
        const uint4 a = *reinterpret_cast<const uint4*>(&coarse_in[r][8 * lane]);
        c[0] += a.x & 0xFFFFu; c[1] += a.x >> 16; c[2] += a.y & 0xFFFFu; c[3] += a.y >> 16;
        c[4] += a.z & 0xFFFFu; c[5] += a.z >> 16; c[6] += a.w & 0xFFFFu; c[7] += a.w >> 16;
      }
      uint32_t sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += c[j];
      const uint32_t incl = warp_scan(sum);
      const int src = __ffs(__ballot_sync(0xFFFFFFFFu, incl >= count)) - 1;
      uint32_t cum = incl - sum, at = 0;
      bool hit = false;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (!hit && cum + c[j] >= count) { hit = true; at = j; }
        if (!hit) cum += c[j];
      }
      const int cb = (int)__shfl_sync(0xFFFFFFFFu, 8 * lane + at, src);
      const uint32_t want = count - __shfl_sync(0xFFFFFFFFu, cum, src);
      const int bin0 = kLinBins - 1 - 32 * cb - lane;                    // lane's bin, from the top
      uint32_t f = 0;
#pragma unroll
      for (int r = 0; r < CL; ++r) f += *peer(&hist_all[bin0], r);       // independent remote loads, all in flight together
      const uint32_t fi = warp_scan(f);
      if (lane == __ffs(__ballot_sync(0xFFFFFFFFu, fi >= want)) - 1) {
        s_bin = (uint32_t)bin0 + 1;
        s_need = want - (fi - f);
        s_cand = f;
      }
    }
    __syncthreads();
  };

  // ---- First try: one histogram over bins linear in the score.
  // Cosine scores lie in [-1, 1]; the maximum over many queries is positive for any row worth keeping (512 bins below
  // zero, 7680 above), a single query's and the mean are centred on zero.  Raw dot products take the row's own range.
  float mul_neg = 512.f, mul_pos = 7680.f, add = 512.f;
  if (P.n_sel == 1 || P.agg_mean) mul_neg = mul_pos = add = 4096.f;
  float x[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i % GRAN == 0 && i >= n_it) break;
    x[i] = __ldcg(row + min(base + 32 * i, T - 1));           // clamped load, no branch per item
  }
  if (CL > 1) cluster_wait();
  if (P.score_dot) {
    row_range();
    const float fmin = order_key_to_float(cmin), range = order_key_to_float(cmax) - fmin;
    const bool spread = range > 0.f && range < INFINITY;      // else (one value; infinities or NaN) all rows share a bin
    mul_neg = mul_pos = spread ? (float)kLinBins / range : 0.f;
    add = spread ? -fmin * mul_pos : nanf("");
  }
  int bin[ITEMS];                               // bin + 1, or 0 past the end of the row
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i % GRAN == 0 && i >= n_it) break;
    // Monotone in the order code: a NaN, whose code is above every number's, falls into the last bin (one with the sign
    // bit, below every number's, is read as -infinity).  Adding 2^23 + 1 rounds to an integer in the low mantissa bits (the
    // conversion instruction runs at a quarter of the rate).
    const float v = __uint_as_float(min(__float_as_uint(x[i]), 0xFF800000u));
    const float y = fmaxf(fminf(fmaf(v, v < 0.f ? mul_neg : mul_pos, add), (float)(kLinBins - 1)), 0.f);
    bin[i] = base + 32 * i < T ? (int)(__float_as_uint(y + 8388609.f) & 0x7FFFFFu) : 0;
    if (bin[i] != 0) atomicAdd(&hist_all[bin[i] - 1], 1u);
  }
  __syncthreads();
  find_bin((uint32_t)B);
  uint32_t before_cta = 0, mine_sel = 0;        // selected rows of the CTAs before this one, and of this one
  const int tb = (int)s_bin;
  uint32_t need = s_need;
  bool found = s_cand <= (uint32_t)kCandMax;    // uniform over the cluster
  if (found) {
    // ---- every row of that bin goes to every CTA; (score, position) pairs are unique, so ranking them by counting
    // gives the exact threshold, equal scores by position
    uint32_t gt = 0;
    uint32_t eq[(ITEMS + 31) / 32] = {};        // this thread's rows of the bin, bit = item
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      if (i % GRAN == 0 && i >= n_it) break;
      gt += bin[i] > tb ? 1u : 0u;
      eq[i / 32] |= bin[i] == tb ? 1u << (i & 31) : 0u;
    }
#pragma unroll
    for (int w = 0; w < (ITEMS + 31) / 32; ++w)
      while (eq[w] != 0) {
        const int i = 32 * w + __ffs(eq[w]) - 1;
        eq[w] &= eq[w] - 1;
        const uint32_t slot = atomicAdd(&s_n, 1u);
        if (slot < (uint32_t)kSeg) list_pos[slot] = (uint32_t)(base + 32 * i);
      }
    gt = __reduce_add_sync(0xFFFFFFFFu, gt);
    if (lane == 0) warp_val[wid] = gt;
    __syncthreads();
    const uint32_t n_mine = s_n;
    static_assert(kCandMax <= kRegThreads, "one listed row per thread");
    if ((uint32_t)tid < n_mine && tid < kSeg) {
      const uint32_t pos = list_pos[tid];
      const key64 key = ((key64)float_order_key(__ldcg(row + pos)) << 32) | (uint32_t)~pos;
#pragma unroll
      for (int r = 0; r < CL; ++r) *peer(&cand_in[rank][tid], r) = key;
    }
    if (wid == kRegWarps - 1) {
      const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, lane < kRegWarps ? warp_val[lane] : 0u);
      if (lane < CL) { uint32_t* d = peer(cnt_in[rank], lane); d[0] = total; d[1] = n_mine; }
    }
    sync_all();
#pragma unroll
    for (int r = 0; r < CL; ++r) found = found && cnt_in[r][1] <= (uint32_t)kSeg;     // (uniform over the cluster)
  }
  if (found) {
    // ---- the listed rows side by side (over the histogram, which is done with), each ranked by a thread
    key64* all = reinterpret_cast<key64*>(hist_all);
    int n = 0;
    {
      const int cr = tid / kSeg, cj = tid % kSeg;
      int off = cj, n_r = 0;
#pragma unroll
      for (int r = 0; r < CL; ++r) {
        const int c = (int)cnt_in[r][1];
        if (r < cr) off += c;
        if (r == cr) n_r = c;
        n += c;
      }
      if (cj < n_r) all[off] = cand_in[cr][cj];
      if (tid < 8) all[n + tid] = 0;            // (a key that counts for nobody)
    }
    __syncthreads();
    if (tid < n) {
      const key64 key = all[tid];
      uint32_t above = 0;
      for (int j = 0; j < n; j += 8) {
        ulonglong2 k2[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) k2[u] = reinterpret_cast<const ulonglong2*>(all + j)[u];
#pragma unroll
        for (int u = 0; u < 4; ++u) above += (k2[u].x > key ? 1u : 0u) + (k2[u].y > key ? 1u : 0u);
      }
      if (above < need) {
        const int pos = (int)~(uint32_t)key, owner = pos / (kRegThreads * n_it), at = pos - owner * (kRegThreads * n_it);
        atomicAdd(&cnt_in[owner][0], 1u);
        if (owner == rank) {
          atomicAdd(&warp_val[at / (32 * n_it)], 1u);
          atomicOr(&sel_bits[at / 32], 1u << (at & 31));
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < CL; ++r) before_cta += r < rank ? cnt_in[r][0] : 0u;
    mine_sel = cnt_in[rank][0];
  }
  uint32_t thr = 0;                             // a crowded bin: the code of the B-th largest score, and the last position
  int cut = -1;                                 // that may still be taken among the rows with exactly that code
  if (!found) {
    // ---- A crowded bin: more than 512 rows in 1/7680 (1/4096) of the cosine's range, or more than a CTA's share of those.
    // The scores are read again for every pass: their range, a histogram per 13 bits of it, the counts, the list.  8 rows of
    // 32768 scores, spread / within 1e-3 of each other / all equal: 6.7 / 14 / 10 us, 128 such rows 15 / 42 / 32 (digits of 12
    // bits, every CTA reading all of every CTA's bins: 6.7 / 146 / 148 and 15 / 73 / 82).
    row_range();                                              // (its barrier is behind every peer's look at the histogram)
    uint32_t lo = cmin, hi = cmax;                            // the threshold's code lies in between
    need = (uint32_t)B;
#pragma unroll 1
    while (lo != hi) {
      for (int i = tid; i < kLinBins / 4; i += kRegThreads) reinterpret_cast<uint4*>(hist_all)[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();
      const int shift = max(32 - kLinBits - __clz((int)(hi - lo)), 0);
      each_code([&](int, uint32_t c, bool in) {
        if (in && lo <= c && c <= hi) atomicAdd(&hist_all[(c - lo) >> shift], 1u);
      });
      __syncthreads();
      find_bin(need);
      need = s_need;
      const uint32_t at = (s_bin - 1) << shift;
      hi = lo + min(at + ((1u << shift) - 1), hi - lo);
      lo += at;
      sync_all();                                             // every peer has looked at this histogram
    }
    // Rows above the threshold and equal to it, per warp, per CTA, and before this CTA: by their codes, as the bins were
    // (NaN scores among them are counted once and only once, so that B rows are listed whatever the scores are).
    thr = lo;
    uint32_t w_gt = 0, w_eq = 0;
    each_code([&](int, uint32_t c, bool in) {
      w_gt += in && c > thr ? 1u : 0u;
      w_eq += in && c == thr ? 1u : 0u;
    });
    w_gt = __reduce_add_sync(0xFFFFFFFFu, w_gt);
    w_eq = __reduce_add_sync(0xFFFFFFFFu, w_eq);
    if (lane == 0) warp_val[wid] = w_gt | (w_eq << 16);      // at most 32 * n_it each
    if (tid == 0) s_cut = -1;
    __syncthreads();
    uint32_t eq_before = 0;                                   // rows equal to the threshold in the warps before this one
    {
      const uint32_t v = lane < kRegWarps ? warp_val[lane] : 0u;
      eq_before = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? v >> 16 : 0u);
      const uint32_t g = __reduce_add_sync(0xFFFFFFFFu, v & 0xFFFFu), e = __reduce_add_sync(0xFFFFFFFFu, v >> 16);
      if (tid < CL) { uint32_t* d = peer(cnt_in[rank], tid); d[0] = g; d[1] = e; }
    }
    sync_all();
    uint32_t eq_cta = 0;                                      // and in the CTAs before this one
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      const uint32_t take = min(cnt_in[r][1], need > eq_cta ? need - eq_cta : 0u);
      if (r < rank) { before_cta += cnt_in[r][0] + take; eq_cta += cnt_in[r][1]; }
      if (r == rank) mine_sel = cnt_in[r][0] + take;
    }
    eq_before += eq_cta;
    // this CTA's last position to be taken among the equal rows: all of them, none, or the need-th
    if (eq_cta + cnt_in[rank][1] <= need) {
      cut = 0x7FFFFFFF;
    } else if (eq_cta < need) {
      if (eq_before < need && need <= eq_before + w_eq) {
        uint32_t seen = eq_before;
        each_code([&](int pos, uint32_t c, bool in) {
          const bool eq = in && c == thr;
          const uint32_t bal = __ballot_sync(0xFFFFFFFFu, eq);
          if (eq && seen + (uint32_t)__popc(bal & ((2u << lane) - 1u)) == need) s_cut = pos;
          seen += (uint32_t)__popc(bal);
        });
      }
      __syncthreads();
      cut = s_cut;
    }
    // selected rows per warp
    __syncthreads();
    const uint32_t sel = w_gt + (cut == 0x7FFFFFFF ? w_eq : (eq_before < need ? min(w_eq, need - eq_before) : 0u));
    if (lane == 0) warp_val[wid] = sel;
    __syncthreads();
  }
  // ---- The list, in position order.  One ballot per item; it is collected in shared memory (over the histogram)
  // and copied out with full-width stores.
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t run = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? warp_val[lane] : 0u);
  const bool staged = mine_sel <= (uint32_t)kHistWords;
  const uint32_t room = staged ? (uint32_t)kHistWords : (uint32_t)B - min((uint32_t)B, before_cta);
  uint32_t* dst = staged ? hist_all : reinterpret_cast<uint32_t*>(out) + before_cta;
  const auto put_at = [&](int pos, uint32_t bal) {
    const uint32_t slot = run + (uint32_t)__popc(bal & lt);
    if ((bal >> lane & 1u) && slot < room) dst[slot] = (uint32_t)pos;
    run += (uint32_t)__popc(bal);
  };
  const auto put = [&](int i, uint32_t bal) { put_at(base + 32 * i, bal); };
  if (found) {
#pragma unroll
    for (int i = 0; i < ITEMS; i += 4) {
      if (i % GRAN == 0 && i >= n_it) break;
      if constexpr (GRAN % 4 == 0) {
        const uint4 also = *reinterpret_cast<const uint4*>(&sel_bits[wid * n_it + i]);
        put(i, __ballot_sync(0xFFFFFFFFu, bin[i] > tb) | also.x);
        put(i + 1, __ballot_sync(0xFFFFFFFFu, bin[i + 1] > tb) | also.y);
        put(i + 2, __ballot_sync(0xFFFFFFFFu, bin[i + 2] > tb) | also.z);
        put(i + 3, __ballot_sync(0xFFFFFFFFu, bin[i + 3] > tb) | also.w);
      } else {
#pragma unroll
        for (int j = i; j < i + 4; ++j)
          if (j < n_it) put(j, __ballot_sync(0xFFFFFFFFu, bin[j] > tb) | sel_bits[wid * n_it + j]);
      }
    }
  } else {
    each_code([&](int pos, uint32_t c, bool in) {
      put_at(pos, __ballot_sync(0xFFFFFFFFu, in && (c > thr || (c == thr && pos <= cut))));
    });
  }
  return Selected{before_cta, mine_sel};
}

}  // namespace quoka
