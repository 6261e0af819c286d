// Pieces shared by the tensor-core attention kernels: tile geometry of a CTA's walk over the key tiles,
// the rows a tile holds, the causal limit, and small softmax helpers.
#pragma once

#include "sm100_ptx.cuh"
#include "tensor_kernels.cuh"

namespace quoka {

using namespace ptx;

constexpr int kAttnThreads = 12 * 32;
constexpr int kLoaderWarps = 2;
constexpr int kPvWarp = 10, kQkWarp = 11;
constexpr int kQTile = 128;
constexpr int kKeyTile = 128;
// The reference point m of the exponentials 2^(s - m) is raised, and O and l rescaled, only when a row's maximum
// exceeds it by more than this many powers of two.  Until then P, l and O are simply larger by a common factor of at
// most 2^32, which floating point carries without loss (bf16 and fp32 both reach 2^127; l <= 2^32 * keys and
// |O| <= l * max|v| stay far below that); the quotient O / l does not change.  With 8 the rescale (a read-modify-
// write of the whole accumulator row on the softmax -> PV chain) still ran often enough to cost 1-2 % of the kernel.
constexpr float kRescaleThreshold = 32.0f;   // log2 units

// Any of the tensor-core attention kernels.
typedef void (*AttnKernel)(DevParams, const CUtensorMap, const CUtensorMap, const CUtensorMap, const __nv_bfloat16*,
                           const __nv_bfloat16*, const int32_t*, const int32_t*, __nv_bfloat16*, float*);
quoka_status launch_attn_plan(const quoka_params* p, const DevParams& P, const AttnPlan& plan, AttnKernel (*pick)(bool, bool, bool),
                              const char* name, int cluster, size_t smem, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
                              const CUtensorMap& tm_v, const void* k, const void* v, const int32_t* k_idx, const int32_t* k_cnt,
                              void* out, float* lse, cudaStream_t st, bool after_selection);

bool encode_kv_tensor_map(CUtensorMap* out, const quoka_params* p, const void* cache, uint32_t box_rows);

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The z-th sequence of a launch, longest cache first (equal lengths in order), so that the last CTAs to start are short
// ones (8 sequences of 8K to 64K, 7 waves: sparse attention 663 -> 644 us); every warp works it out for itself.  Batches
// beyond a warp's lanes keep their order.
__device__ __forceinline__ int longest_first(const DevParams& P, int z) {
  if (P.batch == 1 || P.batch > 32) return z;
  const int lane = threadIdx.x & 31;
  const int T = lane < P.batch ? __ldg(P.ctx_len + lane) : -1;
  int before = 0;
  for (int j = 0; j < P.batch; ++j) {
    const int o = __shfl_sync(0xFFFFFFFFu, T, j);
    before += o > T || (o == T && j < lane) ? 1 : 0;
  }
  return __ffs(__ballot_sync(0xFFFFFFFFu, lane < P.batch && before == z)) - 1;
}

// The query rows of a Q tile: `pack` heads of one KV group at `span` consecutive chunk positions, position by position, so
// that the heads of a group share every key tile and a tile's rows end at nearly the same causal limit; 128 / pack positions
// each, the rows that are left over (two for three heads, three for five, eight for ten) are zero.  `attn_plan` says how many
// heads, as a rule all of a KV group.  Against 128 positions of one head each: a chunk of 777 with eight heads per KV head
// takes 49 tiles instead of 56, one of 68 with three heads 2 instead of 3, the chunk's own tiles that a row block walks end
// 32 positions after its first row and not 256 (four heads).
// A row block is the Q tiles of one CTA (A, or A and B), or of both CTAs of a pair: A of the first, A of the second, then the
// two Bs, so that a row block of no more positions than two tiles have walks one tile in each CTA.
struct QRows {
  int head0;            // first head
  int p0;               // first chunk position of this CTA
  int step;             // from its tile A to its tile B
  // of the CTA `rank` of `ctas` of row block rb
  __device__ __forceinline__ QRows(const DevParams& P, int hg, int rb, int rank, int ctas)
      : head0(hg * P.attn_pack), p0((rb * P.attn_qtiles * ctas + rank) * P.attn_span), step(ctas * P.attn_span) {}
  __device__ __forceinline__ static int groups(const DevParams& P) { return P.n_q / P.attn_pack; }
  __device__ __forceinline__ int position(const DevParams& P, int x, int row_in_tile) const {
    return p0 + x * step + row_in_tile / P.attn_pack;
  }
  __device__ __forceinline__ int head(const DevParams& P, int row_in_tile) const { return head0 + row_in_tile % P.attn_pack; }
  // rows of tile x that exist: the first ones
  __device__ __forceinline__ int count(const DevParams& P, int x) const {
    return x < P.attn_qtiles ? P.attn_pack * max(0, min(P.attn_span, P.chunk - p0 - x * step)) : 0;
  }
};

// This CTA's Q tiles by the copy engine: boxes of [span][pack][64 elements].
template <int D>
__device__ __forceinline__ void load_q_tiles(const DevParams& P, const QRows& qr, unsigned char* q_smem, const CUtensorMap* tm_q,
                                             uint64_t* q_full, int s) {
  mbar_arrive_expect_tx(q_full, P.attn_qtiles * (D / 64) * 128 * P.attn_pack * P.attn_span);
  for (int x = 0; x < P.attn_qtiles; ++x)
    for (int hh = 0; hh < D / 64; ++hh)
      tma_load_5d(q_smem + (x * (D / 64) + hh) * 16384, tm_q, q_full, hh * 64, 0, qr.p0 + x * qr.step, qr.head0 / P.attn_pack, s);
}
// The rows left over: by the calling threads, before the barrier that the issuing warps pass.
template <int D>
__device__ __forceinline__ void zero_spare_q_rows(const DevParams& P, unsigned char* q_smem, int thread, int threads) {
  const int used = P.attn_pack * P.attn_span, spare = (128 - used) * 8;      // 16-byte pieces of a half tile
  if (spare == 0) return;
  for (int i = thread; i < P.attn_qtiles * (D / 64) * spare; i += threads)
    reinterpret_cast<uint4*>(q_smem + (i / spare) * 16384 + used * 128)[i % spare] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
}
bool encode_q_tensor_map(CUtensorMap* out, const DevParams& P, const void* q);

// Every CTA walks ONE sequence of key tiles t = 0 .. n_total-1 for both of its Q tiles (a pair, for all four); Q tile B takes
// part in all of them, A in the tiles t >= skip_a (a suffix, so both finish on the same tile).
//   dense : the tiles of rows [0, T + C) in DESCENDING order.
//   sparse: first the chunk's own tiles, those that not all rows of the block see descending and then the others ascending,
//           THEN the tiles of the selected list.  The chunk's tiles do not depend on the key selection, so this kernel is
//           launched with programmatic stream serialisation: it starts while the selection kernel still runs, works through
//           the chunk tiles, and only then waits for the selection (`resolve`) to learn the list length.
// So the tiles that a row does not see come before the first one that it does: whatever they add to O (their weights are
// zero, but a value may be infinite) is wiped when the row's reference point is first set.
struct AttnGeom {
  int T, C;
  int n_chunk;        // sparse: tiles of the chunk's own rows in the sequence; dense: 0
  int lead;           // sparse: as many of them are not seen by all rows
  int skip_a;         // first tile Q tile A takes part in (B takes part in all); scalars, not arrays: the struct
  bool active_b;      // must live in registers (an indexed member would put it in local memory)
  int n_known;        // tiles known so far (sparse: n_chunk until resolved, then n_chunk + n_sel)
  int cnt;            // sparse: selected rows (valid once resolved)
  int n_dense;        // dense: number of tiles
  bool resolved;
};

// The row block of `ctas` CTAs that begins at chunk position p.
template <bool SPARSE>
__device__ __forceinline__ AttnGeom make_geom(const DevParams& P, int s, int p, int ctas) {
  AttnGeom g;
  g.T = __ldg(P.ctx_len + s);
  g.C = P.chunk;
  const int span = ctas * P.attn_span;
  g.active_b = P.attn_qtiles == 2 && p + span < g.C;
  // last positions of any tile and of any A tile
  const int last = min(p + P.attn_qtiles * span, g.C) - 1, last_a = min(p + span, g.C) - 1;
  g.cnt = 0;
  if (SPARSE) {
    g.n_chunk = last / kKeyTile + 1;
    g.lead = g.n_chunk - (p / kKeyTile + 1);
    g.skip_a = g.active_b ? g.n_chunk - (last_a / kKeyTile + 1) : 0;       // 0 or 1, for a pair up to 2: a Q tile spans at most 128 positions
    g.n_known = g.n_chunk;
    g.n_dense = 0;
    g.resolved = false;
  } else {
    g.n_dense = (g.T + last) / kKeyTile + 1;
    g.skip_a = g.active_b ? g.n_dense - ((g.T + last_a) / kKeyTile + 1) : 0;
    g.n_chunk = 0; g.lead = 0;
    g.n_known = g.n_dense;
    g.resolved = true;
  }
  return g;
}

// Sparse: wait for the selection kernel (a no-op when this kernel was not launched early) and read the list length.
__device__ __forceinline__ void resolve(AttnGeom& g, const int32_t* k_cnt, int s) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  g.cnt = __ldcg(k_cnt + s);
  g.n_known = g.n_chunk + (g.cnt + kKeyTile - 1) / kKeyTile;
  g.resolved = true;
}

// For the warps that issue the products: their loops' bounds in a form the compiler knows to be the same in every lane.
__device__ __forceinline__ void uniform_geom(AttnGeom& g) {
  g.skip_a = warp_uniform(g.skip_a);
  g.active_b = warp_all(g.active_b);
  g.n_known = warp_uniform(g.n_known);
  g.resolved = warp_all(g.resolved);
}

// The same where the selection is known to be complete.
__device__ __forceinline__ void learn_count(AttnGeom& g, const int32_t* k_cnt, int s) {
  g.cnt = __ldcg(k_cnt + s);
  g.n_known = g.n_chunk + (g.cnt + kKeyTile - 1) / kKeyTile;
  g.resolved = true;
}
__device__ __forceinline__ bool attn_last_cta() {
  return blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1;
}

// Rows of tile t: from the selected list (`from_list`, rows list[base .. base + count)), or the consecutive cache
// rows first .. first + count - 1.  `diag` = chunk position of the tile's first row minus one tile-relative
// offset, used by the causal limit: row r sees columns [0, r - col0 + 1).
struct TileRows {
  bool from_list;       // addressing: rows list[first .. first + count), else the consecutive cache rows first ..
  bool causal;          // masking: row r sees columns [0, r - col0 + 1), else columns [0, count)
  int first, count;     // consecutive rows (count may exceed the tile or be <= 0), or list base and remaining count
  int col0;             // causal tiles: chunk position (dense: position in [0, T + C)) of column 0
};

template <bool SPARSE>
__device__ __forceinline__ TileRows tile_rows(const AttnGeom& g, int t) {
  TileRows r;
  if (SPARSE) {
    if (t < g.n_chunk) {
      const int ct = t < g.lead ? g.n_chunk - 1 - t : t - g.lead;
      r.from_list = false;
      r.causal = true;
      r.first = g.T + ct * kKeyTile;
      r.count = g.C - ct * kKeyTile;
      r.col0 = ct * kKeyTile;
    } else {
      // a list as long as the cache is the identity (the budget covers the cache): its tiles are plain row ranges
      const int st = t - g.n_chunk;
      r.from_list = g.cnt != g.T;
      r.causal = false;
      r.first = st * kKeyTile;
      r.count = g.cnt - st * kKeyTile;
      r.col0 = 0;
    }
  } else {
    const int j = g.n_dense - 1 - t;
    r.from_list = false;
    r.causal = true;
    r.first = j * kKeyTile;
    r.count = g.T + g.C - j * kKeyTile;
    r.col0 = j * kKeyTile - g.T;            // chunk position of column 0 (negative inside the cache)
  }
  return r;
}

// Offset of cache row t of a (sequence, head) in 16-byte units, kNoRow for t < 0 (`listed`: an entry of the selected list).
constexpr uint32_t kNoRow = 0xFFFFFFFFu;
__device__ __forceinline__ uint32_t kv_row_off16(const DevParams& P, const int32_t* table, uint32_t st16, uint32_t sb16, int t,
                                                 bool listed, int T) {
#ifdef QUOKA_DEBUG
  // debug build: a listed row outside [0, T) is recorded and treated as absent (zero-filled) instead of read
  if (listed && (t < -1 || t >= T)) { atomicExch(P.status, (int32_t)QUOKA_ERR_BAD_INDEX); t = -1; }
#endif
  const int tc = max(t, 0);
  uint32_t off = (uint32_t)tc * st16;
  if (P.page_size != 0) {
    int page = __ldg(table + (tc >> 6));
#ifdef QUOKA_DEBUG
    // debug build: a page id outside the pool is recorded and the row treated as absent
    if (page < 0 || (long long)page >= P.kv_rows) {
      if (t >= 0) atomicExch(P.status, (int32_t)QUOKA_ERR_BAD_INDEX);
      t = -1;
      page = 0;
    }
#endif
    off = (uint32_t)page * sb16 + (uint32_t)(tc & (kPage - 1)) * st16;
  }
  return t < 0 ? kNoRow : off;
}

// Number of visible columns of tile t for chunk row `row` (columns [0, lim) are visible; may lie outside [0, 128]).
// A softmax thread keeps it up from tile to tile.
template <bool SPARSE>
struct VisibleCols {
  int lim, step;
  __device__ __forceinline__ VisibleCols(const AttnGeom& g, int t, int row) {
    const TileRows tr = tile_rows<SPARSE>(g, t);
    lim = tr.causal ? row - tr.col0 + 1 : tr.count;
    step = !SPARSE || t < g.lead ? kKeyTile : -kKeyTile;
  }
  __device__ __forceinline__ void at(const AttnGeom& g, int t, int row) {
    if (SPARSE && t == g.lead) { lim = row + 1; step = -kKeyTile; }
    if (SPARSE && t == g.n_chunk) lim = g.cnt;
  }
  __device__ __forceinline__ void advance() { lim += step; }
};

// Maximum of 32 score columns.
__device__ __forceinline__ float max32(const uint32_t* v) {
  float m0 = __uint_as_float(v[0]), m1 = __uint_as_float(v[1]);
#pragma unroll
  for (int i = 2; i < 30; i += 4) {
    m0 = max3(m0, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
    m1 = max3(m1, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
  }
  return max3(m0, m1, fmaxf(__uint_as_float(v[30]), __uint_as_float(v[31])));
}

// ---------------------------------------------------------------------------------------------- softmax of one tile
// One thread = one query row of a 128-row Q tile against one 128-key tile: S is read from tensor memory at s_addr, bf16 P
// written at p_addr, 16 columns at a time, the running reference point m_run (log2 units) and sum l_run kept up, the
// accumulator at o_addr rescaled when the reference point moves.  `lim` = visible columns of this row, `masked` = some row
// of the warp sees fewer than all; first_tile: nothing has been accumulated yet; announce(half) (lane 0): a half of P is in
// place; o_idle: no product into O is on its way.  False when a wait gave up.
// APART: P has columns of its own.  All of S is read at once and `s_read` (lane 0) tells so, for the next tile's QK^T to go
// into its columns while the exponentials run; `p_free` waits for the products of the tile before, which read P (as a rule
// they are done; one wait, ahead of the exponentials, which the compiler would not interleave across it).
// Otherwise P goes over the first 64 columns of S and the last 32 scores are read once more, under the third block's
// exponentials: 128 scores and a block of exponentials in flight are a few registers more than the 168.
template <int D, bool APART, typename SRead, typename PFree, typename OIdle, typename Announce>
__device__ __forceinline__ bool attn_softmax_tile(uint32_t s_addr, uint32_t p_addr, uint32_t o_addr, int lim, bool masked,
                                                  float scale_log2, bool first_tile, int lane, float& m_run, float& l_run,
                                                  SRead&& s_read, PFree&& p_free, OIdle&& o_idle, Announce&& announce) {
  // ---- pass 1: the row maximum; all four 32-column loads are issued together (one tensor-memory round trip)
  constexpr int kHeld = APART ? 128 : 96;
  uint32_t v0[kHeld];
  float mx;
  {
    uint32_t c3[APART ? 1 : 32];
    uint32_t* last = APART ? v0 + (kHeld - 32) : c3;
    tmem_ld32(s_addr, v0);
    tmem_ld32(s_addr + 32, v0 + 32);
    tmem_ld32(s_addr + 64, v0 + 64);
    tmem_ld32(s_addr + 96, last);
    tmem_wait_ld();
    if (APART) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) s_read();
    }
    if (masked) {                                          // one branch: four of them were 2 % of the kernel
#pragma unroll
      for (int i = 0; i < kHeld; ++i) if (i >= lim) v0[i] = 0xFF800000u;      // -inf: exp2 gives exactly 0
      if (!APART) {
#pragma unroll
        for (int i = 0; i < 32; ++i) if (96 + i >= lim) last[i] = 0xFF800000u;
      }
    }
    mx = fmaxf(fmaxf(max32(v0), max32(v0 + 32)), fmaxf(max32(v0 + 64), max32(last)));
  }
  const float m_tile = mx * scale_log2;
  // ---- lazy rescale of the accumulator: only when some row's maximum grew by more than the threshold
  const bool grow = m_tile > m_run + kRescaleThreshold;
  if (!p_free()) return false;
  if (__any_sync(0xFFFFFFFFu, grow)) {
    const float m_new = fmaxf(m_run, m_tile);
    if (!first_tile) {
      if (!o_idle()) return false;
      const float alpha = (m_run == -INFINITY) ? 0.f : ex2(m_run - m_new);      // (nothing seen yet: O is wiped)
      l_run *= alpha;
#pragma unroll 1
      for (int c = 0; c < D / 8; ++c) {                       // rare: small pieces, few registers
        uint32_t r[8];
        tmem_ld8(o_addr + c * 8, r);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; ++i) r[i] = m_run == -INFINITY ? 0u : __float_as_uint(__uint_as_float(r[i]) * alpha);
        tmem_st8(o_addr + c * 8, r);
      }
      tmem_wait_st();
    }
    m_run = m_new;
  }
  const float m_use = (m_run == -INFINITY) ? 0.f : m_run;
  // ---- pass 2: p = 2^(s*scale - m) in four blocks of 32 keys, each half of the tile handed to the issuing warp as soon as
  // it is stored, so the first PV products run under the second half's arithmetic.
  const uint64_t sc2 = pack2(scale_log2, scale_log2), nm2 = pack2(-m_use, -m_use);
  uint64_t psa[2] = {0ull, 0ull};                           // four running sums as two packed pairs
  uint32_t vb[APART ? 1 : 32];
#pragma unroll
  for (int blk = 0; blk < 4; ++blk) {
    if (!APART && blk == 2) tmem_ld32(s_addr + 96, vb);
    if (!APART && blk == 3) {
      tmem_wait_ld();
      if (masked) {
#pragma unroll
        for (int i = 0; i < 32; ++i) if (96 + i >= lim) vb[i] = 0xFF800000u;
      }
    }
    uint32_t pk[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t* v = APART || blk < 3 ? v0 + blk * 32 : vb;
      float x0, x1;
      unpack2(fma2(pack2u(v[2 * i], v[2 * i + 1]), sc2, nm2), x0, x1);
      const float p0 = ex2(x0), p1 = ex2(x1);
      psa[i & 1] = add2(psa[i & 1], pack2(p0, p1));
      const __nv_bfloat162 b2 = __floats2bfloat162_rn(p0, p1);
      pk[i] = *reinterpret_cast<const uint32_t*>(&b2);
    }
    tmem_st16(p_addr + blk * 16, pk);
    if (blk & 1) {
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) announce(blk >> 1);
    }
  }
  float ps0, ps1, ps2, ps3;
  unpack2(psa[0], ps0, ps1);
  unpack2(psa[1], ps2, ps3);
  l_run += (ps0 + ps1) + (ps2 + ps3);
  return true;
}

// ---------------------------------------------------------------------------------------------- order of the products
// Two warps issue the products, each in order: one every S = Q K^T, one every O += P V.  An item is one Q tile against one
// key tile; items run A0 B0 A1 B1 ... (a Q tile that does not take part in a key tile has no item there).  S has NBUF
// tensor-memory buffers, used in turn; the QK^T of item i + NBUF waits until item i's is free, and nothing else orders it
// against PV.
//   head_dim 128, pairs: O takes 256 of the 512 columns, one S and two P (one per Q tile) the rest: S is free when item i's scores
//     have been READ, the next QK^T then runs under item i's exponentials.
//   head_dim 64: O takes 128 columns, three S the rest, P in place: free when item i's weights have been multiplied, which
//     is an item and a half before its next scores are wanted.
//   head_dim 128, one CTA: O takes 256 columns, two S the rest, P in place: with two Q tiles a tile's next QK^T waits for its own
//     products (1.91 us a step where a pair takes 1.39), with one it has both buffers (1.02).
// So a softmax warp finds its next scores ready, or nearly, when it is done with a tile.  Two warps because a wait on a
// barrier that is complete already costs 75 to 100 cycles and there are five to a pair of products, which take 1024: one
// warp for both left the tensor core idle for 45 % of a step (3650 cycles at head_dim 128).  Products of two warps
// interleave without loss (2050 cycles for 32, alone).
// The ring holds K0 V0 K1 V1 ...; a slot is released as its last product is issued.
template <int SLOTS>
struct RingCursor {                                         // every second item of the ring
  int slot;
  uint32_t phase = 0;
  __device__ __forceinline__ explicit RingCursor(int first) : slot(first) {}
  __device__ __forceinline__ void advance() {
    slot += 2;
    if (slot >= SLOTS) { slot -= SLOTS; phase ^= 1; }
  }
};

// acquire(slot, phase): the slot's K rows are readable; s_free(buf, parity): S buffer `buf` is free again (both false
// when a wait gave up); qk(x, buf, slot): the products and their commit; release(slot): commit of the slot.
template <int NBUF, int SLOTS, typename Resolve, typename Acquire, typename SFree, typename Qk, typename Release>
__device__ __forceinline__ void attn_issue_qk(AttnGeom& g, int t_lo, Resolve&& resolve_list, Acquire&& acquire, SFree&& s_free,
                                              Qk&& qk, Release&& release) {
  RingCursor<SLOTS> k(0);
  unsigned item = 0;
#pragma unroll 1
  for (int t = t_lo;; ++t, k.advance()) {
    if (t == g.n_known && !g.resolved) resolve_list();
    if (t >= g.n_known) return;
    if (!acquire(k.slot, k.phase)) return;
#pragma unroll 1
    for (int x = t >= g.skip_a ? 0 : 1; x < (g.active_b ? 2 : 1); ++x, ++item) {
      const unsigned buf = item % NBUF;
      if (item >= NBUF && !s_free(buf, (item / NBUF + 1) & 1)) return;
      qk(x, buf, k.slot);
    }
    release(k.slot);
  }
}

// acquire(slot, phase): the slot's V rows are readable; pv(x, half, buf, slot, add): waits for that half of P, products, commit;
// final(x): commit of the finished O.
template <int NBUF, int SLOTS, typename Resolve, typename Acquire, typename Pv, typename Release, typename Final>
__device__ __forceinline__ void attn_issue_pv(AttnGeom& g, int t_lo, Resolve&& resolve_list, Acquire&& acquire, Pv&& pv,
                                              Release&& release, Final&& final) {
  RingCursor<SLOTS> v(1);
  const int first_a = max(g.skip_a, t_lo);
  unsigned item = 0;
#pragma unroll 1
  for (int t = t_lo;; ++t, v.advance()) {
    if (t == g.n_known && !g.resolved) resolve_list();
    if (t >= g.n_known) break;
    if (!acquire(v.slot, v.phase)) return;
#pragma unroll 1
    for (int x = t >= g.skip_a ? 0 : 1; x < (g.active_b ? 2 : 1); ++x, ++item) {
      const unsigned buf = item % NBUF;
      if (!pv(x, 0, buf, v.slot, t != (x ? t_lo : first_a)) || !pv(x, 1, buf, v.slot, true)) return;
      if (g.resolved && t == g.n_known - 1) final(x);
    }
    release(v.slot);
    if (!g.resolved && t == g.n_known - 1) {                // (an empty list: the chunk's last tile was the last)
      resolve_list();
      if (t == g.n_known - 1)
        for (int x = t >= g.skip_a ? 0 : 1; x < (g.active_b ? 2 : 1); ++x) final(x);
    }
  }
}

// Epilogue of a softmax thread: its row of O from tensor memory, divided by l, to global memory as bf16 (and the
// row's log-sum-exp when asked for).
template <int D>
__device__ __forceinline__ void attn_store_row(const DevParams& P, uint32_t o_addr, float m_run, float l_run, int s, int h,
                                               int row, bool store, __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
  const float inv = 1.f / l_run;
  __nv_bfloat16* orow = out + (long long)s * P.o_sb + (long long)h * P.o_sh + (long long)row * P.o_st;
#pragma unroll
  for (int c = 0; c < D / 32; ++c) {
    uint32_t r[32];
    tmem_ld32(o_addr + c * 32, r);
    tmem_wait_ld();
    if (store) {
#pragma unroll
      for (int v4 = 0; v4 < 4; ++v4) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(r[v4 * 8 + 2 * i]) * inv,
                                                           __uint_as_float(r[v4 * 8 + 2 * i + 1]) * inv);
          w[i] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        *reinterpret_cast<uint4*>(orow + c * 32 + v4 * 8) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
  if (store && lse)
    lse[((long long)s * P.n_q + h) * P.chunk + row] = (m_run + log2f(l_run)) * 0.6931471805599453f;
}

// ---------------------------------------------------------------------------------------------- split attention
// A launch whose grid is far smaller than the GPU cuts every row block's key tiles into parts, one CTA (pair) each.
constexpr int kSplitTileFloats = 130 * 128;     // one part's partial result of a 128-row Q tile

// Epilogue of a softmax warp of a split launch.
template <int D>
__device__ __forceinline__ void attn_split_epilogue(const DevParams& P, int job, int part, int n_parts, int x, int quarter,
                                                    int lane, int row_in_tile, int row, bool store, bool have, uint32_t o_addr,
                                                    float m_run, float l_run, int s, int h, __nv_bfloat16* out,
                                                    float* lse) {
  // ---- this part's partial result (reference point m, sum l, un-normalised O; a part without tiles for this
  // Q tile leaves m = -inf), then the merge by whichever part's warp arrives last.  One counter per (row block
  // of a head, softmax warp); nobody waits for anybody.  The parts are added up in part order, so the result
  // does not depend on which part came last.
  constexpr int kTile = kSplitTileFloats;                   // [D columns of O | m | l][128 rows], D <= 128
  float* tile0 = P.attn_partials + ((size_t)job * n_parts * 2 + x) * kTile;
  float* mine = tile0 + (size_t)part * 2 * kTile;
  if (have) {
#pragma unroll
    for (int c = 0; c < D / 32; ++c) {
      uint32_t r[32];
      tmem_ld32(o_addr + c * 32, r);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 32; ++i) mine[(c * 32 + i) * 128 + row_in_tile] = __uint_as_float(r[i]);
    }
  }
  mine[D * 128 + row_in_tile] = have ? m_run : -INFINITY;
  mine[(D + 1) * 128 + row_in_tile] = have ? l_run : 0.f;
  __threadfence();
  __syncwarp();
  int32_t* counter = P.attn_counters + (job * 2 + x) * 4 + quarter;
  int arrived = 0;
  if (lane == 0) arrived = atomicAdd(counter, 1);
  arrived = __shfl_sync(0xFFFFFFFFu, arrived, 0);
  if (arrived == n_parts - 1) {
    if (lane == 0) *counter = 0;                            // as the next launch expects it
    __threadfence();
    float wgt[8];
    float M = -INFINITY;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      wgt[q] = q < n_parts ? __ldcg(tile0 + (size_t)q * 2 * kTile + D * 128 + row_in_tile) : -INFINITY;
      M = fmaxf(M, wgt[q]);
    }
    float l = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float w = wgt[q] == -INFINITY ? 0.f : ex2(wgt[q] - M);
      if (q < n_parts) l += w * __ldcg(tile0 + (size_t)q * 2 * kTile + (D + 1) * 128 + row_in_tile);
      wgt[q] = w;
    }
    const float inv = 1.f / l;
    __nv_bfloat16* orow = out + (long long)s * P.o_sb + (long long)h * P.o_sh + (long long)row * P.o_st;
#pragma unroll 1
    for (int c = 0; c < D / 32; ++c) {
      float acc[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] = 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q < n_parts && wgt[q] != 0.f) {
          const float* src = tile0 + (size_t)q * 2 * kTile + (c * 32) * 128 + row_in_tile;
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] = fmaf(wgt[q], __ldcg(src + i * 128), acc[i]);
        }
      }
      if (store) {
#pragma unroll
        for (int v4 = 0; v4 < 4; ++v4) {
          uint32_t w[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(acc[v4 * 8 + 2 * i] * inv, acc[v4 * 8 + 2 * i + 1] * inv);
            w[i] = *reinterpret_cast<const uint32_t*>(&b2);
          }
          *reinterpret_cast<uint4*>(orow + c * 32 + v4 * 8) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
    if (store && lse) lse[((long long)s * P.n_q + h) * P.chunk + row] = (M + log2f(l)) * 0.6931471805599453f;
  }
}

// The same with the parts of a row block in one cluster: every part leaves its result in its own shared memory, and after a
// cluster barrier each adds up an equal share of the rows, in part order, reading the others through distributed shared
// memory.  Against results through global memory, an arrival counter and a merge by the last part to arrive (five
// dependent L2 round trips) it is about 6 us shorter; `attn_plan` has the times.
constexpr int kPartPitch = 132;                  // floats per row: 16 bytes off a multiple of the banks

// A softmax thread's row of O, its m and l.  Nothing of the CTA may still read the shared memory below `smem` + 2 tiles.
template <int D>
__device__ __forceinline__ void attn_part_to_smem(unsigned char* smem, float* ml, int x, int row_in_tile, bool have, uint32_t o_addr,
                                                  float m_run, float l_run) {
  float* row = reinterpret_cast<float*>(smem) + (x * 128 + row_in_tile) * kPartPitch;
  if (have) {
#pragma unroll 1
    for (int c = 0; c < D / 32; ++c) {
      uint32_t r[32];
      tmem_ld32(o_addr + c * 32, r);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<uint4*>(row + c * 32 + 4 * i) = make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
    }
  }
  ml[x * 256 + row_in_tile] = have ? m_run : -INFINITY;
  ml[x * 256 + 128 + row_in_tile] = have ? l_run : 0.f;
}

// One of n_warps warps; the CTA of part p with this CTA's rows has cluster rank p * stride + offset.  A row at a time, four
// elements per lane, in a loop kept small: this code runs once per launch, and instructions have to be fetched too (four rows
// side by side per warp, 10 KB of code, took 7.3 us for 32 rows of a CTA and four parts; this form 4.8: the reads of other
// CTAs' shared memory, 50 KB at about 14 bytes per clock).
template <int D>
__device__ __forceinline__ void attn_merge_cluster(const DevParams& P, unsigned char* smem, float* ml, int warp, int n_warps, int lane,
                                                   int stride, int offset, int parts, int part, const QRows& qr, int s,
                                                   __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
  constexpr int kMaxParts = 4;
  static_assert(D == 128, "four elements per lane");
  const uint32_t o0 = smem_u32(smem), ml0 = smem_u32(ml);
  const int rows_a = qr.count(P, 0), rows = rows_a + qr.count(P, 1);
#pragma unroll 1
  for (int i = part + parts * warp; i < rows; i += parts * n_warps) {
    const int x = i < rows_a ? 0 : 1, lr = x ? i - rows_a : i;                  // i-th row that exists
    const uint32_t at = map_to_cta(ml0 + (uint32_t)(x * 256 + lr) * 4u, (uint32_t)(min(lane, parts - 1) * stride + offset));
    float m = ld_cluster_f(at), l = ld_cluster_f(at + 512u);                    // lane p: part p's
    // every part's elements before the first use of any (what a part without a result has there is not used)
    float4 v[kMaxParts];
#pragma unroll
    for (int p = 0; p < kMaxParts; ++p)
      v[p] = ld_cluster_f4(map_to_cta(o0 + (uint32_t)((x * 128 + lr) * kPartPitch + 4 * lane) * 4u, (uint32_t)(min(p, parts - 1) * stride + offset)));
    if (lane >= parts) { m = -INFINITY; l = 0.f; }
    float M = m;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
    M = __shfl_sync(0xFFFFFFFFu, M, 0);
    const float wgt = m == -INFINITY ? 0.f : ex2(m - M);
    float L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int p = 0; p < kMaxParts; ++p) {                                       // (lanes past the parts hold a weight of 0)
      const float w = __shfl_sync(0xFFFFFFFFu, wgt, p);
      const float4 o = w != 0.f ? v[p] : make_float4(0.f, 0.f, 0.f, 0.f);
      L = fmaf(w, __shfl_sync(0xFFFFFFFFu, l, p), L);
      acc.x = fmaf(w, o.x, acc.x); acc.y = fmaf(w, o.y, acc.y);
      acc.z = fmaf(w, o.z, acc.z); acc.w = fmaf(w, o.w, acc.w);
    }
    const float inv = 1.f / L;
    const __nv_bfloat162 a = __floats2bfloat162_rn(acc.x * inv, acc.y * inv), b = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
    const int h = qr.head(P, lr), p = qr.position(P, x, lr);
    *reinterpret_cast<uint2*>(out + (long long)s * P.o_sb + (long long)h * P.o_sh + (long long)p * P.o_st + 4 * lane) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    if (lse && lane == 0) lse[((long long)s * P.n_q + h) * P.chunk + p] = (M + log2f(L)) * 0.6931471805599453f;
  }
}

}  // namespace quoka
