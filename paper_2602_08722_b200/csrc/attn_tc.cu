// Flash-style attention on the 5th-generation tensor cores over
//   [selected cached rows | the chunk's own causal rows]      (Algorithm 2's attention line, Eq. 2)
// or, without an index list, over every cached row (Eq. 2, dense chunk attention).  bf16 in, fp32
// softmax and accumulation, P rounded to bf16 for the PV product.
//
// This file: the kernel whose row blocks are those of one CTA, and the plan and the launches of both (attn_tc_pair.cu has the
// one of pairs, for head_dim 128).  A CTA owns two Q tiles (A, B) of 128 rows, or one, chunk positions of all heads of a KV group, and walks the key
// tiles (128 keys) once for both.  Roles:
//   warps 0-3 / 4-7  softmax of Q tile A / B: one thread per query row, S read from tensor memory,
//                    running max / sum in registers, P written back to tensor memory, lazy rescale of
//                    the O accumulator (only when the max grew by more than 2^32), final
//                    normalisation and the global store.
//   warps 8-9        loaders: every K / V row of a tile is fetched with 16-byte cp.async straight
//                    into the 128-byte-swizzled layout the MMA descriptors expect.  The row address
//                    comes from the selected-index list (the gather), the chunk offset, or the page
//                    table, so no compacted copy of K or V is ever made; rows past the end are
//                    zero-filled.  A slot's "full" barrier is armed by the copies themselves.
//   warp 10          issues O += P V (P from tensor memory, V in shared memory, MN-major)
//   warp 11          issues S = Q K^T (both operands in shared memory)
// Where S and P live and what the products wait for: "order of the products" in attn_tiles.cuh.
// K and V tiles share one ring of shared-memory slots in the order K0 V0 K1 V1 ...
// 384 threads and no register re-balancing between roles: every thread may use 168 registers, a thirteenth warp would
// leave it 128.  Sixteen softmax warps with half a row each (96 registers) were slower: 121 us where these take 100
// (777 queries of 32 heads over 5000 listed rows, head_dim 64, the whole call).
#include <algorithm>
#include <cmath>
#include "attn_tiles.cuh"

namespace quoka {

template <int D>
constexpr int kSlotsOf = D == 64 ? 8 : 5;                    // of 16 KB, 32 KB
template <int D>
constexpr size_t kAttnSmem = 1024 + (size_t)(2 + kSlotsOf<D>) * (D / 64) * 16384 + 512;

template <int D, bool SPARSE, bool SPLIT>
__global__ void __launch_bounds__(kAttnThreads, 1)
attn_tc_kernel(DevParams P, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const __nv_bfloat16* __restrict__ kc,
               const __nv_bfloat16* __restrict__ vc, const int32_t* __restrict__ k_idx,
               const int32_t* __restrict__ k_cnt, __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
  constexpr int kSlots = kSlotsOf<D>, HALVES = D / 64;
  constexpr uint32_t kHalfBytes = 128 * 128;                 // 128 rows x 128 B
  constexpr uint32_t kTileBytes = HALVES * kHalfBytes;       // one Q / K / V tile
  // tensor memory (see "order of the products"): S | S | S | O_A | O_B, head_dim 128: S | S | O_A | O_B; P in place
  constexpr int NBUF = D == 64 ? 3 : 2;
  constexpr uint32_t O_COL = NBUF * 128;                     // (Q tile B's O is D columns on)
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* q_smem = smem;                               // [2][HALVES][128][128 B]
  unsigned char* kv_smem = smem + 2 * kTileBytes;             // [kSlots][HALVES][128][128 B]
  uint64_t* bars = reinterpret_cast<uint64_t*>(kv_smem + (size_t)kSlots * kTileBytes);
  uint64_t* kv_full = bars;                 // [kSlots]  the loader threads' cp.async arrivals
  uint64_t* kv_empty = bars + kSlots;       // [kSlots]  MMA commit
  uint64_t* s_full = bars + 2 * kSlots;     // [NBUF]    MMA commit
  uint64_t* p_full = s_full + NBUF;         // [NBUF][2] 4 softmax warps arrive, per half of the key tile
  uint64_t* p_done = p_full + 2 * NBUF;     // [NBUF]    MMA commit: P has been multiplied, the buffer is free
  uint64_t* o_full = p_done + NBUF;         // [2]       MMA commit after the last PV
  uint64_t* q_full = o_full + 2;            // TMA
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(q_full + 1);
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WaitCtx wc{&abort_flag, P.status};
  // grid = (head groups, row blocks, batch): head groups vary fastest, the row blocks run heaviest (most causal tiles)
  // first, lightest last, the sequences longest first
  const int s = longest_first(P, blockIdx.z), hg = blockIdx.x;
  // (SPLIT: grid.y = row blocks times the parts a row block's key tiles are cut into)
  const int n_parts = SPLIT ? P.attn_parts : 1;
  const int rb = (SPLIT ? P.attn_split_rb : P.attn_row_blocks) - 1 - blockIdx.y / n_parts;
  const QRows qr(P, hg, rb, 0, 1);
  const int kv = qr.head0 / P.group;
  AttnGeom g = make_geom<SPARSE>(P, s, qr.p0, 1);
  // SPLIT: this CTA walks the tiles [t_lo, t_hi) of the row block's sequence only and leaves, per row, a partial
  // result; the part that finishes last adds the parts up.  The list length has to be known before the range is, so
  // nothing of the walk starts before the selection has ended.
  int t_lo = 0;
  if (SPLIT) {
    if (SPARSE) { if (P.attn_after_whole) learn_count(g, k_cnt, s); else resolve(g, k_cnt, s); }
    const int part = blockIdx.y % n_parts;
    t_lo = (int)(((long long)part * g.n_known) / n_parts);
    g.n_known = (int)(((long long)(part + 1) * g.n_known) / n_parts);
  }

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int i = 0; i < kSlots; ++i) { mbar_init(&kv_full[i], kLoaderWarps * 32); mbar_init(&kv_empty[i], 1); }
    for (int i = 0; i < NBUF; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_done[i], 1); }
    for (int i = 0; i < 2 * NBUF; ++i) mbar_init(&p_full[i], 4);
    for (int i = 0; i < 2; ++i) mbar_init(&o_full[i], 1);
    mbar_init(q_full, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
  }
  if (warp == kQkWarp) tmem_alloc(tmem_slot, 512);
  zero_spare_q_rows<D>(P, q_smem, threadIdx.x, kAttnThreads);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (!SPARSE && !SPLIT) grid_launch_dependents();

  if (warp < 8) {
    // ================================================================== softmax + epilogue
    const int x = warp >> 2;                                  // Q tile A (0) or B (1)
    const int quarter = warp & 3;
    const int row_in_tile = quarter * 32 + lane;
    const int row = qr.position(P, x, row_in_tile);           // chunk position
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t o_addr = lane_addr + O_COL + x * D;
    const float scale_log2 = P.scale * 1.4426950408889634f;
    float m_run = -INFINITY, l_run = 0.f;
    // S buffers go by items: the first of this Q tile's is item 0, or 1 where the other comes first, the next one `step` on
    uint32_t phase = 0;
    int buf = (x ? t_lo >= g.skip_a : g.skip_a > t_lo) ? 1 : 0;
    const int step = g.active_b ? 2 : 1;
    bool ok = true;
    const int skip_x = max(x ? 0 : g.skip_a, t_lo);         // first tile this Q tile takes part in
    const bool active_x = (x ? g.active_b : true) && (!SPLIT || skip_x < g.n_known);
    VisibleCols<SPARSE> vis(g, skip_x, row);
    for (int t = skip_x; active_x; ++t, vis.advance()) {
      if (t == g.n_known) {                                   // end of what is known: the list length, or the end
        if (g.resolved) break;
        resolve(g, k_cnt, s);
        if (t == g.n_known) break;
      }
      vis.at(g, t, row);
      const bool masked = !__all_sync(0xFFFFFFFFu, vis.lim >= kKeyTile);
      if (!mbar_wait(&s_full[buf], phase, wc)) { ok = false; break; }
      tc_fence_after();
      const uint32_t s_addr = lane_addr + buf * 128;
      ok = attn_softmax_tile<D, false>(
          s_addr, s_addr, o_addr, vis.lim, masked, scale_log2, t == skip_x, lane, m_run, l_run, []() {}, []() { return true; },
          [&]() {                                             // products of this Q tile's item before
            const int before = buf - step;
            if (!mbar_wait_done(&p_done[before < 0 ? before + NBUF : before], before < 0 ? phase ^ 1 : phase, wc)) return false;
            tc_fence_after();
            return true;
          },
          [&](int half) { mbar_arrive(&p_full[2 * buf + half]); });
      if (!ok) break;
      buf += step;
      if (buf >= NBUF) { phase ^= 1; buf -= NBUF; }
    }
    // ---- epilogue: O / l -> bf16 -> global
    if constexpr (!SPLIT) {
      if (ok && active_x && mbar_wait(&o_full[x], 0, wc)) {
        tc_fence_after();
        attn_store_row<D>(P, o_addr, m_run, l_run, s, qr.head(P, row_in_tile), row, row_in_tile < qr.count(P, x), out, lse);
      }
    } else {
      const bool have = ok && active_x && mbar_wait(&o_full[x], 0, wc);
      if (have) tc_fence_after();
      attn_split_epilogue<D>(P, (s * QRows::groups(P) + hg) * P.attn_split_rb + rb, blockIdx.y % n_parts, n_parts, x, quarter, lane,
                             row_in_tile, row, row_in_tile < qr.count(P, x), have, o_addr, m_run, l_run, s, qr.head(P, row_in_tile),
                             out, lse);
    }
  } else if (warp < 8 + kLoaderWarps) {
    // ================================================================== K / V row loaders (gather)
    // One warp instruction copies four whole rows (eight lanes x 16 bytes cover a 128-byte row; head_dim 128: two); the row
    // groups of a tile are dealt round-robin to the loader warps.
    const int lw = warp - 8;
    constexpr int PIECES = D / 8;                             // 16-byte pieces per row (16 or 8)
    constexpr int ROWS_PER_INSTR = 32 / PIECES;               // 2 or 4
    constexpr int GROUPS = kKeyTile / ROWS_PER_INSTR;         // 64 or 32 row groups per tile
    constexpr int RPT = GROUPS / kLoaderWarps;                // row groups per warp
    const int c16 = lane % PIECES;                            // this thread's piece of the row
    const int rsub = lane / PIECES;
    // a thread's rows are 8 apart and have the same swizzle, or 4 apart, and it is turned by 4 rows for every second one
    static_assert(kLoaderWarps * ROWS_PER_INSTR == (HALVES == 1 ? 8 : 4), "rows of a thread");
    const int lrow = lw * ROWS_PER_INSTR + rsub;
    const uint32_t thread_dst = (uint32_t)((c16 >> 3) * kHalfBytes + lrow * 128 + (((c16 & 7) ^ lrow) << 4));
    const auto row_dst = [](uint32_t dst, int i) {
      return (HALVES == 1 || (i & 1) == 0 ? dst : dst ^ 64u) + (uint32_t)(i * kLoaderWarps * ROWS_PER_INSTR * 128);
    };
    const int32_t* idx = SPARSE ? k_idx + ((long long)s * P.n_kv + kv) * P.budget_cap : nullptr;
    uint32_t phase = 0;
    int slot = 0;
    const uint32_t kv_base = smem_u32(kv_smem);
    // Row addressing in 16-byte units, 32 bits wide (the host refuses caches of 2^32 - 1 units and more; strides are
    // multiples of 8 elements): sequence/head base plus this thread's piece, row stride, page stride.
    const uint32_t st16 = (uint32_t)(P.kv_st >> 3), sb16 = (uint32_t)(P.kv_sb >> 3);
    const uint32_t base16 = (uint32_t)(((P.page_size == 0 ? (long long)s * P.kv_sb : 0ll) + (long long)kv * P.kv_sh) >> 3) +
                            (uint32_t)c16;
    const int32_t* table = P.block_table + (long long)s * P.max_pages;
    // The warp's RPT * ROWS_PER_INSTR rows of a tile are numbered p = i * ROWS_PER_INSTR + rsub (i = its i-th row group); lane
    // l looks after rows p = l and p = 32 + l: their row numbers (-1 past the end), for listed rows fetched when the
    // previous tile's copies have been issued and looked at when this tile's are, and their offsets, worked out once per
    // tile.  The thread that copies a row fetches its offset by shuffle.  The per-row code is kept free of branches: a branch
    // per row costs a single warp far more than the arithmetic it skips.
    constexpr int LIST_REGS = RPT * ROWS_PER_INSTR / 32;
    static_assert(GROUPS % kLoaderWarps == 0 && RPT * ROWS_PER_INSTR % 32 == 0, "whole registers of rows");
    int rows[LIST_REGS], rr_of[LIST_REGS];
    uint32_t offs[LIST_REGS];
    bool all_rows = false;
#pragma unroll
    for (int k = 0; k < LIST_REGS; ++k) {
      const int pp = 32 * k + lane;
      rr_of[k] = (lw + (pp / ROWS_PER_INSTR) * kLoaderWarps) * ROWS_PER_INSTR + pp % ROWS_PER_INSTR;
      rows[k] = -1;
      offs[k] = kNoRow;
    }
    auto list_rows = [&](int base, int count) {
      const int last = min(count, kKeyTile) - 1;                   // last valid row of the tile
      if (last >= 0) {
#pragma unroll
        for (int k = 0; k < LIST_REGS; ++k) {
          const int v = __ldcg(idx + base + min(rr_of[k], last));  // written by the kernel before: L2, not the read-only path
          rows[k] = rr_of[k] <= last ? v : -1;
        }
      }
    };
    for (int tile = t_lo;; ++tile) {
      if (tile == g.n_known) {                                // end of what is known: the list length, or the end
        if (g.resolved) break;
        resolve(g, k_cnt, s);
        if (tile == g.n_known) break;
      }
      const TileRows tr = tile_rows<SPARSE>(g, tile);
      bool stop = false;
#pragma unroll 1
      for (int kvi = 0; kvi < 2; ++kvi) {                     // the tile's K rows, then its V rows
        if (!mbar_wait_done(&kv_empty[slot], phase ^ 1, wc)) { stop = true; break; }
        // A whole tile of consecutive rows (page-aligned in a paged cache) is fetched by the copy engine as 64-row
        // boxes: one thread issues them, the others only keep the barrier's arrival count.  Ragged tiles (rows past
        // the end must read as zeros, not as whatever the cache holds there) and listed rows take the copies below.
        if (!tr.from_list && tr.count >= kKeyTile && (P.page_size == 0 || (tr.first & (kPage - 1)) == 0)) {
          if (lw == 0 && lane == 0) {
            fence_proxy_async_smem();             // earlier contents of the slot were written through the generic proxy
            mbar_arrive_expect_tx(&kv_full[slot], kTileBytes);
            unsigned char* dst = kv_smem + (size_t)slot * kTileBytes;
            const CUtensorMap* tm = kvi ? &tm_v : &tm_k;
#pragma unroll
            for (int sub = 0; sub < 2; ++sub) {
              int c1 = tr.first + sub * 64, c3 = s;
              if (P.page_size != 0) { c1 = 0; c3 = __ldg(table + (tr.first >> 6) + sub); }
#pragma unroll
              for (int hh = 0; hh < HALVES; ++hh)
                tma_load_4d(dst + hh * kHalfBytes + sub * 64 * 128, tm, &kv_full[slot], hh * 64, c1, kv, c3);
            }
          } else {
            mbar_arrive(&kv_full[slot]);
          }
          if (++slot == kSlots) { slot = 0; phase ^= 1; }
          continue;
        }
        if (kvi == 0) {
          if (tr.from_list && tile == max(g.n_chunk, t_lo)) list_rows(tr.first, tr.count);   // first list tile
#pragma unroll
          for (int k = 0; k < LIST_REGS; ++k) {
            if (!tr.from_list) rows[k] = rr_of[k] < tr.count ? tr.first + rr_of[k] : -1;
            offs[k] = kv_row_off16(P, table, st16, sb16, rows[k], tr.from_list, g.T);
            all_rows = (k == 0 || all_rows) && offs[k] != kNoRow;
          }
          all_rows = warp_all(all_rows);
        }
        const uint4* src_base = reinterpret_cast<const uint4*>(kvi ? vc : kc) + base16;
        const uint32_t dst = kv_base + slot * kTileBytes + thread_dst;
        if (all_rows) {                                           // no size to select
#pragma unroll
          for (int i = 0; i < RPT; ++i) {
            const uint32_t off = __shfl_sync(0xFFFFFFFFu, offs[(i * ROWS_PER_INSTR) / 32], (i * ROWS_PER_INSTR + rsub) & 31);
            cp_async_16(row_dst(dst, i), src_base + off);
          }
        } else {
#pragma unroll
          for (int i = 0; i < RPT; ++i) {
            const uint32_t off = __shfl_sync(0xFFFFFFFFu, offs[(i * ROWS_PER_INSTR) / 32], (i * ROWS_PER_INSTR + rsub) & 31);
            cp_async_16(row_dst(dst, i), src_base + (off == kNoRow ? 0u : off), off != kNoRow);
          }
        }
        // this thread's share of the slot is signalled by the copy engine itself when the bytes have landed:
        // no wait in the loader, every slot of the ring can be in flight
        cp_async_mbar_arrive_noinc(&kv_full[slot]);
        if (kvi == 1 && tr.from_list) list_rows(tr.first + kKeyTile, tr.count - kKeyTile);   // next list tile
        if (++slot == kSlots) { slot = 0; phase ^= 1; }
      }
      if (stop) break;
    }
    cp_async_wait_all();                                      // nothing of this thread is in flight at exit
  } else {
    // ================================================================== warp 11: QK^T, warp 10: PV
    if (warp == kQkWarp && lane == 0) load_q_tiles<D>(P, qr, q_smem, &tm_q, q_full, s);
    __syncwarp();
    const bool leader = elect_one();
    const uint32_t tmem = (uint32_t)warp_uniform((int)tmem_base);
    t_lo = warp_uniform(t_lo);
    uniform_geom(g);
    const uint32_t kv_base = smem_u32(kv_smem);
    const auto acquire = [&](int sl, uint32_t phase) {
      if (!warp_all(mbar_poll(&kv_full[sl], phase, wc))) return false;
      fence_proxy_async_smem();               // cp.async wrote through the generic proxy, the MMA reads through the async one
      tc_fence_after();
      return true;
    };
    const auto release = [&](int sl) { if (leader) mma_commit(&kv_empty[sl]); };
    // Operand descriptors are built once; a tile, slot or k-step offset is an addition to the 16-byte-unit
    // address field (shared memory addresses stay far below the field's 14 bits).
    // The sparse sequence's length is learnt (resolve) just before the walk past the chunk's own tiles.
    if (warp == kQkWarp) {
      const uint32_t idesc_qk = idesc_bf16_f32(128, kKeyTile, false, false);
      const uint64_t desc_q = smem_desc_sw128(smem_u32(q_smem), 16, 1024);
      const uint64_t desc_k = smem_desc_sw128(kv_base, 16, 1024);            // K-major rows (K tiles)
      if (warp_all(mbar_poll(q_full, 0, wc)))
        attn_issue_qk<NBUF, kSlots>(
            g, t_lo, [&]() { resolve(g, k_cnt, s); uniform_geom(g); grid_launch_dependents(); }, acquire,
            [&](unsigned buf, uint32_t parity) {
              if (!warp_all(mbar_poll(&p_done[buf], parity, wc))) return false;
              tc_fence_after();
              return true;
            },
            [&](int x, unsigned buf, int ks) {
              const uint64_t da = desc_q + (uint64_t)(x * (kTileBytes >> 4));
              const uint64_t db = desc_k + (uint64_t)((uint32_t)ks * (kTileBytes >> 4));
#pragma unroll
              for (int hh = 0; hh < HALVES; ++hh)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                  const uint64_t o = (uint64_t)((hh * kHalfBytes + kk * 32) >> 4);
                  if (leader) mma_ss(tmem + buf * 128, da + o, db + o, idesc_qk, (hh | kk) ? 1u : 0u);
                }
              if (leader) mma_commit(&s_full[buf]);
            },
            release);
    } else {
      const uint32_t idesc_pv = idesc_bf16_f32(128, D, false, true);
      const uint64_t desc_v = smem_desc_sw128(kv_base, HALVES == 1 ? 16 : kHalfBytes, 1024);      // MN-major rows (V tiles)
      uint32_t p_phase = 0;
      attn_issue_pv<NBUF, kSlots>(
          g, t_lo, [&]() { resolve(g, k_cnt, s); uniform_geom(g); }, acquire,
          [&](int x, int half, unsigned buf, int vs, bool add) {
            if (!warp_all(mbar_poll(&p_full[2 * buf + half], (p_phase >> buf) & 1u, wc))) return false;
            tc_fence_after();
            const uint64_t dv = desc_v + (uint64_t)((uint32_t)vs * (kTileBytes >> 4) + half * 4 * (2048 >> 4));
            const uint32_t pa = tmem + buf * 128 + half * 32, oa = tmem + O_COL + x * D;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)             // 16 keys per MMA: 8 packed columns of P, 16 rows of V
              if (leader) mma_ts(oa, pa + kk * 8, dv + (uint64_t)(kk * (2048 >> 4)), idesc_pv, add || kk ? 1u : 0u);
            if (half) {
              if (leader) mma_commit(&p_done[buf]);
              p_phase ^= 1u << buf;
            }
            return true;
          },
          release, [&](int x) { if (leader) mma_commit(&o_full[x]); });
    }
  }
  if (SPLIT && attn_last_cta()) grid_dependency_wait();       // this grid's end is the whole row blocks' end too
  tc_fence_before();
  __syncthreads();
  if (warp == kQkWarp) tmem_dealloc(tmem_base, 512);
}

// ---------------------------------------------------------------------------------------------- host
// How an attention call is laid out on the GPU: the form of its row blocks, and parts of their key tiles.
//
// Forms: two Q tiles per CTA or one; at head_dim 128 a row block is that of a pair of CTAs or of one.  A pair's step (a key tile)
// is the faster one per row, one CTA's row blocks are smaller: chunks of a few positions, or few heads per KV head, leave
// a pair with CTAs or tiles without rows.
// Parts: a grid of fewer CTAs than SMs (short chunks, few heads) leaves part of the GPU idle while every CTA walks its whole
// key sequence; cutting each row block's tiles into parts, one CTA (pair) each, fills it.  Parts merge through memory, or,
// a pair's, in a cluster of 2 * parts CTAs where all of a grid's clusters are resident at once: the device holds 33, 22 or 15
// of 4, 6 or 8 CTAs of this shared memory, the limits leave some free (a second wave costs more than any split gives).
//
// The model, in microseconds: start and end of a CTA, its steps, and what parts cost on top; the parts of a sparse call start
// only when the selection has ended, whole row blocks walk the chunk's own tiles under it (half of these count).  Measured with
// one thing varied at a time, a step with one / two Q tiles: a pair 1.09 / 1.39 us (listed rows 1.25 / 1.45), one CTA at head_dim
// 128 1.02 / 1.91 (1.41 / 1.93: it gathers whole rows of its own), at head_dim 64 1.02 / 1.38 (1.13 / 1.42); parts through memory
// 9 us for two and 20 for eight, at head_dim 64 8 and 12; in a cluster 3 to 6.  Then moved, most by less than a tenth, to fit
// whole calls: 284 of them, 1 to 8 sequences, 5 to 32 heads, chunks of 16 to 3238, 2 to 516 tiles, each with every form
// and number of parts (5000 times).  The plan's choice takes 0.8 % more time than the best form in the geometric mean; pairs
// only and the same cost of parts for both head dims took 2 % (25 % at most).  For instance, this choice / the one
// before, us: dense, 8 heads of 8 KV heads, 1100 queries over 8192 rows 56 (one CTA, one tile, 2 parts) / 60 (pairs); 32 heads of 8,
// 128 over 8192 38 / 45; 32 heads of 32, 64 over 32768 96 / 176; sparse, 8 heads of 8, 1100 queries, 983 of 8192 rows 48 (pairs,
// one tile, whole) / 55 (two tiles, clusters of two parts).
//
// A grid of q full waves and a rest has its lightest row blocks, as many as the rest, cut instead: the whole ones then
// end after about q waves and the parts level the end.  The model is the total work over the SMs plus a third of a part
// for the uneven end, against q + 1 waves of average jobs.  48 calls without / with parts, in turns over the same buffers: what
// the model puts below 0.92 of the whole row blocks (sparse) and 0.94 (dense) gains 1 to 11 %,
// around the line some gain 5 % and some lose 7, above it nearly all lose 4 to 10.  32 heads, us, and the model: sparse, 3700 queries
// over 8192 of 65536 rows 621 / 561 (0.82), 1550 over 3932 of 32768 165 / 154 (0.86), 2900 over 8192 415 / 404 (0.91), 4096 over
// 15729 of 131072 1132 / 1086 (0.91), 1700 over 3932 168 / 182 (0.925), 3072 over 16384 828 / 784 (0.93), 1850 over 8192 270 / 287 (0.95), 2000
// over 8192 276 / 297 (1.01); head_dim 64 3800 over 3932 304 / 284 (0.85), 1850 over 8192 243 / 228 (0.91), 2000 over 8192 246 / 260 (0.99);
// dense, 1850 over 16384 411 / 392 (0.91), 3000 over 32768 1444 / 1331 (0.91), 2048 over 32768 967 / 914 (0.94), 1850 over 8192 217 / 241
// (0.95), 2150 over 32768 945 / 1002 (1.00); head_dim 64 2000 over 32768 746 / 682 (0.92), 3050 over 8192 331 / 344 (0.95).  Sparse
// calls of a batch stay whole (their budgets differ).
// Partial results above 128 MiB are not written where a call has as many blocks of 256 positions of a head as there are SMs
// (most such have waves enough; of those whose heads packed into tiles make fewer CTAs, eight parts of 127 CTAs and more,
// which only dense calls over 94,000 rows and more would take, for a promised tenth).

// How the query rows of a call are laid out: see QRows.
struct AttnShape {
  int span, block;                 // chunk positions of a Q tile and of a row block
  long long blocks, per_rb, jobs;  // row blocks of a head group; CTAs of one row block of every head; CTAs
};
static AttnShape attn_shape(const quoka_params* p, const AttnPlan& plan) {
  AttnShape a;
  a.span = kQTile / plan.pack;
  a.block = plan.q_tiles * plan.ctas * a.span;
  a.blocks = (p->chunk_len + a.block - 1) / a.block;
  a.per_rb = (long long)(p->n_q_heads / plan.pack) * plan.ctas * p->batch;
  a.jobs = a.per_rb * a.blocks;
  return a;
}
// Whole row blocks of two Q tiles per CTA (head_dim 128: of a pair of CTAs), `pack` heads to a tile.
static AttnPlan attn_whole(const quoka_params* p, int pack) {
  AttnPlan plan;
  plan.ctas = p->head_dim == 128 ? 2 : 1;
  plan.pack = pack;
  return plan;
}
// Heads that may share a Q tile: divisors of the group whose row blocks the grid's second dimension holds (32 heads to a tile
// at head_dim 64: chunks of 524280 positions; one head: of 16.7 million).
static bool attn_pack_fits(const quoka_params* p, int pack) {
  return p->n_q_heads / p->n_kv_heads % pack == 0 && (pack == 1 || attn_shape(p, attn_whole(p, pack)).blocks <= 65535);
}
static int attn_largest_pack(const quoka_params* p) {
  int pack = std::min(p->n_q_heads / p->n_kv_heads, 32);
  while (pack > 1 && !attn_pack_fits(p, pack)) --pack;
  return pack;
}
static double attn_step_us(const quoka_params* p, int q_tiles, int ctas, bool sparse) {
  static constexpr double us[3][2][2] = {{{1.02, 1.13}, {1.38, 1.42}},     // head_dim 64: one Q tile, two; dense, listed
                                         {{0.95, 1.35}, {2.00, 2.05}},     // head_dim 128, one CTA
                                         {{1.09, 1.25}, {1.35, 1.30}}};    // and a pair
  return us[p->head_dim == 64 ? 0 : ctas][q_tiles - 1][sparse ? 1 : 0];
}
// The plan for `pack` heads to a tile over `tiles` key tiles besides the chunk's own, with no more scratch than `room`;
// *model_us: what the model says.
static AttnPlan attn_plan_of(const quoka_params* p, int pack, int tiles, bool sparse, size_t room, long long sms, double* model_us) {
  constexpr double kStart[3] = {6.0, 9.0, 9.5}, kStartTwoOfPair = 11.5;                // head_dim 64, 128, a pair
  constexpr double kParts128 = 5.2, kPart128 = 1.6, kParts64 = 5.5, kPart64 = 1.0, kCluster = 3.8, kSparseParts = 3.0, kOwn = 0.5;
  const bool wide = p->head_dim == 128;
  AttnPlan plan = attn_whole(p, pack);
  const AttnShape two = attn_shape(p, plan);
  const auto own = [](long long positions) { return (double)((positions + kKeyTile - 1) / kKeyTile); };
  // at least as many blocks of 256 positions of a head as SMs
  const bool bounded = (long long)p->n_q_heads * p->batch * ((p->chunk_len + 255) / 256) >= sms;
  double best = 1e30;
  for (int ctas = wide ? 2 : 1; ctas >= 1; --ctas) {
    for (int q_tiles = 2; q_tiles >= 1; --q_tiles) {
      AttnPlan form = attn_whole(p, pack);
      form.q_tiles = q_tiles; form.ctas = ctas;
      const AttnShape a = attn_shape(p, form);
      // the last row block, which may have no second tiles, and the one before it
      const double step = attn_step_us(p, q_tiles, ctas, sparse);
      const long long before = (a.blocks - 1) * a.block;
      const double step_last = p->chunk_len - before <= ctas * a.span ? attn_step_us(p, 1, ctas, sparse) : step;
      const auto walk = [&](double w) {
        return std::max(step_last * (tiles + w * own(p->chunk_len)), before > 0 ? step * (tiles + w * own(before)) : 0.0);
      };
      const double start = ctas == 2 && q_tiles == 2 ? kStartTwoOfPair : kStart[wide ? ctas : 0];
      const double w = sparse ? kOwn : 1.0, x = (double)a.jobs / (double)sms;
      // (CTAs of a grid of waves do not start in step: between the number of waves and the mean)
      const double mean = step * (tiles + 0.5 * w * (own(p->chunk_len) + (double)a.block / kKeyTile));
      const double whole = a.jobs <= sms ? start + walk(w) : 0.5 * (x + std::ceil(x)) * (start + mean);
      // what lies further from the calls that the model was fitted to has to promise some percent: one CTA in the place of a pair,
      // parts through memory, more than a wave; in grids of a wave and more every other form
      const double sure = (wide && ctas == 1 ? 1.04 : 1.0) * (a.jobs > sms ? 1.02 : 1.0);
      const auto consider = [&](double us, int parts, bool in_cluster) {
        AttnPlan next = form;
        next.parts = parts; next.in_cluster = in_cluster;
        next.split_rb = parts > 1 ? (int)a.blocks : 0;
        us *= parts > 1 && !in_cluster ? 1.02 * sure : sure;
        if (best < 1e30 && (us >= (two.jobs >= sms ? 0.97 : 1.0) * best || a.blocks * parts > 65535)) return;
        if (attn_plan_scratch_bytes(p, next) > room || (bounded && attn_split_partial_bytes(p, next) > kMostAttnPartials)) return;
        best = us;
        plan = next;
      };
      consider(whole, 1, false);
      if (a.jobs > sms) continue;
      const double rest = start + (sparse ? kSparseParts : 0.0), t = walk(1.0);
      for (int parts = 2; parts <= 8 && 2 * parts <= tiles + 1; ++parts) {
        const double waves = (double)(((int)a.jobs * parts - 1) / (int)sms + 1);
        consider(rest + waves * (t / parts + (wide ? kParts128 + kPart128 * parts : kParts64 + kPart64 * parts)), parts, false);
        if (ctas == 2 && parts <= 4 && a.jobs / 2 <= (parts == 2 ? 28 : parts == 3 ? 20 : 14))
          consider(rest + t / parts + kCluster, parts, true);
      }
    }
  }
  *model_us = best;
  const long long n_rb = two.blocks, per_rb = two.per_rb, jobs = two.jobs;
  const long long q = jobs / sms, rest = jobs % sms;
  if (jobs < sms || rest == 0 || (sparse && p->batch > 1) || plan.q_tiles != 2 || plan.ctas != (wide ? 2 : 1)) return plan;
  constexpr double kPartCost = 6.0;
  const double own_step = (double)two.block / kKeyTile;                      // the chunk's own tiles grow by this per row block
  const long long split = (rest + per_rb - 1) / per_rb;                      // row blocks to cut; block r has about (r + 1) * own_step of its own tiles
  const double t_all = tiles + 3 + 0.5 * own_step * n_rb, t_whole = tiles + 3 + 0.5 * own_step * (split + n_rb), t_split = tiles + 3 + 0.5 * own_step * split;
  double least = (sparse ? 0.92 : 0.94) * (double)(q + 1) * t_all;
  for (int parts = 2; parts <= 8 && parts <= (tiles + 1) / 6; ++parts) {
    const double t_part = t_split / parts + kPartCost;
    const double cost = ((double)(jobs - split * per_rb) * t_whole + (double)(split * per_rb * parts) * t_part) / (double)sms + 0.3 * t_part;
    AttnPlan cand = attn_whole(p, pack);
    cand.split_rb = (int)split; cand.parts = parts;
    if (cost < least && attn_split_partial_bytes(p, cand) <= kMostAttnPartials && attn_plan_scratch_bytes(p, cand) <= room) {
      least = cost;
      plan = cand;
      *model_us = std::min(*model_us, kStartTwoOfPair + attn_step_us(p, 2, plan.ctas, sparse) * cost / 0.9);
    }
  }
  return plan;
}
// How many heads share a tile: the whole group where its heads fill tiles (1, 2, 4, 8, 16 or 32 of them), else the largest
// divisor that the model puts within 2 % of the best one.  More heads make fewer CTAs of a short chunk, and leave rows over in
// those of a long one.  Two KV heads over 16384 rows, every divisor of 15 groups of 9 to 40 heads, 64, 600 and 2048 queries, both head
// dims, sparse and dense: the choice takes 1.0 % more time than the best one in the geometric mean (18 % at most), the largest
// divisor up to 32 6 % (45 %).  Dense, 26 heads to a KV head, 1 / 2 / 13 / 26 of them to a tile: 64 queries, head_dim 128, 154 /
// 94 / 57 / 57 us; 2048 queries, head_dim 64, 597 / 586 / 630 / 791.
static AttnPlan attn_plan(const quoka_params* p, int tiles, bool sparse, size_t room) {
  const int largest = attn_largest_pack(p);
  const long long sms = device_sm_count();
  if (p->dtype != QUOKA_BF16 || p->impl == QUOKA_IMPL_SIMT || p->chunk_len <= 1 || sms <= 0) return attn_whole(p, largest);
  double best, us;
  AttnPlan plan = attn_plan_of(p, largest, tiles, sparse, room, sms, &best);
  if (kQTile % largest == 0) return plan;
  for (int pack = largest - 1; pack >= 1; --pack) {
    if (!attn_pack_fits(p, pack)) continue;
    const AttnPlan other = attn_plan_of(p, pack, tiles, sparse, room, sms, &us);
    if (us < 0.98 * best) { plan = other; best = us; }
  }
  return plan;
}
AttnPlan attn_plan_sparse(const quoka_params* p, int budget_cap, size_t room) { return attn_plan(p, (budget_cap + kKeyTile - 1) / kKeyTile, true, room); }
AttnPlan attn_plan_dense(const quoka_params* p, size_t room) { return attn_plan(p, (p->max_ctx_len + kKeyTile - 1) / kKeyTile, false, room); }
static size_t attn_split_jobs(const quoka_params* p, const AttnPlan& plan) { return (size_t)attn_shape(p, plan).per_rb * plan.split_rb; }
size_t attn_split_partial_bytes(const quoka_params* p, const AttnPlan& plan) {
  return plan.in_cluster ? 0 : attn_split_jobs(p, plan) * plan.parts * 2 * kSplitTileFloats * sizeof(float);
}
size_t attn_split_counter_bytes(const quoka_params* p, const AttnPlan& plan) { return plan.in_cluster ? 0 : attn_split_jobs(p, plan) * 8 * sizeof(int32_t); }
size_t attn_plan_scratch_bytes(const quoka_params* p, const AttnPlan& plan) {
  return (attn_split_counter_bytes(p, plan) + 255) / 256 * 256 + (attn_split_partial_bytes(p, plan) + 255) / 256 * 256;
}

// The launches of an attention call: the whole row blocks, then the ones in parts.
//
// Programmatic stream serialisation, (1) inside the fused call: the first launch may start while the kernel before it on
// the stream (the key selection, which signals early and writes none of this kernel's other inputs) still runs; it touches
// the selection's outputs only after its own griddepcontrol.wait.  A stand-alone call keeps the ordinary stream order:
// whatever ran before it may have written q, k or v.  (2) The parts always: their CTAs take the SMs that the whole row
// blocks' last wave leaves idle.  The whole row blocks let them start once every CTA has begun (dense) or has learnt the
// list length (sparse: the selection is complete by then, so the parts need not wait for it), and the parts' last CTA
// waits for the whole row blocks before it ends.
quoka_status launch_attn_plan(const quoka_params* p, const DevParams& P, const AttnPlan& plan, AttnKernel (*pick)(bool, bool, bool),
                              const char* name, int cluster, size_t smem, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
                              const CUtensorMap& tm_v, const void* k, const void* v, const int32_t* k_idx, const int32_t* k_cnt,
                              void* out, float* lse, cudaStream_t st, bool after_selection) {
  const bool sparse = k_idx != nullptr, split = plan.split_rb > 0 && (P.attn_partials || plan.in_cluster);
  DevParams PP = P;
  const AttnShape shape = attn_shape(p, plan);
  PP.attn_row_blocks = (int)shape.blocks;
  PP.attn_split_rb = split ? plan.split_rb : 0;
  PP.attn_parts = split ? plan.parts : 1;
  const int whole = PP.attn_row_blocks - PP.attn_split_rb;
  PP.attn_after_whole = whole > 0 ? 1 : 0;
  if (split && !plan.in_cluster && !after_selection &&          // (the fused call clears the counters in an earlier kernel)
      cudaMemsetAsync(P.attn_counters, 0, attn_split_counter_bytes(p, plan), st) != cudaSuccess)
    return QUOKA_ERR_CUDA;
  for (int parts = whole > 0 ? 0 : 1; parts <= (split ? 1 : 0); ++parts) {
    AttnKernel kernel = pick(sparse, parts != 0, plan.in_cluster);
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return QUOKA_ERR_CUDA;
    const bool early = parts && whole > 0 ? true : sparse && after_selection;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(shape.per_rb / P.batch), parts ? PP.attn_split_rb * PP.attn_parts : whole, P.batch);
    cfg.blockDim = dim3(kAttnThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    if (early) {
      attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (parts && plan.in_cluster) {           // (the other kernels' clusters are part of the kernel)
      attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
      attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
      attr[cfg.numAttrs].val.clusterDim.y = (unsigned)PP.attn_parts;
      attr[cfg.numAttrs++].val.clusterDim.z = 1;
    }
    log_launch(name, cfg.gridDim, cfg.blockDim, smem, parts && plan.in_cluster ? cluster * PP.attn_parts : cluster, early);
    if (cudaLaunchKernelEx(&cfg, kernel, PP, tm_q, tm_k, tm_v, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, k_idx, k_cnt,
                           (__nv_bfloat16*)out, lse) != cudaSuccess)
      return QUOKA_ERR_CUDA;
    count_launch();
  }
  return cudaGetLastError() == cudaSuccess ? QUOKA_OK : QUOKA_ERR_CUDA;
}

static AttnShape attn_usual_shape(const quoka_params* p) { return attn_shape(p, attn_whole(p, attn_largest_pack(p))); }
bool attn_below_a_wave(const quoka_params* p) { return attn_usual_shape(p).jobs < device_sm_count(); }
// (above a wave the cost of a plan with parts is more than q waves of average jobs, its line at most 0.94 (q + 1): none from q = 16 on)
bool attn_may_have_parts(const quoka_params* p) { return attn_usual_shape(p).jobs < 17ll * device_sm_count(); }
int attn_same_plan_up_to(const quoka_params* p, int chunk) {
  int last = (chunk + kKeyTile - 1) / kKeyTile * kKeyTile;
  for (int pack = attn_largest_pack(p); pack >= 1; --pack) {
    const int span = kQTile / pack;
    if (attn_pack_fits(p, pack)) last = std::min(last, (chunk + span - 1) / span * span);
  }
  return last;
}

bool attn_tc_supported(const quoka_params* p) {
  if (p->dtype != QUOKA_BF16) return false;
  // the loaders address cache rows in 32-bit units of 16 bytes
  const int64_t extent = (p->page_size ? p->kv_rows : (int64_t)p->batch) * p->kv_stride_b;
  if (extent / 8 >= (int64_t)0xFFFFFFFFll) return false;
  return true;
}

bool encode_q_tensor_map(CUtensorMap* out, const DevParams& P, const void* q) {
  const uint64_t dims[5] = {(uint64_t)P.d, (uint64_t)P.attn_pack, (uint64_t)P.chunk, (uint64_t)(P.n_q / P.attn_pack), (uint64_t)P.batch};
  const uint64_t strides[4] = {(uint64_t)P.q_sh * 2, (uint64_t)P.q_st * 2, (uint64_t)P.q_sh * 2 * P.attn_pack, (uint64_t)P.q_sb * 2};
  const uint32_t box[5] = {64, (uint32_t)P.attn_pack, (uint32_t)P.attn_span, 1, 1};
  return encode_tensor_map_bf16(out, q, 5, dims, strides, box);
}

template <int D>
static AttnKernel pick_attn_tc(bool sparse, bool parts, bool) {
  if (parts) return sparse ? attn_tc_kernel<D, true, true> : attn_tc_kernel<D, false, true>;
  return sparse ? attn_tc_kernel<D, true, false> : attn_tc_kernel<D, false, false>;
}

quoka_status launch_attn_tc(const quoka_params* p, const DevParams& P0, const void* q, const void* k, const void* v,
                            const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st,
                            bool after_selection, const AttnPlan& plan) {
  DevParams P = P0;
  P.attn_pack = plan.pack;
  P.attn_span = attn_shape(p, plan).span;
  P.attn_qtiles = plan.q_tiles;
  if (plan.ctas == 2) return launch_attn_tc_pair(p, P, q, k, v, k_idx, k_cnt, out, lse, st, after_selection, plan);
  CUtensorMap tm_q, tm_k, tm_v;
  if (!encode_q_tensor_map(&tm_q, P, q)) return QUOKA_ERR_CUDA;
  if (!encode_kv_tensor_map(&tm_k, p, k, 64) || !encode_kv_tensor_map(&tm_v, p, v, 64)) return QUOKA_ERR_CUDA;
  const bool wide = P.d == 128;
  return launch_attn_plan(p, P, plan, wide ? pick_attn_tc<128> : pick_attn_tc<64>, "attn_tc", /*cluster=*/1,
                          wide ? kAttnSmem<128> : kAttnSmem<64>, tm_q, tm_k, tm_v, k, v, k_idx, k_cnt, out, lse, st, after_selection);
}

}  // namespace quoka
