// The tensor-core attention kernel for head_dim 128: two CTAs with neighbouring chunk positions of one KV group run as a
// PAIR (a cluster of two on neighbouring SMs) and share every K / V tile.
//
// Both walk the same key tiles in the same order (the selected list depends on the KV head only; the causal limits end
// within a few tiles of each other), so one `tcgen05.mma.cta_group::2` covers both: 256 rows of S (or O), 128 per CTA, with
// the K (or V) operand split between the two CTAs' shared memories.
//   S = Q K^T : each CTA supplies its own Q tile and 64 of the tile's 128 keys (all 128 elements of each).
//   O += P V  : each CTA supplies its own P (tensor memory) and 64 of V's 128 columns (all 128 keys).
// So a CTA fetches HALF of every K and V tile (the 16-byte cp.async gather of listed rows tops out near 20 bytes per
// clock and SM, which a one-CTA step of 64 KB all but needs), its loaders execute half the instructions, and per
// key tile and Q tile the tensor core reads 48 KB + 16 KB of a CTA's shared memory instead of 64 KB + 32 KB.
// What bounds a step (one key tile for both Q tiles; the products alone take 2050 cycles, the exponentials 2100): the chain
// S ready -> read by the softmax warps of both CTAs -> next QK^T, twice, which meets the second half of the PV products of
// the other Q tile; about 2750 cycles where P over S and one issuing thread took 3550.  2048 queries at 32K: sparse call 211
// -> 196 us, dense 1052 -> 952; 4096 at 128K 1245 -> 1140; paged mix of 8 sequences 950 -> 875.
//
// Roles per CTA as in the one-CTA kernel, except:
//   * only the first CTA's warps 10 and 11 issue MMAs.  A slot of its ring is ready when its own loaders AND the second
//     CTA's have filled it: the second CTA's warps 10 and 11 forward the "full" barriers of its V and K slots to a barrier
//     of the first CTA;
//   * completions (S ready, P multiplied, slot free, O final) are delivered to both CTAs' barriers by one multicast commit;
//   * the softmax warps of both CTAs announce "S read" and "P ready" on the first CTA's barriers;
//   * nobody leaves before a cluster barrier: the other CTA's MMAs read this one's shared and tensor memory.
// Tensor memory (512 columns per CTA): S | P_A | P_B | O_A | O_B.
// Ring slots are 16 KB: a K item holds [2 halves of d][64 keys][128 B], a V item [128 keys][128 B], both in the
// 128-byte-swizzled layout of the operand descriptors.
#include "attn_tiles.cuh"

namespace quoka {

constexpr int kPairSlots = 8;
constexpr int kPairLoaderWarps = kLoaderWarps;
constexpr uint32_t kPairSlotBytes = 16384;
constexpr uint32_t kPairQTileBytes = 32768;

enum { kWhole = 0, kParts = 1, kPartsCluster = 2 };     // a row block per pair; parts merged through memory / in a cluster

template <bool SPARSE, int MODE>
__device__ __forceinline__ void
attn_tc_pair_body(const DevParams& P, const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v,
                  const __nv_bfloat16* __restrict__ kc, const __nv_bfloat16* __restrict__ vc,
                  const int32_t* __restrict__ k_idx, const int32_t* __restrict__ k_cnt, __nv_bfloat16* __restrict__ out,
                  float* __restrict__ lse) {
  constexpr bool SPLIT = MODE != kWhole;
  constexpr int D = 128;
  constexpr uint32_t S_COL = 0, P_COL = 128, O_COL = 256;     // Q tile B's P and O are 64 and 128 columns on
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* q_smem = smem;                               // [2][2 halves][128][128 B]
  unsigned char* kv_smem = smem + 2 * kPairQTileBytes;        // [kPairSlots][16 KB]
  uint64_t* bars = reinterpret_cast<uint64_t*>(kv_smem + (size_t)kPairSlots * kPairSlotBytes);
  uint64_t* kv_full = bars;                       // [kPairSlots]  this CTA's loaders
  uint64_t* kv_empty = kv_full + kPairSlots;      // [kPairSlots]  MMA commit (both CTAs)
  uint64_t* peer_full = kv_empty + kPairSlots;    // [kPairSlots]  first CTA only: the second CTA's slot is full
  uint64_t* s_full = peer_full + kPairSlots;      // [2]           MMA commit (both CTAs)
  uint64_t* s_free = s_full + 2;                  //               first CTA only: S has been read, 4 softmax warps of each CTA
  uint64_t* p_full = s_free + 1;                  // [2][2]        first CTA only: 4 softmax warps of each CTA
  uint64_t* p_done = p_full + 4;                  // [2]           MMA commit (both CTAs): P has been multiplied
  uint64_t* o_full = p_done + 2;                  // [2]           MMA commit (both CTAs)
  uint64_t* q_full = o_full + 2;                  // this CTA's Q tiles (TMA)
  uint64_t* peer_q = q_full + 1;                  // first CTA only: the second CTA's Q tiles have landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(peer_q + 1);
  float* part_ml = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(bars) + 512);   // [2][m | l][128], kPartsCluster
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WaitCtx wc{&abort_flag, P.status};
  const uint32_t cta = cluster_cta_rank();
  const uint32_t rank = MODE == kPartsCluster ? cta & 1u : cta;   // 0: issues the MMAs, has the first positions
  const uint32_t first = MODE == kPartsCluster ? cta & ~1u : 0u;  // the pair's first CTA
  const int s = longest_first(P, blockIdx.z), hg = blockIdx.x >> 1;
  // grid.y = row blocks (heaviest first), times the parts a row block's key tiles are cut into (SPLIT)
  const int n_parts = SPLIT ? P.attn_parts : 1;
  const int rb = (SPLIT ? P.attn_split_rb : P.attn_row_blocks) - 1 - blockIdx.y / n_parts;
  const QRows qr(P, hg, rb, (int)rank, 2);
  const int kv = qr.head0 / P.group;
  AttnGeom g = make_geom<SPARSE>(P, s, rb * 2 * P.attn_qtiles * P.attn_span, 2);
  int t_lo = 0;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int i = 0; i < kPairSlots; ++i) {
      mbar_init(&kv_full[i], kPairLoaderWarps * 32);
      mbar_init(&kv_empty[i], 1);
      mbar_init(&peer_full[i], 1);
    }
    for (int i = 0; i < 2; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_done[i], 1); mbar_init(&o_full[i], 1); }
    for (int i = 0; i < 4; ++i) mbar_init(&p_full[i], 8);
    mbar_init(s_free, 8);
    mbar_init(q_full, 1);
    mbar_init(peer_q, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
  }
  if (warp == kQkWarp) tmem_alloc_pair(tmem_slot, 512);
  zero_spare_q_rows<D>(P, q_smem, threadIdx.x, kAttnThreads);
  tc_fence_before();
  cluster_sync_all();                                         // both CTAs' barriers exist before anyone signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint16_t both = MODE == kPartsCluster ? (uint16_t)(3u << first) : (uint16_t)3;   // this pair in the cluster
  const auto load_q = [&]() { load_q_tiles<D>(P, qr, q_smem, &tm_q, q_full, s); };
  // SPLIT: this CTA walks the tiles [t_lo, t_hi) of the row block's sequence only and leaves, per row, a partial
  // result (reference point, sum, un-normalised output); the part that finishes last, or the cluster, adds the
  // parts up.  The list length has to be known before the range is, so nothing of the walk starts before the selection has
  // ended.
  if (SPLIT) {
    if (warp == kQkWarp && lane == 0) load_q();
    if (SPARSE) { if (P.attn_after_whole) learn_count(g, k_cnt, s); else resolve(g, k_cnt, s); }
    const int part = blockIdx.y % n_parts;
    t_lo = (int)(((long long)part * g.n_known) / n_parts);
    g.n_known = (int)(((long long)(part + 1) * g.n_known) / n_parts);
  }

  if (!SPARSE && !SPLIT) grid_launch_dependents();

  if (warp < 8) {
    // ================================================================== softmax + epilogue
    const int x = warp >> 2;                                  // Q tile A (0) or B (1)
    const int quarter = warp & 3;
    const int row_in_tile = quarter * 32 + lane;
    const int row = qr.position(P, x, row_in_tile);           // chunk position
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t p_addr = lane_addr + P_COL + x * 64, o_addr = lane_addr + O_COL + x * D;
    const float scale_log2 = P.scale * 1.4426950408889634f;
    const uint32_t s_bar = map_to_cta(smem_u32(s_free), first);            // the first CTA's barriers
    const uint32_t p_bar = map_to_cta(smem_u32(&p_full[2 * x]), first);
    float m_run = -INFINITY, l_run = 0.f;
    uint32_t phase = 0;
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
      if (!mbar_wait(&s_full[x], phase, wc)) { ok = false; break; }
      tc_fence_after();
      ok = attn_softmax_tile<D, true>(
          lane_addr + S_COL, p_addr, o_addr, vis.lim, masked, scale_log2, t == skip_x, lane, m_run, l_run, [&]() { mbar_arrive_cluster(s_bar); },
          [&]() {
            if (!mbar_wait_done(&p_done[x], phase ^ 1, wc)) return false;
            tc_fence_after();
            return true;
          },
          []() { return true; }, [&](int half) { mbar_arrive_cluster(p_bar + 8u * half); });
      if (!ok) break;
      phase ^= 1;
    }
    // ---- epilogue: O / l -> bf16 -> global
    if constexpr (!SPLIT) {
      if (ok && active_x && mbar_wait(&o_full[x], 0, wc)) {
        tc_fence_after();
        attn_store_row<D>(P, o_addr, m_run, l_run, s, qr.head(P, row_in_tile), row, row_in_tile < qr.count(P, x), out, lse);
      }
    } else if constexpr (MODE == kPartsCluster) {
      // every product of the CTA has been formed when both are final: the ring and the Q tiles are free
      const bool other = x ? max(g.skip_a, t_lo) < g.n_known : g.active_b && t_lo < g.n_known;
      bool have = ok && active_x && mbar_wait(&o_full[x], 0, wc);
      if (have && other) have = mbar_wait(&o_full[x ^ 1], 0, wc);
      if (have) tc_fence_after();
      attn_part_to_smem<D>(smem, part_ml, x, row_in_tile, have, o_addr, m_run, l_run);
    } else {
      const bool have = ok && active_x && mbar_wait(&o_full[x], 0, wc);
      if (have) tc_fence_after();
      attn_split_epilogue<D>(P, ((s * QRows::groups(P) + hg) * P.attn_split_rb + rb) * 2 + (int)rank, blockIdx.y % n_parts, n_parts, x,
                             quarter, lane, row_in_tile, row, row_in_tile < qr.count(P, x), have, o_addr, m_run, l_run, s,
                             qr.head(P, row_in_tile), out, lse);
    }
  } else if (warp < 8 + kPairLoaderWarps) {
    // ================================================================== K / V loaders: this CTA's half of every tile
    // K item: tile rows [64 * rank, 64 * rank + 64), 256 bytes each (16 pieces, 2 rows per warp instruction).
    // V item: all 128 tile rows, bytes [128 * rank, 128 * rank + 128) of each (8 pieces, 4 rows per instruction).
    // Either way an item is 32 row groups, dealt round-robin to the loader warps.
    const int lw = warp - 8;
    constexpr int GROUPS = 32;
    constexpr int RPT = GROUPS / kPairLoaderWarps;             // row groups per warp
    const int kc16 = lane & 15, krsub = lane >> 4;
    const int vc16 = lane & 7, vrsub = lane >> 3;
    const int krow0 = (int)rank * 64;
    const int32_t* idx = SPARSE ? k_idx + ((long long)s * P.n_kv + kv) * P.budget_cap : nullptr;
    uint32_t phase = 0;
    int slot = 0;
    const uint32_t kv_base = smem_u32(kv_smem);
    // Row addressing in 16-byte units, 32 bits wide (the host refuses caches of 2^32 - 1 units and more; strides are
    // multiples of 8 elements): sequence/head base plus this thread's piece, row stride, page stride.
    const uint32_t st16 = (uint32_t)(P.kv_st >> 3), sb16 = (uint32_t)(P.kv_sb >> 3);
    const uint32_t head16 = (uint32_t)(((P.page_size == 0 ? (long long)s * P.kv_sb : 0ll) + (long long)kv * P.kv_sh) >> 3);
    const uint32_t kbase16 = head16 + (uint32_t)kc16, vbase16 = head16 + rank * 8u + (uint32_t)vc16;
    const int32_t* table = P.block_table + (long long)s * P.max_pages;
    // The warp's K rows of a tile are numbered p = 2 i + rsub (i = its i-th row group), its V rows p = 4 i + rsub; lane l
    // looks after K row p = l and V rows p = l, 32 + l: their row numbers (-1 past the end), for listed rows fetched one
    // tile ahead, and their offsets, worked out once per tile.  The thread that copies a row fetches its offset by shuffle.
    static_assert(kPairLoaderWarps == 2, "rows 4 apart from one K row group of a warp to the next, 8 for V");
    const int klr = lw * 2 + krsub, vlr = lw * 4 + vrsub;
    const uint32_t k_dst = (uint32_t)((kc16 >> 3) * 8192 + klr * 128 + (((kc16 & 7) ^ klr) << 4));
    const uint32_t v_dst = (uint32_t)(vlr * 128 + ((vc16 ^ vlr) << 4));
    int k_row = -1, v_row[2] = {-1, -1};
    uint32_t k_off = kNoRow, v_off[2] = {kNoRow, kNoRow};
    const int krr = krow0 + (lw + (lane >> 1) * kPairLoaderWarps) * 2 + (lane & 1);
    const int vrr = (lw + (lane >> 2) * kPairLoaderWarps) * 4 + (lane & 3);       // the second one is kVStep rows on
    constexpr int kVStep = 8 * kPairLoaderWarps * 4;
    static_assert(GROUPS % kPairLoaderWarps == 0 && RPT == 16, "a lane per K row, two V rows per lane");
    auto list_rows = [&](int base, int count) {
      const int last = min(count, kKeyTile) - 1;                   // last valid row of the tile
      if (last >= 0) {                                             // written by the kernel before: L2, not the read-only path
        const int vk = __ldcg(idx + base + min(krr, last));
        const int v0 = __ldcg(idx + base + min(vrr, last)), v1 = __ldcg(idx + base + min(vrr + kVStep, last));
        k_row = krr <= last ? vk : -1;
        v_row[0] = vrr <= last ? v0 : -1;
        v_row[1] = vrr + kVStep <= last ? v1 : -1;
      }
    };
    auto row_off = [&](int t, bool listed) -> uint32_t { return kv_row_off16(P, table, st16, sb16, t, listed, g.T); };
    // One ring item of tile `tr`: K (is_v = false) or V.  Returns false when a wait gave up.
    auto item = [&](auto is_v_c, const TileRows& tr, bool first_list_tile) -> bool {
      constexpr bool V = decltype(is_v_c)::value;
      constexpr int RPI = V ? 4 : 2;                            // rows per warp instruction
      if (!mbar_wait_done(&kv_empty[slot], phase ^ 1, wc)) return false;
      // A whole tile of consecutive rows (page-aligned in a paged cache) is fetched by the copy engine as two
      // 8 KB boxes: one thread issues them, the others only keep the barrier's arrival count.  Ragged tiles (rows
      // past the end must read as zeros) and listed rows take the copies below.
      if (!tr.from_list && tr.count >= kKeyTile && (P.page_size == 0 || (tr.first & (kPage - 1)) == 0)) {
        if (lw == 0 && lane == 0) {
          fence_proxy_async_smem();             // earlier contents of the slot were written through the generic proxy
          mbar_arrive_expect_tx(&kv_full[slot], kPairSlotBytes);
          unsigned char* dst = kv_smem + (size_t)slot * kPairSlotBytes;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            // K: box j = elements [64 j, 64 j + 64) of this CTA's 64 rows; V: box j = rows [64 j, 64 j + 64), this
            // CTA's 64 elements
            const int c0 = V ? (int)rank * 64 : j * 64;
            const int sub = V ? j : (int)rank;
            int c1 = tr.first + sub * 64, c3 = s;
            if (P.page_size != 0) { c1 = 0; c3 = __ldg(table + (tr.first >> 6) + sub); }
            tma_load_4d(dst + j * 8192, V ? &tm_v : &tm_k, &kv_full[slot], c0, c1, kv, c3);
          }
        } else {
          mbar_arrive(&kv_full[slot]);
        }
      } else {
        if (!V) {
          if (tr.from_list) {
            if (first_list_tile) list_rows(tr.first, tr.count);
          } else {
            k_row = krr < tr.count ? tr.first + krr : -1;
            v_row[0] = vrr < tr.count ? tr.first + vrr : -1;
            v_row[1] = vrr + kVStep < tr.count ? tr.first + vrr + kVStep : -1;
          }
          k_off = row_off(k_row, tr.from_list);
          v_off[0] = row_off(v_row[0], tr.from_list);
          v_off[1] = row_off(v_row[1], tr.from_list);
        }
        const uint4* src_base = reinterpret_cast<const uint4*>(V ? vc : kc) + (V ? vbase16 : kbase16);
        const uint32_t dst = kv_base + (uint32_t)slot * kPairSlotBytes + (V ? v_dst : k_dst);
        // row (lw + i * warps) * RPI + rsub of the item: its swizzle is the thread's own, turned by 4 rows for odd i (K)
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const uint32_t off = V ? __shfl_sync(0xFFFFFFFFu, v_off[i / 8], (i * 4 + vrsub) & 31) : __shfl_sync(0xFFFFFFFFu, k_off, i * 2 + krsub);
          cp_async_16((V || (i & 1) == 0 ? dst : dst ^ 64u) + (uint32_t)(i * kPairLoaderWarps * RPI * 128),
                      src_base + (off == kNoRow ? 0u : off), off != kNoRow);
        }
        // this thread's share of the slot is signalled by the copy engine itself when the bytes have landed
        cp_async_mbar_arrive_noinc(&kv_full[slot]);
        if (V && tr.from_list) list_rows(tr.first + kKeyTile, tr.count - kKeyTile);   // next list tile
      }
      if (++slot == kPairSlots) { slot = 0; phase ^= 1; }
      return true;
    };
    for (int tile = t_lo;; ++tile) {
      if (tile == g.n_known) {                                // end of what is known: the list length, or the end
        if (g.resolved) break;
        resolve(g, k_cnt, s);
        if (tile == g.n_known) break;
      }
      const TileRows tr = tile_rows<SPARSE>(g, tile);
      const bool first_list_tile = tr.from_list && tile == max(g.n_chunk, t_lo);
      if (!item(std::false_type{}, tr, first_list_tile)) break;
      if (!item(std::true_type{}, tr, first_list_tile)) break;
    }
    cp_async_wait_all();                                      // nothing of this thread is in flight at exit
  } else if (rank != 0) {
    // ================================================================== second CTA, one thread of warps 10 and 11: forward
    // the "full" of the V (10) and K (11) slots to the first CTA
    if (lane == 0) {
      bool ok = true;
      if (warp == kQkWarp) {
        if (!SPLIT) load_q();
        ok = mbar_wait(q_full, 0, wc);
        if (ok) mbar_arrive_cluster(map_to_cta(smem_u32(peer_q), first));
      }
      const uint32_t peer_full0 = map_to_cta(smem_u32(peer_full), first);
      RingCursor<kPairSlots> r(warp == kQkWarp ? 0 : 1);
      for (int tile = t_lo; ok; ++tile, r.advance()) {
        if (tile == g.n_known) {
          if (g.resolved) break;
          resolve(g, k_cnt, s);
          if (warp == kQkWarp) grid_launch_dependents();
          if (tile == g.n_known) break;
        }
        ok = mbar_wait(&kv_full[r.slot], r.phase, wc);
        if (!ok) break;
        fence_proxy_async_smem();             // the loaders' cp.async wrote through the generic proxy
        mbar_arrive_cluster(peer_full0 + (uint32_t)r.slot * 8u);
      }
    }
  } else {
    // ================================================================== first CTA, warps 10 and 11: issue the pair's products
    if (!SPLIT && warp == kQkWarp && lane == 0) load_q();
    __syncwarp();
    const bool leader = elect_one();
    const uint32_t tmem = (uint32_t)warp_uniform((int)tmem_base);
    t_lo = warp_uniform(t_lo);
    uniform_geom(g);
    // Descriptors are built once; a tile, slot or k-step offset is an addition to the 16-byte-unit address field.
    const uint64_t desc_kv = smem_desc_sw128(smem_u32(kv_smem), 16, 1024);
    const auto acquire = [&](int sl, uint32_t phase) {
      if (!warp_all(mbar_poll(&kv_full[sl], phase, wc) && mbar_poll(&peer_full[sl], phase, wc))) return false;
      fence_proxy_async_smem();               // cp.async wrote through the generic proxy, the MMA reads through the async one
      tc_fence_after();
      return true;
    };
    const auto release = [&](int sl) { if (leader) mma_pair_commit(both, &kv_empty[sl]); };
    if (warp == kQkWarp) {
      const uint32_t idesc_qk = idesc_bf16_f32(256, kKeyTile, false, false);
      const uint64_t desc_q = smem_desc_sw128(smem_u32(q_smem), 16, 1024);
      if (warp_all(mbar_poll(q_full, 0, wc) && mbar_poll(peer_q, 0, wc)))
        attn_issue_qk<1, kPairSlots>(
            g, t_lo, [&]() { resolve(g, k_cnt, s); uniform_geom(g); grid_launch_dependents(); }, acquire,
            [&](unsigned, uint32_t parity) {
              if (!warp_all(mbar_poll(s_free, parity, wc))) return false;
              tc_fence_after();
              return true;
            },
            [&](int x, unsigned, int ks) {
              const uint64_t da = desc_q + (uint64_t)(x * (kPairQTileBytes >> 4));
              const uint64_t db = desc_kv + (uint64_t)((uint32_t)ks * (kPairSlotBytes >> 4));
#pragma unroll
              for (int hh = 0; hh < 2; ++hh)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                  const uint64_t offa = (uint64_t)((hh * 16384 + kk * 32) >> 4);   // Q: halves of 128 rows
                  const uint64_t offb = (uint64_t)((hh * 8192 + kk * 32) >> 4);    // K: halves of 64 rows
                  if (leader) mma_pair_ss(tmem + S_COL, da + offa, db + offb, idesc_qk, (hh | kk) ? 1u : 0u);
                }
              if (leader) mma_pair_commit(both, &s_full[x]);
            },
            release);
    } else {
      const uint32_t idesc_pv = idesc_bf16_f32(256, D, false, true);
      uint32_t p_phase = 0;
      attn_issue_pv<1, kPairSlots>(
          g, t_lo, [&]() { resolve(g, k_cnt, s); uniform_geom(g); }, acquire,
          [&](int x, int half, unsigned, int vs, bool add) {
            if (!warp_all(mbar_poll(&p_full[2 * x + half], (p_phase >> x) & 1u, wc))) return false;
            tc_fence_after();
            const uint64_t dv = desc_kv + (uint64_t)((uint32_t)vs * (kPairSlotBytes >> 4) + half * 4 * (2048 >> 4));
            const uint32_t pa = tmem + P_COL + x * 64 + half * 32, oa = tmem + O_COL + x * D;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)             // 16 keys per MMA: 8 packed columns of P, 16 rows of V
              if (leader) mma_pair_ts(oa, pa + kk * 8, dv + (uint64_t)(kk * (2048 >> 4)), idesc_pv, add || kk ? 1u : 0u);
            if (half) {
              if (leader) mma_pair_commit(both, &p_done[x]);
              p_phase ^= 1u << x;
            }
            return true;
          },
          release, [&](int x) { if (leader) mma_pair_commit(both, &o_full[x]); });
    }
  }
  if (SPLIT && attn_last_cta()) grid_dependency_wait();       // this grid's end is the whole row blocks' end too
  tc_fence_before();
  if constexpr (MODE == kPartsCluster) {
    cluster_sync_all();                                       // every part's result is in its shared memory
    attn_merge_cluster<D>(P, smem, part_ml, warp, kAttnThreads / 32, lane, 2, (int)rank, n_parts, blockIdx.y % n_parts, qr, s, out, lse);
  }
  cluster_sync_all();                                         // the other CTA's MMAs no longer read this CTA
  if (warp == kQkWarp) tmem_dealloc_pair(tmem_base, 512);
}

#define QUOKA_PAIR_PARAMS                                                                                               \
  DevParams P, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,                      \
      const __grid_constant__ CUtensorMap tm_v, const __nv_bfloat16 *__restrict__ kc, const __nv_bfloat16 *__restrict__ vc, \
      const int32_t *__restrict__ k_idx, const int32_t *__restrict__ k_cnt, __nv_bfloat16 *__restrict__ out, float *__restrict__ lse
template <bool SPARSE, bool SPLIT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kAttnThreads, 1) attn_tc_pair_kernel(QUOKA_PAIR_PARAMS) {
  attn_tc_pair_body<SPARSE, SPLIT ? kParts : kWhole>(P, tm_q, tm_k, tm_v, kc, vc, k_idx, k_cnt, out, lse);
}
// clusters of (2, parts): the pairs of a row block's parts
template <bool SPARSE>
__global__ void __launch_bounds__(kAttnThreads, 1) attn_tc_pair_cluster_kernel(QUOKA_PAIR_PARAMS) {
  attn_tc_pair_body<SPARSE, kPartsCluster>(P, tm_q, tm_k, tm_v, kc, vc, k_idx, k_cnt, out, lse);
}

// ---------------------------------------------------------------------------------------------- host
quoka_status launch_attn_tc_pair(const quoka_params* p, const DevParams& P, const void* q, const void* k, const void* v,
                                 const int32_t* k_idx, const int32_t* k_cnt, void* out, float* lse, cudaStream_t st,
                                 bool after_selection, const AttnPlan& plan) {
  CUtensorMap tm_q;
  if (!encode_q_tensor_map(&tm_q, P, q)) return QUOKA_ERR_CUDA;
  CUtensorMap tm_k, tm_v;
  if (!encode_kv_tensor_map(&tm_k, p, k, 64) || !encode_kv_tensor_map(&tm_v, p, v, 64)) return QUOKA_ERR_CUDA;
  const size_t smem = 1024 + 2 * kPairQTileBytes + (size_t)kPairSlots * kPairSlotBytes + 512 + (plan.in_cluster ? 2048 : 0);
  const auto pick = [](bool sparse, bool parts, bool in_cluster) -> AttnKernel {
    if (parts && in_cluster) return sparse ? attn_tc_pair_cluster_kernel<true> : attn_tc_pair_cluster_kernel<false>;
    if (parts) return sparse ? attn_tc_pair_kernel<true, true> : attn_tc_pair_kernel<false, true>;
    return sparse ? attn_tc_pair_kernel<true, false> : attn_tc_pair_kernel<false, false>;
  };
  return launch_attn_plan(p, P, plan, pick, "attn_tc_pair", /*cluster=*/2, smem, tm_q, tm_k, tm_v, k, v, k_idx, k_cnt, out, lse, st, after_selection);
}

}  // namespace quoka
