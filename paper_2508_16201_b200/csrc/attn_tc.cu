// Streaming softmax attention over a bf16 K/V cache on the 5th-generation tensor cores of sm_100a:
// (gamma+1)-query verification attention and tree verification, windows of up to 128 rows per KV head
// (chains of up to 16 rows run on the kernel of attn.cu, wider windows on that of attn_pair.cu).
//
// One persistent CTA per SM streams a contiguous slice of the flat (layer, sequence, KV head, tile)
// list (attn_sched.h), so the cache is read exactly once, every SM moves the same number of bytes
// and only two partial results per CTA ever touch scratch memory (attn_merge_kernel folds them).  A tile is 128 tokens: two
// 64-token sub-tiles (one cache page each) as the TMA moves them.
//
// Roles inside a CTA (12 warps = 3 warpgroups; the first gives registers to the other two):
//   warp 0     TMA producer of the item's query rows and of the K tiles
//   warp 3     TMA producer of the V tiles.  K and V have rings of their own because a K tile is
//              free again as soon as S = Q K^T has been computed, long before its V tile; and
//              producers of their own because one thread cannot issue all copies of a tile
//              within the time HBM needs to deliver it.
//   warp 1     issues S = Q K^T (one thread, tcgen05.mma, accumulator in TMEM)
//   warp 2     issues O += P V (one thread)
//   warps 4-7  softmax group 0: the even tiles of the slice
//   warps 8-11 softmax group 1: the odd tiles.  Each group has its own S buffer, P buffer, running
//              (max, sum) and its own O accumulator; the two are merged once per item.
// 128-token tiles keep the two issuing threads, whose per-tile cost in barrier round trips is
// fixed, below the time HBM needs to deliver a tile.
// The GQA group's heads times the query tokens are the M rows of the tiles: M = 64 when they fit
// (row r lives in TMEM lane 32 (r / 16) + r % 16), else M = 128 (row r in lane r); a softmax warp
// owns the rows of its 32 TMEM lanes.
//
// The running maximum of a row is only raised when a tile's maximum exceeds it by more than 2^8; O
// is then rescaled in place in TMEM.  Probabilities stay below 2^8, well inside bf16 / fp32 range,
// and the common tile needs no pass over O at all.
#include "attn_tc.cuh"

namespace specvlm {

// Shared-memory plan.  A small region (barriers, flags, per-sequence tile counts, the softmax
// groups' row statistics) sits at the start of the dynamic shared memory; the tile rings and the
// operand tiles follow at the next 1024-byte boundary.
template <int D, int M>
struct TcCfg {
  static constexpr int SUB_BYTES = kTileTokens * D * 2;         // one 64-token K (or V) sub-tile
  static constexpr int NKP = D == 128 ? 2 : 3;                  // K ring: pair slots (128 tokens)
  static constexpr int NVP = D == 128 ? (M == 64 ? 3 : 2) : 3;  // V ring: pair slots
  static constexpr int NQ = (D == 128 && M == 128) ? 1 : 2;     // query buffers
  static constexpr int Q_BYTES = M * D * 2;                     // A operand of S = Q K^T
  static constexpr int P_BYTES = M * kBigTokens * 2;            // A operand of O += P V
  static constexpr int OFF_K = 0;
  static constexpr int OFF_V = OFF_K + NKP * 2 * SUB_BYTES;
  static constexpr int OFF_Q = OFF_V + NVP * 2 * SUB_BYTES;
  static constexpr int OFF_P = OFF_Q + NQ * Q_BYTES;
  static constexpr int BIG = OFF_P + 2 * P_BYTES;
  static constexpr int N_BARS = 2 * NKP + 2 * NVP + 15;
  static constexpr int SM_BAR = 0;
  static constexpr int SM_MISC = SM_BAR + 8 * N_BARS;
  static constexpr int SM_PLAN = SM_MISC + 16;
  static constexpr int SM_PREFIX = SM_PLAN + (kPlanBytes + 7) / 8 * 8;
  static constexpr int SM_STATS = SM_PREFIX + (kSchedMaxBatch + 1) * 4;     // [2 groups][M rows] float2
  static constexpr int SMALL_USED = SM_STATS + 2 * M * 8;
  static constexpr int SMALL = (SMALL_USED + 1023) / 1024 * 1024;
  static constexpr int kMaxSmem = 232448;                       // 227 KB
  // a spare KB for a base that is not 1024-byte aligned, where there is room for it
  static constexpr int TOTAL = SMALL + BIG + (SMALL + BIG + 1024 <= kMaxSmem ? 1024 : 0);
  static constexpr uint32_t COL_S = 0, COL_O = 2 * kBigTokens;  // TMEM: S of group g at 128 g, O at 256 + D g
  static constexpr uint32_t TMEM_COLS = 512;
  static_assert(SMALL + BIG <= kMaxSmem, "shared-memory plan does not fit");
};

// TREE: the window's visibility comes from per-token ancestor masks instead of the chain rule.
// A template parameter, not a run-time branch: the chain kernel's code is untouched by the tree
// variant (the softmax loop's speed proved sensitive to what is compiled around it).
template <int D, int M, bool TREE>
__global__ void __launch_bounds__(kTcThreads, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
               const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ AttnTcParams p) {
  using C = TcCfg<D, M>;
  constexpr int SUB_BYTES = C::SUB_BYTES, NKP = C::NKP, NVP = C::NVP, NQ = C::NQ;
  constexpr int Q_BYTES = C::Q_BYTES, P_BYTES = C::P_BYTES;
  constexpr int NH = M / 64;                          // 16-lane halves a softmax warp may own
  constexpr uint32_t kIdescQK = umma_idesc_bf16(M, kBigTokens, false, false);
  constexpr uint32_t kIdescPV = umma_idesc_bf16(M, D, false, true);   // V tile: channels run along the row

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t big = (raw_addr + C::SMALL_USED + 1023u) & ~1023u;
  uint8_t* const big_ptr = smem_raw + (big - raw_addr);
  const uint32_t k_sm = big + C::OFF_K, v_sm = big + C::OFF_V, q_sm = big + C::OFF_Q, p_sm = big + C::OFF_P;
  const uint32_t bar0 = raw_addr + C::SM_BAR;
  const uint32_t bar_k_full = bar0, bar_k_empty = bar_k_full + 8 * NKP;
  const uint32_t bar_v_full = bar_k_empty + 8 * NKP, bar_v_empty = bar_v_full + 8 * NVP;
  const uint32_t bar_q_full = bar_v_empty + 8 * NVP;   // [2]
  const uint32_t bar_q_empty = bar_q_full + 16;        // [2]
  const uint32_t bar_s_full = bar_q_empty + 16;        // [2]: one per softmax group
  const uint32_t bar_s_empty = bar_s_full + 16;        // [2]
  const uint32_t bar_p_full = bar_s_empty + 16;        // [2]
  const uint32_t bar_p_empty = bar_p_full + 16;        // [2]
  const uint32_t bar_o_full = bar_p_empty + 16;
  const uint32_t bar_o_empty = bar_o_full + 8;
  const uint32_t bar_ep_stats = bar_o_empty + 8;       // both groups' row statistics are in shared memory
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(smem_raw + C::SM_MISC);
  volatile uint32_t* const tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_raw + C::SM_MISC + 8);
  CtaSlice* const slice = reinterpret_cast<CtaSlice*>(smem_raw + C::SM_PLAN);
  int* const prefix = reinterpret_cast<int*>(smem_raw + C::SM_PREFIX);
  float2* const stats = reinterpret_cast<float2*>(smem_raw + C::SM_STATS);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // the plan needs the tiles inside the allocation (true whenever the base is 1024-byte aligned)
  if (big + C::BIG > raw_addr + C::TOTAL) {
    pdl_wait();
    if (tid == 0) {
      p.ws_cut[blockIdx.x] = make_int4(0, 0, 0, 0);
      if (p.d_status) *p.d_status = SPECVLM_ERR_CUDA;
    }
    return;
  }

  // ------------------------------------------------------------------ set-up
  // Everything up to griddepcontrol.wait touches no global memory and runs while the kernel before
  // this one drains; one barrier separates the set-up from the roles.
  if (tid == 0) {
    for (int s = 0; s < NKP; ++s) {
      mbar_init(bar_k_full + 8 * s, 1);
      mbar_init(bar_k_empty + 8 * s, 1);
    }
    for (int s = 0; s < NVP; ++s) {
      mbar_init(bar_v_full + 8 * s, 1);
      mbar_init(bar_v_empty + 8 * s, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_q_full + 8 * i, 1);
      mbar_init(bar_q_empty + 8 * i, 1);
      mbar_init(bar_s_full + 8 * i, 1);
      mbar_init(bar_s_empty + 8 * i, 4);
      mbar_init(bar_p_full + 8 * i, 4);
      mbar_init(bar_p_empty + 8 * i, 1);
    }
    mbar_init(bar_o_full, 1);
    mbar_init(bar_o_empty, 8);
    mbar_init(bar_ep_stats, 8);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc_launch_next(smem_u32(const_cast<uint32_t*>(tmem_slot)), C::TMEM_COLS);
  if (warp == 3 && lane == 0) {
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
    tma_prefetch_desc(&tm_q);
  }
  if (warp >= 4) {
    // query rows that no item uses stay zero (the TMA only ever writes the first p.rows rows of a
    // 64-channel block)
    const int n16 = (M - p.rows) * 8;
    for (int idx = tid - 128; idx < NQ * (D / 64) * n16; idx += kTcThreads - 128) {
      const int blk = idx / n16;
      *reinterpret_cast<uint4*>(big_ptr + C::OFF_Q + blk * (M * 128) + p.rows * 128 + (idx - blk * n16) * 16) =
          make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async();
  }
  pdl_wait();
  if (warp == 3) unwritten_parts(p, blockIdx.x, D, lane, 32);
  if (warp == 0) plan_slice<kBigTokens>(p, prefix, slice, blockIdx.x, gridDim.x, lane);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const int hkv = p.n_kv_heads;
  const int cta = blockIdx.x;
  const int rows = p.rows;                              // rows in use (of the M rows of a tile)
  const int64_t T0 = slice->begin, T1 = slice->end;
  const bool active = T0 < T1;
  const int n_items = p.n_layers * p.batch * hkv;
  const int n_my = (int)(T1 - T0);

  if (warp == 0 || warp == 3) {
    // ================================================================ TMA producers
    // warp 0: query rows + K tiles; warp 3: V tiles.  Both walk the same slice.
    setmaxnreg_dec<kRegsLight>();
    if (active) {
      const bool leader = elect_one();
      const bool is_k = warp == 0;
      const CUtensorMap* const tm = is_k ? &tm_k : &tm_v;
      const uint64_t policy = l2_policy_evict_first();
      const uint64_t policy_q = l2_policy_evict_last();
      const int subs_per_block = p.block_table ? p.block_tokens / kTileTokens : 1;
      const int n_ring = is_k ? NKP : NVP;
      const uint32_t ring_sm = is_k ? k_sm : v_sm, bar_full = is_k ? bar_k_full : bar_v_full;
      const uint32_t bar_empty = is_k ? bar_k_empty : bar_v_empty;
      // K tile: [64-channel block][128 tokens][128 B], the two sub-tiles stacked inside each block;
      // V tile: two sub-tiles of [64-channel block][64 tokens][128 B] one after the other
      const uint32_t blk_stride = is_k ? kBigTokens * 128 : kTileTokens * 128;
      const uint32_t sub_stride = is_k ? kTileTokens * 128 : SUB_BYTES;
      SliceCursor c;
      c.start(T0, T1, slice->first);
      bool ok = true;
      int i = 0;
      while (!c.done() && ok) {
        const Segment sg = c.sg;
        if (is_k) {
          // the item's query rows: a box of (64 channels) x (group heads) x (n_q tokens) per 64-channel block
          const int qb = c.seg_idx % NQ;
          if (c.seg_idx >= NQ) ok = warp_wait_soon(bar_q_empty + 8 * qb, ((c.seg_idx / NQ) - 1) & 1, abort_flag);
          if (!ok) break;
          if (leader) {
            mbar_arrive_expect_tx(bar_q_full + 8 * qb, (uint32_t)p.rows * 128u * (D / 64));
#pragma unroll
            for (int h = 0; h < D / 64; ++h)
              tma_load_5d(q_sm + qb * Q_BYTES + h * (M * 128), &tm_q, bar_q_full + 8 * qb, h * 64, 0, 0, sg.g,
                          sg.layer * p.batch + sg.b, policy_q);
          }
        }
        const int n_sub_seq = (clamp_len(p.seq_lens[sg.b], p.max_seq_len) + kTileTokens - 1) / kTileTokens;
        const int32_t* table = p.block_table ? p.block_table + (size_t)sg.b * p.max_blocks : nullptr;
        int blk[2], blk_next[2] = {sg.b, sg.b};
        if (table) {
          const int s0 = 2 * sg.tile0;
          blk_next[0] = __ldcg(table + s0 / subs_per_block);
          blk_next[1] = s0 + 1 < n_sub_seq ? __ldcg(table + (s0 + 1) / subs_per_block) : 0;
        }
        for (int j = 0; j < sg.n_tiles; ++j, ++i) {
          const int s0 = 2 * (sg.tile0 + j);                    // first sub-tile of this tile
          const int n_sub = n_sub_seq - s0 < 2 ? n_sub_seq - s0 : 2;
          blk[0] = blk_next[0];
          blk[1] = blk_next[1];
          if (table && j + 1 < sg.n_tiles) {                    // table entries of the next tile, one tile ahead
            blk_next[0] = __ldcg(table + (s0 + 2) / subs_per_block);
            blk_next[1] = s0 + 3 < n_sub_seq ? __ldcg(table + (s0 + 3) / subs_per_block) : 0;
          }
          const int slot = i % n_ring;
          if (i >= n_ring) ok = warp_wait_soon(bar_empty + 8 * slot, ((i / n_ring) - 1) & 1, abort_flag);
          if (!ok) break;
          if (leader) {
            mbar_arrive_expect_tx(bar_full + 8 * slot, n_sub * SUB_BYTES);
            for (int u = 0; u < n_sub; ++u) {
              const int tok = table ? ((s0 + u) % subs_per_block) * kTileTokens : (s0 + u) * kTileTokens;
#pragma unroll
              for (int h = 0; h < D / 64; ++h)
                tma_load_5d(ring_sm + slot * 2 * SUB_BYTES + h * blk_stride + u * sub_stride, tm, bar_full + 8 * slot,
                            h * 64, tok, sg.g, blk[u], sg.layer, policy);
            }
          }
        }
        if (ok) c.next_segment(prefix, p.batch, hkv);
      }
      if (!ok) {
        // a wait expired: report, then stay until this warp's copies in flight have landed (bounded)
        if (p.d_status && leader) *p.d_status = SPECVLM_ERR_TIMEOUT;
        const uint64_t t0 = global_timer_ns();
        for (int k = i > n_ring ? i - n_ring : 0; k < i; ++k)
          while (!mbar_test_wait(bar_full + 8 * (k % n_ring), (k / n_ring) & 1) && global_timer_ns() - t0 < kWaitLimitNs) {
          }
      }
    }
  } else if (warp == 1) {
    // ================================================================ S = Q K^T issuer
    setmaxnreg_dec<kRegsLight>();
    if (lane == 0) publish_cut_item(p, *slice, cta, cta, prefix);
    if (active) {
      const bool leader = elect_one();
      SliceCursor c;
      c.start(T0, T1, slice->first);
      const uint64_t dq0 = umma_desc_sw128(q_sm, 16, 1024), dk0 = umma_desc_sw128(k_sm, 16, 1024);
      bool ok = true;
      for (int i = 0; i < n_my; ++i) {
        const int g = i & 1, kp = i % NKP, qb = c.seg_idx % NQ;
        ok = mbar_wait_soon(bar_k_full + 8 * kp, (i / NKP) & 1, abort_flag);
        if (ok && c.j == 0) ok = mbar_wait_soon(bar_q_full + 8 * qb, (c.seg_idx / NQ) & 1, abort_flag);
        if (ok && i >= 2) ok = mbar_wait_soon(bar_s_empty + 8 * g, ((i >> 1) - 1) & 1, abort_flag);
        ok = warp_all(ok);
        if (!ok) break;
        tc_fence_after_sync();
        const uint64_t da = umma_desc_advance(dq0, qb * Q_BYTES), db = umma_desc_advance(dk0, kp * 2 * SUB_BYTES);
        const uint32_t d_tmem = tmem_base + C::COL_S + g * kBigTokens;
        if (leader) {
#pragma unroll
          for (int s = 0; s < D / 16; ++s)
            // 16 channels per step = 32 bytes along the swizzled 128-byte row; channels 64.. are the
            // second 64-channel block of each operand
            umma_bf16_ss(d_tmem, umma_desc_advance(da, (s >> 2) * (M * 128) + (s & 3) * 32),
                         umma_desc_advance(db, (s >> 2) * (kBigTokens * 128) + (s & 3) * 32), kIdescQK, s > 0 ? 1u : 0u);
          umma_commit(bar_s_full + 8 * g);
          umma_commit(bar_k_empty + 8 * kp);
          if (c.last_of_segment()) umma_commit(bar_q_empty + 8 * qb);
        }
        c.next_tile(prefix, p.batch, hkv);
      }
      if (!ok && p.d_status && leader) *p.d_status = SPECVLM_ERR_TIMEOUT;
    }
  } else if (warp == 2) {
    // ================================================================ O += P V issuer
    // The whole warp walks the slice; one lane issues.  The others lend a hand where a sequence ends inside a sub-tile: the V
    // rows past its end hold whatever the page held, and are cleared so that a zero probability times a stale non-finite
    // value cannot reach O.
    setmaxnreg_dec<kRegsLight>();
    if (active) {
      const bool leader = elect_one();
      SliceCursor c;
      c.start(T0, T1, slice->first);
      const uint64_t dp0 = umma_desc_sw128(p_sm, 16, 1024);
      const uint64_t dv0 = umma_desc_sw128(v_sm, kTileTokens * 128, 1024);   // 64-channel blocks 8 KB apart
      bool ok = true;
      int n_sub_seq = 0, kv_len = 0;
      for (int i = 0; i < n_my; ++i) {
        const int g = i & 1, vp = i % NVP;
        if (c.j == 0) {
          kv_len = clamp_len(p.seq_lens[c.sg.b], p.max_seq_len);
          n_sub_seq = (kv_len + kTileTokens - 1) / kTileTokens;
        }
        const int s0 = 2 * (c.sg.tile0 + c.j);
        const int n_sub = n_sub_seq - s0 < 2 ? n_sub_seq - s0 : 2;
        ok = warp_wait_soon(bar_v_full + 8 * vp, (i / NVP) & 1, abort_flag);
        if (!ok) break;
        if (s0 + n_sub == n_sub_seq && (kv_len & (kTileTokens - 1)) != 0) {
          uint8_t* vt = big_ptr + C::OFF_V + vp * 2 * SUB_BYTES + (n_sub - 1) * SUB_BYTES;
          const int first = kv_len - (n_sub_seq - 1) * kTileTokens;
          for (int idx = lane; idx < (kTileTokens - first) * (D / 8); idx += 32) {
            const int t = first + idx / (D / 8), c16 = idx % (D / 8);
            *reinterpret_cast<uint4*>(vt + (c16 >> 3) * (kTileTokens * 128) + t * 128 + (c16 & 7) * 16) =
                make_uint4(0, 0, 0, 0);
          }
          fence_proxy_async();
          __syncwarp();
        }
        // the first product of each group overwrites that group's O: the previous item must be out
        if (c.j < 2 && c.seg_idx >= 1) ok = warp_wait_soon(bar_o_empty, (c.seg_idx - 1) & 1, abort_flag);
        if (ok) ok = warp_wait_soon(bar_p_full + 8 * g, (i >> 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after_sync();
        if (leader) {
          const uint64_t da = umma_desc_advance(dp0, g * P_BYTES), db = umma_desc_advance(dv0, vp * 2 * SUB_BYTES);
          const uint32_t d_tmem = tmem_base + C::COL_O + g * D;
          const uint32_t acc0 = c.j >= 2 ? 1u : 0u;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (u < n_sub) {
#pragma unroll
              for (int kt = 0; kt < kTileTokens / 16; ++kt)
                // 16 tokens per step: 32 bytes along P's row, 16 rows of 128 bytes down the V sub-tile
                umma_bf16_ss(d_tmem, umma_desc_advance(da, u * (M * 128) + kt * 32),
                             umma_desc_advance(db, u * SUB_BYTES + kt * 2048), kIdescPV, (u > 0 || kt > 0) ? 1u : acc0);
            }
          }
          umma_commit(bar_p_empty + 8 * g);
          umma_commit(bar_v_empty + 8 * vp);
          if (c.last_of_segment()) umma_commit(bar_o_full);
        }
        c.next_tile(prefix, p.batch, hkv);
      }
      if (!ok && p.d_status && leader) *p.d_status = SPECVLM_ERR_TIMEOUT;
    }
  } else {
    // ================================================================ softmax / epilogue (warps 4..11)
    setmaxnreg_inc<kRegsSoftmax>();
    const int grp = (warp - 4) >> 2;              // tiles with (index & 1) == grp
    const int quarter = warp & 3;                 // TMEM lanes [32 * quarter, +32)
    const int gt = (warp & 3) * 32 + lane;        // 0..127 inside the group
    const int st = grp * 128 + gt;                // 0..255 over both groups
    const int lr = lane >> 2, lc = (lane & 3) * 2;   // row inside a 16-lane half (and +8), first column of a pair
    // rows of this warp: half h covers item rows row0(h) + [0, 16), held in TMEM lanes 32 * quarter + 16 h + [0, 16)
    auto row0 = [&](int h) { return M == 64 ? 16 * quarter : 32 * quarter + 16 * h; };
    const int nh = (rows > row0(0) ? 1 : 0) + (NH > 1 && rows > row0(1) ? 1 : 0);

    // sequences without any token: their outputs are zero, their LSE -inf
    if (slice->any_empty) {
      for (int item = cta; item < n_items; item += (int)gridDim.x) {
        const int lb = item / hkv, g = item - lb * hkv, b = lb % p.batch;
        if (prefix[b + 1] != prefix[b]) continue;
        if constexpr (TREE) check_tree(p.parents + (size_t)b * p.n_win, p.n_win, lane, p.d_status);
        for (int idx = st; idx < rows * (D / 8); idx += 256) {
          const int r = idx / (D / 8), c8 = idx - r * (D / 8);
          const int t = r / p.group, h = g * p.group + (r - t * p.group);
          const size_t orow = ((size_t)lb * p.n_win + t) * p.n_q_heads + h;
          *reinterpret_cast<uint4*>(p.out + orow * D + c8 * 8) = make_uint4(0, 0, 0, 0);
          if (p.lse && c8 == 0) p.lse[orow] = -INFINITY;
        }
      }
    }

    SliceCursor c;
    c.start(T0, T1, slice->first);
    bool ok = true;
    int i0 = 0;           // index (inside the slice) of the current segment's first tile
#define SM_WAIT(bar, parity)                                                        \
  do {                                                                              \
    ok = warp_wait_soon((bar), (parity), abort_flag);                                \
    if (!ok) goto softmax_done;                                                     \
  } while (0)

    while (!c.done()) {
      const Segment sg = c.sg;
      const int seg_idx = c.seg_idx;
      const int kv_len = clamp_len(p.seq_lens[sg.b], p.max_seq_len);
      // Visibility of key `tok` for a row of query token t: every key before the window of the n_q
      // new tokens, and inside the window the positions whose bit is set in the row's mask -- bits
      // 0..t for a chain, the token's ancestors and itself for a tree.  Rows no item uses see nothing.
      // (A used row always has its own bit set, so a zero mask also marks an unused row.)
      // The chain keeps the equivalent limit form: key tok is visible to token t when tok < lim.
      const int win0 = kv_len - p.n_win;
      float2* const seg_stats = stats;
      if constexpr (M == 128) {
        // ------------------------------------------------------------ 128-row windows: a thread owns a row
        // With M = 128 row r sits in TMEM lane r, so thread `lane` of the warp of quadrant q reads row
        // 32 q + lane whole (tcgen05.ld 32x32b): its maximum and sum need no shuffles, its 128
        // probabilities leave as sixteen 16-byte stores into the swizzled P tile, and the TMEM load of
        // the next 16 columns is in flight while the current 16 are worked on.
        const int my_row = 32 * quarter + lane;
        const bool warp_on = rows > 32 * quarter;         // warp-uniform: some row of this quadrant is in use
        uint64_t my_a;                                       // the row's window mask (tree) or key limit (chain)
        if constexpr (TREE) {
          const uint64_t a = tree_mask(p.parents + (size_t)sg.b * p.n_win, p.n_win, my_row < rows ? my_row / p.group : 0, p.d_status);
          my_a = my_row < rows ? a : 0ull;
        } else {
          my_a = my_row < rows ? (uint64_t)(win0 + my_row / p.group + 1) : 0ull;
        }
        float m_row = -INFINITY, l_row = 0.f;
        const uint32_t prow = p_sm + grp * P_BYTES + my_row * 128;
        const uint32_t psw = (uint32_t)(my_row & 7);

        for (int j = (i0 + grp) & 1; j < sg.n_tiles; j += 2) {
          const int i = i0 + j;
          const int tile_tok0 = (sg.tile0 + j) * kBigTokens;
          const bool need_mask = tile_tok0 + kBigTokens > win0 + (TREE ? 0 : 1);
          SM_WAIT(bar_s_full + 8 * grp, (i >> 1) & 1);
          tc_fence_after_sync();
          if (!warp_on) {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_s_empty + 8 * grp);
            if (i >= 2) SM_WAIT(bar_p_empty + 8 * grp, ((i >> 1) - 1) & 1);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p_full + 8 * grp);
            continue;
          }
          const uint32_t saddr = tmem_base + ((uint32_t)(32 * quarter) << 16) + C::COL_S + grp * kBigTokens;
          if (__builtin_expect(need_mask, 0)) {
            // the out-of-line mask routine works on 16-lane halves with two rows per thread
#pragma unroll 1
            for (int h = 0; h < nh; ++h) {
              const uint64_t a0 = __shfl_sync(0xffffffffu, my_a, 16 * h + lr);
              const uint64_t a1 = __shfl_sync(0xffffffffu, my_a, 16 * h + lr + 8);
              mask_s_half<TREE>(saddr + ((uint32_t)(16 * h) << 16), tile_tok0, win0, lc, a0, a1);
            }
          }
          uint32_t va[16], vb[16];
          // the group's previous product has completed: P may be overwritten, O may be rescaled
          if (i >= 2) SM_WAIT(bar_p_empty + 8 * grp, ((i >> 1) - 1) & 1);
          if (j < 2) {
            // The group's first tile of the item (O is overwritten by its product): the row's reference
            // maximum is the tile's own, found by a pass of its own over the 128 logits (raw products:
            // the scale is positive).
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            tmem_ld_x16(saddr, va);
#pragma unroll 1
            for (int cc = 0; cc < 4; ++cc) {
              tmem_ld_wait();
              tmem_ld_x16(saddr + 32 * cc + 16, vb);
#pragma unroll
              for (int k = 0; k < 16; ++k) mx4[k & 3] = fmaxf(mx4[k & 3], __uint_as_float(va[k]));
              tmem_ld_wait();
              if (cc < 3) tmem_ld_x16(saddr + 32 * cc + 32, va);
#pragma unroll
              for (int k = 0; k < 16; ++k) mx4[k & 3] = fmaxf(mx4[k & 3], __uint_as_float(vb[k]));
            }
            m_row = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * p.scale_log2;
          }
          // Every later tile takes ONE pass: p = 2^(s * scale - m) against the reference maximum the row
          // already has, the tile's own maximum being gathered on the way.  Only if that maximum turns
          // out more than the lazy-rescale threshold above the reference (a warp vote; rare after the
          // first tiles) is the reference raised, O rescaled in tensor memory and the pass repeated: S
          // stays in place until the decision is taken, and the probabilities of the abandoned pass are
          // simply overwritten (whatever they were, up to infinity, they never reach a product).
          // The pass is a rolled loop of four rounds of 32 logits, two TMEM loads of 16 columns each:
          // with 64 logits per round unrolled the code outgrew the instruction cache (the 9-token
          // window of 8 heads per KV head: 357 -> 336 us on 80 layers of 6400 tokens).
          float ps[2];
#pragma unroll 1
          for (int attempt = 0; attempt < 2; ++attempt) {
            const float nmu = m_row == -INFINITY ? 0.f : -m_row;   // a row that sees nothing yet stays at zero
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            ps[0] = ps[1] = 0.f;
            tmem_ld_x16(saddr, va);
#pragma unroll 1
            for (int cc = 0; cc < 4; ++cc) {     // 32 logits per round: four 16-byte chunks of the row
              const uint32_t pblk = prow + (cc >> 1) * (M * 128);
              const uint32_t ch0 = (uint32_t)(cc & 1) * 4;
              tmem_ld_wait();
              tmem_ld_x16(saddr + 32 * cc + 16, vb);
#pragma unroll
              for (int k4 = 0; k4 < 2; ++k4) {
                uint32_t w[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const float s0 = __uint_as_float(va[8 * k4 + 2 * u]), s1 = __uint_as_float(va[8 * k4 + 2 * u + 1]);
                  mx4[u] = fmaxf(mx4[u], fmaxf(s0, s1));
                  const float p0 = fast_exp2(fmaf(s0, p.scale_log2, nmu));
                  const float p1 = fast_exp2(fmaf(s1, p.scale_log2, nmu));
                  ps[u & 1] += p0 + p1;
                  w[u] = pack_bf16x2(p0, p1);
                }
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(pblk + (((ch0 + k4) ^ psw) << 4)),
                             "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
              }
              tmem_ld_wait();
              if (cc < 3) tmem_ld_x16(saddr + 32 * cc + 32, va);
#pragma unroll
              for (int k4 = 0; k4 < 2; ++k4) {
                uint32_t w[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const float s0 = __uint_as_float(vb[8 * k4 + 2 * u]), s1 = __uint_as_float(vb[8 * k4 + 2 * u + 1]);
                  mx4[u] = fmaxf(mx4[u], fmaxf(s0, s1));
                  const float p0 = fast_exp2(fmaf(s0, p.scale_log2, nmu));
                  const float p1 = fast_exp2(fmaf(s1, p.scale_log2, nmu));
                  ps[u & 1] += p0 + p1;
                  w[u] = pack_bf16x2(p0, p1);
                }
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(pblk + (((ch0 + 2 + k4) ^ psw) << 4)),
                             "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
              }
            }
            const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * p.scale_log2;
            const bool up = mx > m_row + kRescaleThreshold;
            if (__builtin_expect(__any_sync(0xffffffffu, up) == 0, 1)) break;
            // raise the reference maximum of those rows, rescale their sums and their O rows, go again
            const float a = up ? fast_exp2(m_row - mx) : 1.f;
            if (up) m_row = mx;
            l_row *= a;
            tc_fence_after_sync();
#pragma unroll 1
            for (int h = 0; h < nh; ++h) {
              const float f0 = __shfl_sync(0xffffffffu, a, 16 * h + lr);
              const float f1 = __shfl_sync(0xffffffffu, a, 16 * h + lr + 8);
              rescale_o_half<D>(tmem_base + ((uint32_t)(32 * quarter + 16 * h) << 16) + C::COL_O + grp * D, f0, f1);
            }
            tc_fence_before_sync();
          }
          tc_fence_before_sync();                // every read of the tile's logits is complete: S is free
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_s_empty + 8 * grp);
          l_row += ps[0] + ps[1];
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_p_full + 8 * grp);
        }
        // publish this group's row statistics for the merge below
        if (seg_idx >= 1) SM_WAIT(bar_o_empty, (seg_idx - 1) & 1);
        if (warp_on) seg_stats[grp * M + my_row] = make_float2(m_row, l_row);
      } else {
      uint64_t vis[NH][2];
      int lim[NH][2];
      float m_used[NH][2], l_sum[NH][2];
#pragma unroll
      for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int r = row0(h) + lr + 8 * e;
          const int t = r / p.group;
          if constexpr (TREE) {
            const uint64_t a = tree_mask(p.parents + (size_t)sg.b * p.n_win, p.n_win, r < rows ? t : 0, p.d_status);
            vis[h][e] = r < rows ? a : 0ull;
          } else {
            lim[h][e] = r < rows ? win0 + t + 1 : 0;
          }
          m_used[h][e] = -INFINITY;
          l_sum[h][e] = 0.f;
        }

      for (int j = (i0 + grp) & 1; j < sg.n_tiles; j += 2) {
        const int i = i0 + j;
        const int tile_tok0 = (sg.tile0 + j) * kBigTokens;
        const bool need_mask = tile_tok0 + kBigTokens > win0 + (TREE ? 0 : 1);
        SM_WAIT(bar_s_full + 8 * grp, (i >> 1) & 1);
        tc_fence_after_sync();
        if (nh == 0) {
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_s_empty + 8 * grp);
        }
        // (none where the window has no rows for this warp)
#pragma unroll 1
        for (int h = 0; h < nh; ++h) {
          // The warp's 16 rows x 128 columns are read from TMEM twice, 64 columns at a time, by the
          // same (rolled) code: once for the row maxima, once for the probabilities.  That halves
          // the live registers and the code of the loop; a TMEM load costs far less than the spills.
          const uint32_t saddr = tmem_base + ((uint32_t)(32 * quarter + 16 * h) << 16) + C::COL_S + grp * kBigTokens;
          if (__builtin_expect(need_mask, 0)) {
            if constexpr (TREE) mask_s_half<true>(saddr, tile_tok0, win0, lc, vis[0][0], vis[0][1]);
            else mask_s_half<false>(saddr, tile_tok0, win0, lc, (uint64_t)lim[0][0], (uint64_t)lim[0][1]);
          }
          float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            uint32_t v[32];
            tmem_ld_16x256b_x8(saddr + 64 * c, v);
            tmem_ld_wait();
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int k = 0; k < 32; ++k) mx[k & 3] = fmaxf(mx[k & 3], __uint_as_float(v[k]));
            mx0 = fmaxf(mx0, fmaxf(mx[0], mx[1]));
            mx1 = fmaxf(mx1, fmaxf(mx[2], mx[3]));
          }
          mx0 *= p.scale_log2;                                     // the scale is positive
          mx1 *= p.scale_log2;
          mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
          mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
          mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
          mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
          // the group's previous product has completed: P may be overwritten, O may be rescaled
          if (h == 0 && i >= 2) SM_WAIT(bar_p_empty + 8 * grp, ((i >> 1) - 1) & 1);
          if (j < 2) {
            // the group's first tile of the item: O is overwritten by this tile's product
            m_used[0][0] = mx0;
            m_used[0][1] = mx1;
          } else {
            const bool up0 = mx0 > m_used[0][0] + kRescaleThreshold, up1 = mx1 > m_used[0][1] + kRescaleThreshold;
            if (__builtin_expect(__any_sync(0xffffffffu, up0 || up1) != 0, 0)) {
              // raise the reference maximum of those rows and rescale their O rows in TMEM
              const float a0 = up0 ? fast_exp2(m_used[0][0] - mx0) : 1.f;
              const float a1 = up1 ? fast_exp2(m_used[0][1] - mx1) : 1.f;
              if (up0) m_used[0][0] = mx0;
              if (up1) m_used[0][1] = mx1;
              l_sum[0][0] *= a0;
              l_sum[0][1] *= a1;
              tc_fence_after_sync();
              rescale_o_half<D>(tmem_base + ((uint32_t)(32 * quarter + 16 * h) << 16) + C::COL_O + grp * D, a0, a1);
              tc_fence_before_sync();
            }
          }
          // probabilities: p = 2^(s * scale - m), with a row that sees nothing yet kept at zero
          const float nmu0 = m_used[0][0] == -INFINITY ? 0.f : -m_used[0][0];
          const float nmu1 = m_used[0][1] == -INFINITY ? 0.f : -m_used[0][1];
          float ps[4] = {0.f, 0.f, 0.f, 0.f};
          // rows of the A operand of O += P V: the item's rows
          const int m0 = row0(h) + lr, m1 = m0 + 8;
          const uint32_t prow0 = p_sm + grp * P_BYTES + m0 * 128 + lc * 2;
          const uint32_t prow1 = p_sm + grp * P_BYTES + m1 * 128 + lc * 2;
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {                            // the tile's two 64-token blocks
            uint32_t v[32];
            tmem_ld_16x256b_x8(saddr + 64 * c, v);
            tmem_ld_wait();
            if (c == 1 && h == nh - 1) {
              tc_fence_before_sync();
              __syncwarp();
              if (lane == 0) mbar_arrive(bar_s_empty + 8 * grp);
            }
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const float p0 = fast_exp2(fmaf(__uint_as_float(v[4 * jj]), p.scale_log2, nmu0));
              const float p1 = fast_exp2(fmaf(__uint_as_float(v[4 * jj + 1]), p.scale_log2, nmu0));
              const float p2 = fast_exp2(fmaf(__uint_as_float(v[4 * jj + 2]), p.scale_log2, nmu1));
              const float p3 = fast_exp2(fmaf(__uint_as_float(v[4 * jj + 3]), p.scale_log2, nmu1));
              ps[jj & 1] += p0 + p1;
              ps[2 + (jj & 1)] += p2 + p3;
              asm volatile("st.shared.b32 [%0], %1;" ::"r"(prow0 + c * (M * 128) + ((jj ^ (m0 & 7)) << 4)),
                           "r"(pack_bf16x2(p0, p1)) : "memory");
              asm volatile("st.shared.b32 [%0], %1;" ::"r"(prow1 + c * (M * 128) + ((jj ^ (m1 & 7)) << 4)),
                           "r"(pack_bf16x2(p2, p3)) : "memory");
            }
          }
          l_sum[0][0] += ps[0] + ps[1];
          l_sum[0][1] += ps[2] + ps[3];
        }
        if (nh == 0 && i >= 2) SM_WAIT(bar_p_empty + 8 * grp, ((i >> 1) - 1) & 1);
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_p_full + 8 * grp);
      }

        // publish this group's row statistics for the merge below.  A group may get here while the
        // other one still reads the previous segment's statistics: wait until both have left that
        // epilogue (the barrier the PV issuer waits on as well)
        if (seg_idx >= 1) SM_WAIT(bar_o_empty, (seg_idx - 1) & 1);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          if (h >= nh) break;
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float lt = l_sum[h][e];
            lt += __shfl_xor_sync(0xffffffffu, lt, 1);
            lt += __shfl_xor_sync(0xffffffffu, lt, 2);
            if ((lane & 3) == 0) seg_stats[grp * M + row0(h) + lr + 8 * e] = make_float2(m_used[h][e], lt);
          }
        }
      }

      // ---------------------------------------------------------------- end of the item's segment
      // merge the two groups' accumulators:
      //   O = (w0 O0 + w1 O1) / (w0 l0 + w1 l1),  w_g = 2^(m_g - max(m0, m1))
      const bool complete = sg.tile0 == 0 && sg.n_tiles == sg.item_tiles;
      const int lb = sg.layer * p.batch + sg.b;
      const int slot = partial_slot(cta, T0, sg.item_begin);
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_ep_stats);
      SM_WAIT(bar_ep_stats, seg_idx & 1);
      SM_WAIT(bar_o_full, seg_idx & 1);
      tc_fence_after_sync();
      // a group without a tile in this segment (one-tile segments) has nothing in its accumulator
      const bool has0 = sg.n_tiles >= 2 || (i0 & 1) == 0, has1 = sg.n_tiles >= 2 || (i0 & 1) == 1;
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        if (h >= nh) break;
        float w0[2], w1[2], lse2[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int ln = row0(h) + lr + 8 * e;
          const float2 s0 = seg_stats[ln], s1 = seg_stats[M + ln];
          const float l0 = has0 ? s0.y : 0.f, l1 = has1 ? s1.y : 0.f;
          const float ma = l0 > 0.f ? s0.x : -INFINITY, mb = l1 > 0.f ? s1.x : -INFINITY;
          const float mm = fmaxf(ma, mb);
          const float a = l0 > 0.f ? fast_exp2(ma - mm) : 0.f, b = l1 > 0.f ? fast_exp2(mb - mm) : 0.f;
          const float den = a * l0 + b * l1;
          const float inv = den > 0.f ? 1.f / den : 0.f;
          w0[e] = a * inv;
          w1[e] = b * inv;
          lse2[e] = den > 0.f ? mm + log2f(den) : -INFINITY;
        }
#pragma unroll
        for (int cc = 0; cc < D / 64; ++cc) {
          if ((cc & 1) != (D == 128 ? grp : 0)) continue;       // the groups share the column chunks
          if (D == 64 && grp == 1) continue;
          uint32_t oa[32], ob[32];
          const uint32_t oaddr = tmem_base + ((uint32_t)(32 * quarter + 16 * h) << 16) + C::COL_O + cc * 64;
          if (has0) tmem_ld_16x256b_x8(oaddr, oa);
          if (has1) tmem_ld_16x256b_x8(oaddr + D, ob);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int r = row0(h) + lr + 8 * e;
            if (r >= rows) continue;
            float res[16];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj)
#pragma unroll
              for (int x = 0; x < 2; ++x) {
                const int k = 4 * jj + 2 * e + x;
                float acc = 0.f;
                if (has0) acc = __uint_as_float(oa[k]) * w0[e];
                if (has1) acc += __uint_as_float(ob[k]) * w1[e];
                res[2 * jj + x] = acc;
              }
            if (complete) {
              const int t = r / p.group, hq = sg.g * p.group + (r - t * p.group);
              const size_t orow = ((size_t)lb * p.n_win + t) * p.n_q_heads + hq;
              __nv_bfloat16* dst = p.out + orow * D + cc * 64 + lc;
#pragma unroll
              for (int jj = 0; jj < 8; ++jj)
                *reinterpret_cast<uint32_t*>(dst + jj * 8) = pack_bf16x2(res[2 * jj], res[2 * jj + 1]);
              if (p.lse && cc == 0 && (lane & 3) == 0) p.lse[orow] = lse2[e] * kLn2;
            } else {
              float* dst = p.ws_o + ((size_t)slot * p.rows + r) * D + cc * 64 + lc;
#pragma unroll
              for (int jj = 0; jj < 8; ++jj)
                *reinterpret_cast<float2*>(dst + jj * 8) = make_float2(res[2 * jj], res[2 * jj + 1]);
              if ((lane & 3) == 0) p.ws_lse[(size_t)cc * p.lse_block + (size_t)slot * p.rows + r] = lse2[e];
            }
          }
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_o_empty);

      i0 += sg.n_tiles;
      c.next_segment(prefix, p.batch, hkv);
    }
  softmax_done:
    if (!ok && p.d_status && gt == 0) *p.d_status = SPECVLM_ERR_TIMEOUT;
#undef SM_WAIT
  }

  // every role ends here; the allocating warp returns the tensor memory
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------------------------
// Merge of the items that slice boundaries cut, a kernel of its own behind the attention kernel
// (launched with programmatic stream serialization).  A unit of work is a cut item and a block of its output
// positions (four channels of a row each).  The parts of an item sit in the scratch slots first_slot and
// 2 (c + 1), 2 (c + 2), ..
//   out = sum_s w_s o_s / sum_s w_s,  w_s = 2^(lse_s - max),  parts folded in slice order (fixed).
// A row with a part that was never written (its CTA gave up) is left alone.
// LANES warps share an item's parts: 1 where most items are cut in two, 4 where few items are cut into many parts.
// blockIdx.x = the CTA that holds an item's first part, blockIdx.y the block of positions; most CTAs of few items hold
// no first part, and their blocks leave.  Where that would take several rounds of blocks (TABLE) every block reads the
// whole table of cut items (2.4 KB), finds the valid entries by ballots and takes units in turn: one layer of 6400
// tokens launched 3552 blocks for 192 units, in eight rounds, and the merge took 6.4 of the call's 19.2 us; now 17.3
// (208 rows: 43.9 -> 31.2).  Elsewhere the table costs more than it saves (4 layers x 4 heads of 6400 tokens, one
// query row: 13.3 -> 14.5; 1 layer of 12 800: 13.6 -> 14.1).
// ---------------------------------------------------------------------------------------------
constexpr int kMergeThreads = 256;
constexpr int kMergeMaxCtas = 640;                       // entries of the table: CTAs of all sets (4 per SM at most)

template <int D, int LANES, bool TABLE>
__global__ void __launch_bounds__(kMergeThreads) attn_merge_kernel(const __grid_constant__ AttnTcParams p, int n_ctas) {
  // parts whose loads are in flight together: most cut items have two parts, and the registers of more would
  // keep blocks off the SMs (26-node tree under sustained load 677 -> 668 us, and 80-layer chain 359.5 -> 358.1); the
  // many parts of a few items are what LANES is for
  constexpr int kMergeChunk = LANES == 1 ? 2 : 8;
  constexpr int kPos = kMergeThreads / LANES;              // output positions of a unit
  constexpr int kRounds = (kMergeMaxCtas + kMergeThreads - 1) / kMergeThreads;
  __shared__ int4 cuts[TABLE ? kMergeMaxCtas : 1];
  __shared__ uint32_t valid[TABLE ? kRounds * (kMergeThreads / 32) : 1];
  __shared__ float4 acc_sm[LANES > 1 ? LANES - 1 : 1][kPos];
  __shared__ float2 md_sm[LANES > 1 ? LANES - 1 : 1][kPos];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wl = warp % LANES;                              // this warp's share of the parts: wl, wl + LANES, ..
  const int pos = (warp / LANES) * 32 + lane;
  pdl_launch_next();
  pdl_wait();
  int n_units = 0, chunks = 1;
  if constexpr (TABLE) {
    for (int r = 0, i = threadIdx.x; r * kMergeThreads < n_ctas; ++r, i += kMergeThreads) {
      const int4 c = i < n_ctas ? __ldcg(p.ws_cut + i) : make_int4(0, 0, 0, 0);
      if (i < n_ctas) cuts[i] = c;
      const uint32_t v = __ballot_sync(0xffffffffu, c.w != 0);
      if (lane == 0) valid[r * (kMergeThreads / 32) + warp] = v;
    }
    __syncthreads();
    for (int w = 0; w < (n_ctas + 31) / 32; ++w) n_units += __popc(valid[w]);
    chunks = (p.rows * (D / 4) + kPos - 1) / kPos;
    n_units *= chunks;
  }
  const int ctas_per_part = n_ctas / p.n_parts;
  for (int unit = blockIdx.x; !TABLE || unit < n_units; unit += gridDim.x) {
    int gcta, idx;
    int4 cut;
    if constexpr (!TABLE) {
      gcta = unit;
      cut = __ldcg(p.ws_cut + gcta);
      if (cut.w == 0) return;
      idx = blockIdx.y * kPos + pos;
    } else {
      int k_th = unit / chunks;
      idx = (unit - k_th * chunks) * kPos + pos;
      int word = 0;
      for (int n = __popc(valid[0]); k_th >= n; n = __popc(valid[++word])) k_th -= n;
      uint32_t bits = valid[word];
      for (; k_th > 0; --k_th) bits &= bits - 1;
      gcta = word * 32 + __ffs((int)bits) - 1;
      cut = cuts[gcta];
    }
    const int part = gcta / ctas_per_part, q0 = part * p.q_per;
    const int rows = (p.n_win - q0 < p.q_per ? p.n_win - q0 : p.q_per) * p.group;
    const bool on = idx < rows * (D / 4);
    const int r = on ? idx / (D / 4) : 0, c4 = on ? idx - r * (D / 4) : 0;
    float mm = -INFINITY, den = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    bool lost = false;
    for (int k0 = wl; k0 < cut.w; k0 += LANES * kMergeChunk) {
      float ls[kMergeChunk];
      float4 x[kMergeChunk];
#pragma unroll
      for (int q = 0; q < kMergeChunk; ++q) {
        const int k = k0 + q * LANES;
        ls[q] = -INFINITY;
        x[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (on && k < cut.w) {
          const size_t row = (size_t)(k == 0 ? cut.z : 2 * (gcta + k)) * p.rows + r;
          ls[q] = ldg_cg_f32(p.ws_lse + (size_t)(c4 >> 4) * p.lse_block + row);
          lost |= unwritten(ls[q]);
          x[q] = ldg_cg_f32x4(p.ws_o + row * D + c4 * 4);
        }
      }
      float m2 = mm;
#pragma unroll
      for (int q = 0; q < kMergeChunk; ++q) m2 = fmaxf(m2, ls[q]);
      if (m2 == -INFINITY) continue;
      const float sc = mm == -INFINITY ? 0.f : fast_exp2(mm - m2);
      acc.x *= sc;
      acc.y *= sc;
      acc.z *= sc;
      acc.w *= sc;
      den *= sc;
#pragma unroll
      for (int q = 0; q < kMergeChunk; ++q) {
        const float w = ls[q] == -INFINITY ? 0.f : fast_exp2(ls[q] - m2);
        acc.x += w * x[q].x;
        acc.y += w * x[q].y;
        acc.z += w * x[q].z;
        acc.w += w * x[q].w;
        den += w;
      }
      mm = m2;
    }
    if constexpr (LANES > 1) {
      if (wl > 0) {
        acc_sm[wl - 1][pos] = acc;
        md_sm[wl - 1][pos] = make_float2(lost ? __uint_as_float(kUnwritten) : mm, den);
      }
      __syncthreads();
      if (wl == 0) {
        float m2 = mm;
#pragma unroll
        for (int w = 0; w < LANES - 1; ++w) {
          lost |= unwritten(md_sm[w][pos].x);
          m2 = fmaxf(m2, md_sm[w][pos].x);
        }
        const float sc = mm == -INFINITY ? 0.f : fast_exp2(mm - m2);
        acc.x *= sc;
        acc.y *= sc;
        acc.z *= sc;
        acc.w *= sc;
        den *= sc;
#pragma unroll
        for (int w = 0; w < LANES - 1; ++w) {
          const float2 md = md_sm[w][pos];
          const float4 x = acc_sm[w][pos];
          const float f = md.x == -INFINITY ? 0.f : fast_exp2(md.x - m2);
          acc.x += f * x.x;
          acc.y += f * x.y;
          acc.z += f * x.z;
          acc.w += f * x.w;
          den += f * md.y;
        }
        mm = m2;
      }
      if (TABLE) __syncthreads();                           // the next unit's sums overwrite these
    }
    if (!TABLE && (wl > 0 || !on || lost)) return;
    if (wl > 0 || !on || lost) continue;
    const float inv = den > 0.f ? 1.f / den : 0.f;
    const int t = r / p.group, h = cut.y * p.group + (r - t * p.group);
    const size_t orow = ((size_t)cut.x * p.n_win + q0 + t) * p.n_q_heads + h;
    uint2 packed;
    packed.x = pack_bf16x2(acc.x * inv, acc.y * inv);
    packed.y = pack_bf16x2(acc.z * inv, acc.w * inv);
    *reinterpret_cast<uint2*>(p.out + orow * D + c4 * 4) = packed;
    if (p.lse && c4 == 0) p.lse[orow] = den > 0.f ? (mm + log2f(den)) * kLn2 : -INFINITY;
    if (!TABLE) return;
  }
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
// How a window of `rows` rows is cut: n_parts parts of q_per query tokens (at most 128 rows each).
static void tc_parts(int rows, int group, int& n_parts, int& q_per) {
  const int n_q = rows / group;
  const int q_max = 128 / group;                       // whole query tokens that fit the 128 rows of a part
  n_parts = (n_q + q_max - 1) / q_max;
  q_per = (n_q + n_parts - 1) / n_parts;               // the parts are made as equal as the tokens allow
}

// The most CTAs of a launch's set.  A window of one part is one set; a wider one has a set per two parts (attn_pair.cu),
// the sets side by side in one launch over the same slices, so that all but the first reader of a tile find it in the L2
// cache.
static int tc_ctas_max(int n_parts) {
  const int per_set = sm_count() / ((n_parts + 1) / 2);
  return per_set < 1 ? 1 : per_set;
}
static int64_t tc_tiles_max(const specvlm_kv_t* kv, int32_t batch) {
  return (int64_t)kv->n_layers * batch * kv->n_kv_heads * ((kv->max_seq_len + kBigTokens - 1) / kBigTokens);
}

// CTAs of a launch's set (as many as the SMs allow and the tile count is worth).
static int tc_set_ctas(const specvlm_kv_t* kv, int32_t batch, int n_parts) {
  const int per_set = tc_ctas_max(n_parts);
  const int even = sched_active_ctas(tc_tiles_max(kv, batch), per_set);
  // slices that keep to item boundaries may use more CTAs: every item rounds its own up
  const int64_t items = (int64_t)kv->n_layers * batch * kv->n_kv_heads;
  const int64_t aligned = items * sched_active_ctas((kv->max_seq_len + kBigTokens - 1) / kBigTokens, per_set);
  return aligned > even && items <= per_set ? (int)(aligned < per_set ? aligned : per_set) : even;
}

SlicePlan attn_tc_plan(const specvlm_kv_t* kv, int32_t batch, int32_t group, int32_t n_q) {
  SlicePlan pl;
  tc_parts(group * n_q, group, pl.n_parts, pl.q_per);
  pl.ctas = tc_set_ctas(kv, batch, pl.n_parts);
  return pl;
}

static SliceScratch tc_scratch(const specvlm_kv_t* kv, const SlicePlan& pl, int group) {
  return SliceScratch(pl.n_parts * pl.ctas, pl.q_per * group, kv->head_dim);
}

size_t attn_tc_ws_bytes(const specvlm_kv_t* kv, int32_t batch, int rows, int group) {
  SlicePlan pl;
  tc_parts(rows, group, pl.n_parts, pl.q_per);
  pl.ctas = sched_scratch_ctas(tc_tiles_max(kv, batch), tc_ctas_max(pl.n_parts));
  return tc_scratch(kv, pl, group).bytes();
}

// Queries as a 5-D tensor (channel, head in group, query token, KV head, layer * batch + sequence):
// the box (64 channels, group, n_q, 1, 1) at token q0 is one item's rows of a launch, r = t * group + head.
static int32_t encode_q_map(CUtensorMap* map, const void* q, int D, int group, int n_win, int n_q, int n_kv_heads,
                            int64_t lb) {
  encode_tiled_fn enc = get_encode_tiled();
  if (!enc) return SPECVLM_ERR_CUDA;
  const int hq = group * n_kv_heads;
  const cuuint64_t dims[5] = {(cuuint64_t)D, (cuuint64_t)group, (cuuint64_t)n_win, (cuuint64_t)n_kv_heads, (cuuint64_t)lb};
  const cuuint64_t strides[4] = {(cuuint64_t)D * 2, (cuuint64_t)hq * D * 2, (cuuint64_t)group * D * 2,
                                 (cuuint64_t)n_win * hq * D * 2};
  const cuuint32_t box[5] = {64u, (cuuint32_t)group, (cuuint32_t)n_q, 1u, 1u};
  const cuuint32_t estr[5] = {1u, 1u, 1u, 1u, 1u};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(q), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? SPECVLM_OK : SPECVLM_ERR_CUDA;
}

template <int D>
static int32_t launch_merge(const AttnTcParams& p, int ctas, cudaStream_t st) {
  if (ctas <= 1) return SPECVLM_OK;                       // no slice boundary: nothing is ever cut
  const int grid = p.n_parts * ctas;
  // Two parts per cut item where the items outnumber the CTAs; many where a few items fill the chip.
  const int64_t items = (int64_t)p.n_layers * p.batch * p.n_kv_heads;
  const int positions = p.rows * (D / 4);
  const int chunks1 = (positions + kMergeThreads - 1) / kMergeThreads, chunks4 = (4 * positions + kMergeThreads - 1) / kMergeThreads;
  if (ctas <= 4 * items)
    return launch_after(attn_merge_kernel<D, 1, false>, dim3((unsigned)grid, (unsigned)chunks1), dim3(kMergeThreads), 0, st, p, grid);
  const int64_t resident = 3 * sm_count();                // blocks that the chip holds at once
  if ((int64_t)grid * chunks4 <= 2 * resident || grid > kMergeMaxCtas)
    return launch_after(attn_merge_kernel<D, 4, false>, dim3((unsigned)grid, (unsigned)chunks4), dim3(kMergeThreads), 0, st, p, grid);
  const int64_t units = p.n_parts * items * chunks4;
  return launch_after(attn_merge_kernel<D, 4, true>, dim3((unsigned)(units < resident ? units : resident)), dim3(kMergeThreads), 0,
                      st, p, grid);
}

int32_t attn_merge_launch(const AttnTcParams& p, int head_dim, int ctas, cudaStream_t st) {
  return head_dim == 128 ? launch_merge<128>(p, ctas, st) : launch_merge<64>(p, ctas, st);
}

template <int D, int M>
static int32_t launch_tc(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const AttnTcParams& p,
                         int grid, cudaStream_t st) {
  constexpr int kSmem = TcCfg<D, M>::TOTAL;
  return p.parents ? launch_tc_kernel<attn_tc_kernel<D, M, true>>(kSmem, tk, tv, tq, p, grid, st)
               : launch_tc_kernel<attn_tc_kernel<D, M, false>>(kSmem, tk, tv, tq, p, grid, st);
}

// attn_pair.cu
int32_t attn_pair_launch(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const AttnTcParams& p,
                         int head_dim, int grid, cudaStream_t st);

int32_t attn_tc_launch(const specvlm_kv_t* kv, const void* q, int32_t batch, int32_t n_q_heads, int32_t n_q,
                       float sm_scale, void* out, float* lse, void* ws, size_t ws_bytes, int32_t* d_status,
                       cudaStream_t st, const int32_t* tree_parents) {
  const int group = n_q_heads / kv->n_kv_heads;
  const int rows = group * n_q;
  if (group > 16 || batch > kSchedMaxBatch) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  const int64_t items = (int64_t)kv->n_layers * batch * kv->n_kv_heads;
  if (items > 0x3fffffff) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return SPECVLM_ERR_INVALID_ARG;
  // A window of more than 128 rows is cut into parts of equal numbers of query tokens that share one launch.
  const SlicePlan pl = attn_tc_plan(kv, batch, group, n_q);
  const SliceScratch sc = tc_scratch(kv, pl, group);
  if (ws_bytes < attn_tc_ws_bytes(kv, batch, rows, group)) return SPECVLM_ERR_WORKSPACE_TOO_SMALL;
  if (tree_parents && n_q > kMaxTreeNodes) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  if (pl.q_per * group > 128) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  const int ctas = pl.ctas, n_parts = pl.n_parts;

  CUtensorMap tk, tv;
  int32_t rc = encode_kv_map(&tk, kv, kv->k, kTileTokens);
  if (rc != SPECVLM_OK) return rc;
  rc = encode_kv_map(&tv, kv, kv->v, kTileTokens);
  if (rc != SPECVLM_OK) return rc;

  AttnTcParams p = slice_params(kv, q, batch, n_q_heads, n_q, sm_scale, out, lse, d_status, n_parts, pl.q_per, ws, sc);
  p.parents = tree_parents;

  CUtensorMap tq;
  rc = encode_q_map(&tq, q, kv->head_dim, group, n_q, pl.q_per, kv->n_kv_heads, (int64_t)kv->n_layers * batch);
  if (rc != SPECVLM_OK) return rc;
  if (n_parts > 1)
    rc = attn_pair_launch(tk, tv, tq, p, kv->head_dim, (n_parts + 1) / 2 * ctas, st);
  else if (kv->head_dim == 128)
    rc = p.rows <= 64 ? launch_tc<128, 64>(tk, tv, tq, p, ctas, st) : launch_tc<128, 128>(tk, tv, tq, p, ctas, st);
  else
    rc = p.rows <= 64 ? launch_tc<64, 64>(tk, tv, tq, p, ctas, st) : launch_tc<64, 128>(tk, tv, tq, p, ctas, st);
  if (rc != SPECVLM_OK) return rc;
  return attn_merge_launch(p, kv->head_dim, ctas, st);
}

}  // namespace specvlm

// Host-only: how a verification window of n_q query tokens at `group` heads per KV head is cut into
// parts (see tc_parts); lets a CPU test sweep the rule.
extern "C" int32_t specvlm_debug_window_parts(int32_t n_q, int32_t group, int32_t* n_parts, int32_t* q_per) {
  if (n_q < 1 || group < 1 || group > 16 || !n_parts || !q_per) return SPECVLM_ERR_INVALID_ARG;
  int a, b;
  specvlm::tc_parts(n_q * group, group, a, b);
  *n_parts = a;
  *q_per = b;
  return SPECVLM_OK;
}
