// Verification windows of more than 128 rows per KV head (a 26-node draft tree at 8 heads per KV head has
// 208) on the 5th-generation tensor cores: one CTA works on TWO parts of the window, at most 128 rows
// each, over the same K/V tiles.
//
// As in attn_tc.cu a persistent CTA per SM streams a contiguous slice of the flat (layer, sequence, KV
// head, 128-token tile) list; a tile is loaded once and serves both parts.  Warps:
//   warp 0     TMA producer of the two parts' query rows and of the K tiles
//   warp 3     TMA producer of the V tiles
//   warps 1, 2 issue the products (one thread each) S_g = Q_g K^T and O_g += P_g V of part g = 0, 1
//   warps 4-7  softmax of part 0, every tile; warps 8-11 the same for part 1
// With M = 128 row r sits in TMEM lane r, so a softmax thread owns a row.  Its probabilities go back to tensor
// memory as bf16 over the logits they came from and are the A operand of P V from there: shared
// memory holds no P tile, which is what makes room for two query tiles next to the K and V rings.  A part's
// products come from one thread and run in issue order, so S_g of the next tile is issued right
// behind the P_g V that reads the same columns, and one commit tells the softmax both that its new
// logits are there and that its O is at rest.
//
// What bounds it: per tile and SM two parts cost 32 UMMAs of 64 cycles and 2 x 128 exponentials per
// thread, 2048 cycles each of the tensor pipe and of a scheduler's special-function unit, against about
// 2500 cycles in which HBM delivers the tile; a part's chain Q K^T -> softmax -> P V is serial (one S
// buffer per part fits the tensor memory), some 3700 cycles of which the two parts overlap.
//
// 26 nodes at 8 heads per KV head, 80 layers of 6400 tokens, cool / under sustained load at the power cap, in us:
//   a set of CTAs per part, each streaming K and V                                        642 / 827
//   two parts a CTA, in step (both softmaxes, then both waiting for the tensor pipe)      684
//   taking turns                                                                          610
//   the next S issued before the bookkeeping commits, waits that test before they
//   suspend, P handed over in two halves                                                  554 / 677
//   products issued by an elected lane of a whole warp instead of by lane 0 (of 4310
//   cycles a tile the issuers took 2750; then 3700)                                       548 / 648 (669 before, same box)
//   P handed over as 96 and 32 tokens                                                           643 (651)
// A share of the exponentials on the FMA pipe is slower (2 / 4 of 16 pairs: 571 / 604 against 554).
#include "attn_tc.cuh"

namespace specvlm {

template <int D>
struct PairCfg {
  static constexpr int M = 128;
  static constexpr int SUB_BYTES = kTileTokens * D * 2;         // one 64-token K (or V) sub-tile
  static constexpr int NKP = D == 128 ? 2 : 3;                  // K ring: pair slots (128 tokens)
  static constexpr int NVP = 3;                                 // V ring
  static constexpr int Q_BYTES = M * D * 2;                     // A operand of S = Q K^T, one part
  static constexpr int OFF_K = 0;
  static constexpr int OFF_V = OFF_K + NKP * 2 * SUB_BYTES;
  static constexpr int OFF_Q = OFF_V + NVP * 2 * SUB_BYTES;
  static constexpr int BIG = OFF_Q + 2 * Q_BYTES;
  static constexpr int N_BARS = 2 * NKP + 2 * NVP + 20;
  static constexpr int SM_MISC = 8 * N_BARS;
  static constexpr int SM_PLAN = SM_MISC + 16;
  static constexpr int SM_PREFIX = SM_PLAN + (kPlanBytes + 7) / 8 * 8;
  static constexpr int SMALL_USED = SM_PREFIX + (kSchedMaxBatch + 1) * 4;
  static constexpr int SMALL = (SMALL_USED + 1023) / 1024 * 1024;
  static constexpr int kMaxSmem = 232448;                       // 227 KB
  static constexpr int TOTAL = SMALL + BIG + (SMALL + BIG + 1024 <= kMaxSmem ? 1024 : 0);
  static constexpr uint32_t COL_S = 0, COL_O = 2 * kBigTokens;  // TMEM: S (and P) of part g at 128 g, O at 256 + D g
  static constexpr uint32_t TMEM_COLS = 512;
  static_assert(SMALL + BIG <= kMaxSmem, "shared-memory plan does not fit");
};

// D[tmem] (+)= A[tmem] * B[smem]: A = 128 rows of bf16 pairs, one row per lane
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// this warp's 32 lanes x 16 columns
__device__ __forceinline__ void tmem_st_x16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

template <int D, bool TREE>
__global__ void __launch_bounds__(kTcThreads, 1)
attn_pair_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                 const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ AttnTcParams p) {
  using C = PairCfg<D>;
  constexpr int M = C::M, SUB_BYTES = C::SUB_BYTES, NKP = C::NKP, NVP = C::NVP, Q_BYTES = C::Q_BYTES;
  constexpr uint32_t kIdescQK = umma_idesc_bf16(M, kBigTokens, false, false);
  constexpr uint32_t kIdescPV = umma_idesc_bf16(M, D, false, true);   // V tile: channels run along the row

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t big = (raw_addr + C::SMALL_USED + 1023u) & ~1023u;
  uint8_t* const big_ptr = smem_raw + (big - raw_addr);
  const uint32_t k_sm = big + C::OFF_K, v_sm = big + C::OFF_V, q_sm = big + C::OFF_Q;
  const uint32_t bar_k_full = raw_addr, bar_k_empty = bar_k_full + 8 * NKP;
  const uint32_t bar_v_full = bar_k_empty + 8 * NKP, bar_v_empty = bar_v_full + 8 * NVP;
  const uint32_t bar_q_full = bar_v_empty + 8 * NVP, bar_q_empty = bar_q_full + 8;
  const uint32_t bar_s_full = bar_q_empty + 8;         // [2]: one per part
  const uint32_t bar_p_most = bar_s_full + 16;         // [2]: the first 96 tokens' probabilities are in place
  const uint32_t bar_p_full = bar_p_most + 16;         // [2]: ... and the rest
  const uint32_t bar_o_full = bar_p_full + 16;         // [2]
  const uint32_t bar_o_empty = bar_o_full + 16;        // [2]
  const uint32_t bar_turn = bar_o_empty + 16;          // [2][4]: the turn of part g's warp of a TMEM lane quadrant
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(smem_raw + C::SM_MISC);
  volatile uint32_t* const tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_raw + C::SM_MISC + 8);
  CtaSlice* const slice = reinterpret_cast<CtaSlice*>(smem_raw + C::SM_PLAN);
  int* const prefix = reinterpret_cast<int*>(smem_raw + C::SM_PREFIX);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_sets = (p.n_parts + 1) / 2;              // a set of CTAs takes two parts (the last perhaps one)
  const int ctas = (int)gridDim.x / n_sets;
  const int set = blockIdx.x / ctas, cta = blockIdx.x - set * ctas;
  const int n_here = p.n_parts - 2 * set < 2 ? p.n_parts - 2 * set : 2;

  // the plan needs the tiles inside the allocation (true whenever the base is 1024-byte aligned)
  if (big + C::BIG > raw_addr + C::TOTAL) {
    pdl_wait();
    if (tid < n_here) {
      p.ws_cut[(2 * set + tid) * ctas + cta] = make_int4(0, 0, 0, 0);
      if (p.d_status) *p.d_status = SPECVLM_ERR_CUDA;
    }
    return;
  }

  // ------------------------------------------------------------------ set-up (see attn_tc.cu)
  if (tid == 0) {
    for (int s = 0; s < NKP; ++s) {
      mbar_init(bar_k_full + 8 * s, 1);
      mbar_init(bar_k_empty + 8 * s, n_here);
    }
    for (int s = 0; s < NVP; ++s) {
      mbar_init(bar_v_full + 8 * s, 1);
      mbar_init(bar_v_empty + 8 * s, n_here);
    }
    mbar_init(bar_q_full, 1);
    mbar_init(bar_q_empty, n_here);
    for (int g = 0; g < 2; ++g) {
      mbar_init(bar_s_full + 8 * g, 1);
      mbar_init(bar_p_most + 8 * g, 4);
      mbar_init(bar_p_full + 8 * g, 4);
      mbar_init(bar_o_full + 8 * g, 1);
      mbar_init(bar_o_empty + 8 * g, 4);
    }
    for (int k = 0; k < 8; ++k) mbar_init(bar_turn + 8 * k, 1);
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
    for (int idx = tid - 128; idx < 2 * (D / 64) * n16; idx += kTcThreads - 128) {
      const int blk = idx / n16;
      *reinterpret_cast<uint4*>(big_ptr + C::OFF_Q + blk * (M * 128) + p.rows * 128 + (idx - blk * n16) * 16) =
          make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async();
  }
  pdl_wait();
  if (warp >= 2 && warp - 2 < n_here) unwritten_parts(p, (2 * set + warp - 2) * ctas + cta, D, lane, 32);
  if (warp == 0) plan_slice<kBigTokens>(p, prefix, slice, cta, ctas, lane);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const int hkv = p.n_kv_heads;
  const int64_t T0 = slice->begin, T1 = slice->end;
  const bool active = T0 < T1;
  const int n_my = (int)(T1 - T0);

  if (warp == 0 || warp == 3) {
    // ================================================================ TMA producers
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
      int i = 0, n_q = 0;
      while (!c.done() && ok) {
        const Segment sg = c.sg;
        if (is_k) {
          // both parts' query rows: a box of (64 channels) x (group heads) x (q_per tokens) per 64-channel block
          if (c.seg_idx >= 1) ok = warp_wait_soon(bar_q_empty, (c.seg_idx - 1) & 1, abort_flag);
          if (!ok) break;
          if (leader) {
            mbar_arrive_expect_tx(bar_q_full, (uint32_t)(n_here * p.rows) * 128u * (D / 64));
            for (int g = 0; g < n_here; ++g)
#pragma unroll
              for (int h = 0; h < D / 64; ++h)
                tma_load_5d(q_sm + g * Q_BYTES + h * (M * 128), &tm_q, bar_q_full, h * 64, 0, (2 * set + g) * p.q_per, sg.g,
                            sg.layer * p.batch + sg.b, policy_q);
          }
          n_q = c.seg_idx + 1;
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
        while (n_q > 0 && !mbar_test_wait(bar_q_full, (n_q - 1) & 1) && global_timer_ns() - t0 < kWaitLimitNs) {
        }
      }
    }
  } else if (warp < 3) {
    // ================================================================ product issuers, a warp per part, one lane of which issues
    setmaxnreg_dec<kRegsLight>();
    const int g = warp - 1;
    if (g < n_here && lane == 0)
      publish_cut_item(p, *slice, cta, (2 * set + g) * ctas + cta, prefix);
    if (g < n_here && active) {
      const bool leader = elect_one();
      SliceCursor c;
      c.start(T0, T1, slice->first);
      const uint64_t dq = umma_desc_sw128(q_sm + g * Q_BYTES, 16, 1024), dk0 = umma_desc_sw128(k_sm, 16, 1024);
      const uint64_t dv0 = umma_desc_sw128(v_sm, kTileTokens * 128, 1024);   // 64-channel blocks 8 KB apart
      const uint32_t s_tmem = tmem_base + C::COL_S + g * kBigTokens, o_tmem = tmem_base + C::COL_O + g * D;
      bool ok = true;
      int n_sub_seq = 0, last_rows = 0;
      auto issue_qk = [&](int i) {                       // S of tile i
        const uint64_t db = umma_desc_advance(dk0, (i % NKP) * 2 * SUB_BYTES);
        if (!leader) return;
#pragma unroll
        for (int s = 0; s < D / 16; ++s)
          // 16 channels per step = 32 bytes along the swizzled 128-byte row; channels 64.. are the
          // second 64-channel block of each operand
          umma_bf16_ss(s_tmem, umma_desc_advance(dq, (s >> 2) * (M * 128) + (s & 3) * 32),
                       umma_desc_advance(db, (s >> 2) * (kBigTokens * 128) + (s & 3) * 32), kIdescQK, s > 0 ? 1u : 0u);
        umma_commit(bar_s_full + 8 * g);
      };
      ok = warp_all(mbar_wait_soon(bar_q_full, 0, abort_flag) && mbar_wait_soon(bar_k_full, 0, abort_flag));
      if (ok) {
        issue_qk(0);
        if (leader) {
          umma_commit(bar_k_empty);
          if (c.last_of_segment()) umma_commit(bar_q_empty);
        }
      }
      for (int i = 0; i < n_my && ok; ++i) {
        const int vp = i % NVP, seg_idx = c.seg_idx, j = c.j;
        const bool last = c.last_of_segment();
        if (j == 0) {
          const int kv_len = clamp_len(p.seq_lens[c.sg.b], p.max_seq_len);
          n_sub_seq = (kv_len + kTileTokens - 1) / kTileTokens;
          last_rows = kv_len - (n_sub_seq - 1) * kTileTokens;       // rows of the last sub-tile, 1 .. 64
        }
        const int s0 = 2 * (c.sg.tile0 + j);
        const int n_sub = n_sub_seq - s0 < 2 ? n_sub_seq - s0 : 2;
        const bool tail = s0 + n_sub == n_sub_seq;
        c.next_tile(prefix, p.batch, hkv);               // the cursor stands on tile i + 1 from here on
        const bool more = i + 1 < n_my;
        // waits that are over by the time P arrives come before the wait for P
        ok = warp_wait_soon(bar_v_full + 8 * vp, (i / NVP) & 1, abort_flag);
        if (ok && tail && (last_rows & 15) != 0) {
          // Steps of 16 tokens past the sequence's end are left out; inside the last step the V rows past
          // the end hold whatever the page held and are cleared (a zero probability times a stale
          // non-finite value must not reach O).  Both issuers do it: either may come first.
          uint8_t* const vt = big_ptr + C::OFF_V + vp * 2 * SUB_BYTES + (n_sub - 1) * SUB_BYTES;
          const int n_clear = (((last_rows + 15) & ~15) - last_rows) * (D / 8);
          for (int idx = lane; idx < n_clear; idx += 32) {
            const int t = last_rows + idx / (D / 8), c16 = idx % (D / 8);
            *reinterpret_cast<uint4*>(vt + (c16 >> 3) * (kTileTokens * 128) + t * 128 + (c16 & 7) * 16) =
                make_uint4(0, 0, 0, 0);
          }
          fence_proxy_async();
          __syncwarp();
        }
        if (ok && more) ok = warp_wait_soon(bar_k_full + 8 * ((i + 1) % NKP), ((i + 1) / NKP) & 1, abort_flag);
        // the first product of an item overwrites O: the previous item's must have been read
        if (ok && j == 0 && seg_idx >= 1) ok = warp_wait_soon(bar_o_empty + 8 * g, (seg_idx - 1) & 1, abort_flag);
        const uint64_t db = umma_desc_advance(dv0, vp * 2 * SUB_BYTES);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (ok) ok = warp_wait_soon((u ? bar_p_full : bar_p_most) + 8 * g, i & 1, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
          // 16 tokens per step: 8 columns of bf16 pairs of P, 16 rows of 128 bytes down the V sub-tile; the tile's first
          // 96 tokens, then the other 32
          const int n_kt = 4 * (n_sub - 1) + (tail ? (last_rows + 15) >> 4 : kTileTokens / 16);
#pragma unroll
          for (int kt = u ? 6 : 0; kt < (u ? 8 : 6); ++kt)
            if (leader && kt < n_kt)
              umma_bf16_ts(o_tmem, s_tmem + kt * 8, umma_desc_advance(db, (kt >> 2) * SUB_BYTES + (kt & 3) * 2048), kIdescPV,
                           kt > 0 || j > 0 ? 1u : 0u);
        }
        if (!ok) break;
        // S of the next tile first: the softmax is waiting for it
        if (more && !last) issue_qk(i + 1);
        if (leader) {
          if (last) umma_commit(bar_o_full + 8 * g);
          umma_commit(bar_v_empty + 8 * vp);
        }
        if (more) {
          if (last) {
            ok = warp_wait_soon(bar_q_full, (seg_idx + 1) & 1, abort_flag);
            if (!ok) break;
            issue_qk(i + 1);
          }
          if (leader) {
            umma_commit(bar_k_empty + 8 * ((i + 1) % NKP));
            if (c.last_of_segment()) umma_commit(bar_q_empty);
          }
        }
      }
      if (!ok && p.d_status && leader) *p.d_status = SPECVLM_ERR_TIMEOUT;
    }
  } else {
    // ================================================================ softmax / epilogue (warps 4..11)
    setmaxnreg_inc<kRegsSoftmax>();
    const int g = (warp - 4) >> 2;                // the part of this group
    const int quarter = warp & 3;                 // TMEM lanes [32 * quarter, +32)
    const int my_row = 32 * quarter + lane;
    const int lr = lane >> 2, lc = (lane & 3) * 2;   // the mask and rescale routines' rows and columns of a 16-lane half
    const int part = 2 * set + g;
    const int q0 = part * p.q_per;                // first window token of the part
    const int n_q_part = g < n_here ? (p.n_win - q0 < p.q_per ? p.n_win - q0 : p.q_per) : 0;
    const int rows = n_q_part * p.group;          // rows in use (of the 128 of a tile)
    const bool warp_on = rows > 32 * quarter;     // warp-uniform: some row of this quadrant is in use
    const int nh = rows > 32 * quarter + 16 ? 2 : (warp_on ? 1 : 0);
    const bool row_on = my_row < rows;
    const int my_t = row_on ? my_row / p.group : 0;
    const uint32_t lane_base = tmem_base + ((uint32_t)(32 * quarter) << 16);
    const uint32_t saddr = lane_base + C::COL_S + g * kBigTokens, oaddr = lane_base + C::COL_O + g * D;

    // sequences without any token: their outputs are zero, their LSE -inf
    if (slice->any_empty && rows > 0) {
      const int n_items = p.n_layers * p.batch * hkv;
      for (int item = cta; item < n_items; item += ctas) {
        const int lb = item / hkv, kvh = item - lb * hkv, b = lb % p.batch;
        if (prefix[b + 1] != prefix[b]) continue;
        if constexpr (TREE) check_tree(p.parents + (size_t)b * p.n_win, p.n_win, lane, p.d_status);
        for (int idx = my_row; idx < rows * (D / 8); idx += 128) {
          const int r = idx / (D / 8), c8 = idx - r * (D / 8);
          const int t = r / p.group, h = kvh * p.group + (r - t * p.group);
          const size_t orow = ((size_t)lb * p.n_win + q0 + t) * p.n_q_heads + h;
          *reinterpret_cast<uint4*>(p.out + orow * D + c8 * 8) = make_uint4(0, 0, 0, 0);
          if (p.lse && c8 == 0) p.lse[orow] = -INFINITY;
        }
      }
    }

    SliceCursor c;
    if (rows > 0) c.start(T0, T1, slice->first);
    else c.start(0, 0, slice->first);     // no second part here: the group has nothing to do
    bool ok = true;
    int i = 0;
#define SM_WAIT(bar, parity)                                                        \
  do {                                                                              \
    ok = warp_wait_soon((bar), (parity), abort_flag);                                \
    if (!ok) goto softmax_done;                                                     \
  } while (0)
    // The two parts' warps of a lane quadrant sit on the same scheduler and take turns with its
    // special-function unit: left alone, both parts drift into step -- both softmaxes at half speed,
    // then both waiting for the tensor pipe.
    const uint32_t my_turn = bar_turn + 8 * (4 * g + quarter), other_turn = bar_turn + 8 * (4 * (1 - g) + quarter);
    const bool turns = n_here == 2;
    auto take_turn = [&](int n) {               // part 0 goes first: its n-th turn follows part 1's (n - 1)-th
      if (turns && (g == 1 || n > 0)) ok = warp_wait_soon(my_turn, (g == 1 ? n : n - 1) & 1, abort_flag);
    };
    auto pass_turn = [&]() {
      __syncwarp();
      if (turns && lane == 0) mbar_arrive(other_turn);
    };
    while (!c.done()) {
      const Segment sg = c.sg;
      const int seg_idx = c.seg_idx;
      const int kv_len = clamp_len(p.seq_lens[sg.b], p.max_seq_len);
      // visibility inside the window: the row's ancestor mask (tree) or key limit (chain); see mask_s_half
      const int win0 = kv_len - p.n_win;
      uint64_t my_a;
      if constexpr (TREE) {
        const uint64_t a = tree_mask(p.parents + (size_t)sg.b * p.n_win, p.n_win, row_on ? q0 + my_t : 0, p.d_status);
        my_a = row_on ? a : 0ull;
      } else {
        my_a = row_on ? (uint64_t)(win0 + q0 + my_t + 1) : 0ull;
      }
      float m_row = -INFINITY, l_row = 0.f;
      for (int j = 0; j < sg.n_tiles; ++j, ++i) {
        const int tile_tok0 = (sg.tile0 + j) * kBigTokens;
        const bool need_mask = tile_tok0 + kBigTokens > win0 + (TREE ? 0 : 1);
        SM_WAIT(bar_s_full + 8 * g, i & 1);
        tc_fence_after_sync();
        if (!warp_on) {
          take_turn(i);
          if (!ok) goto softmax_done;
          pass_turn();
          // no row of the window here: whatever S holds (zeros, or NaN from K rows past a sequence's end) may stand as P,
          // since rows of a product do not mix and nobody reads these
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(bar_p_most + 8 * g);
            mbar_arrive(bar_p_full + 8 * g);
          }
          continue;
        }
        if (__builtin_expect(need_mask, 0)) {
#pragma unroll 1
          for (int h = 0; h < nh; ++h) {
            const uint64_t a0 = __shfl_sync(0xffffffffu, my_a, 16 * h + lr);
            const uint64_t a1 = __shfl_sync(0xffffffffu, my_a, 16 * h + lr + 8);
            mask_s_half<TREE>(saddr + ((uint32_t)(16 * h) << 16), tile_tok0, win0, lc, a0, a1);
          }
        }
        // the row's 128 logits stay in registers from here on
        uint32_t v[4][32];
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) tmem_ld_x32(saddr + 32 * cc, v[cc]);
        tmem_ld_wait();
        // the tile's maximum (of the raw products: the scale is positive)
        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
#pragma unroll
          for (int k = 0; k < 32; k += 2)
            mx4[cc] = max3(mx4[cc], __uint_as_float(v[cc][k]), __uint_as_float(v[cc][k + 1]));
        const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * p.scale_log2;
        if (j == 0) {
          m_row = mx;                              // O is overwritten by this tile's product
        } else {
          const bool up = mx > m_row + kRescaleThreshold;
          if (__builtin_expect(__any_sync(0xffffffffu, up) != 0, 0)) {
            // raise the reference maximum of those rows, rescale their sums and their O rows
            const float a = up ? fast_exp2(m_row - mx) : 1.f;
            if (up) m_row = mx;
            l_row *= a;
#pragma unroll 1
            for (int h = 0; h < nh; ++h) {
              const float f0 = __shfl_sync(0xffffffffu, a, 16 * h + lr);
              const float f1 = __shfl_sync(0xffffffffu, a, 16 * h + lr + 8);
              rescale_o_half<D>(oaddr + ((uint32_t)(16 * h) << 16), f0, f1);
            }
          }
        }
        take_turn(i);
        if (!ok) goto softmax_done;
        // p = 2^(s * scale - m), a row that sees nothing yet kept at zero; P's bf16 pairs overwrite S
        const float nmu = m_row == -INFINITY ? 0.f : -m_row;
        const uint64_t sc2 = f2_pack(p.scale_log2, p.scale_log2), nmu2 = f2_pack(nmu, nmu);
        uint64_t ps2[2] = {0ull, 0ull};
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          uint32_t w[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const uint64_t t2 = f2_fma(f2_pack(__uint_as_float(v[cc][2 * u]), __uint_as_float(v[cc][2 * u + 1])), sc2, nmu2);
            const uint64_t e2 = f2_exp2_sfu(t2);
            ps2[u & 1] = f2_add(ps2[u & 1], e2);
            float e0, e1;
            f2_unpack(e2, e0, e1);
            w[u] = pack_bf16x2(e0, e1);
          }
          tmem_st_x16(saddr + 16 * cc, w);
          if (cc == 2) {
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p_most + 8 * g);
          }
        }
        pass_turn();
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_p_full + 8 * g);
        {
          float s0, s1, s2, s3;
          f2_unpack(ps2[0], s0, s1);
          f2_unpack(ps2[1], s2, s3);
          l_row += (s0 + s1) + (s2 + s3);
        }
      }

      // ---------------------------------------------------------------- end of the item's segment
      const bool complete = sg.tile0 == 0 && sg.n_tiles == sg.item_tiles;
      const int lb = sg.layer * p.batch + sg.b;
      SM_WAIT(bar_o_full + 8 * g, seg_idx & 1);
      tc_fence_after_sync();
      if (warp_on) {
        const float inv = l_row > 0.f ? 1.f / l_row : 0.f;
        const float lse2 = l_row > 0.f ? m_row + log2f(l_row) : -INFINITY;
        const size_t orow = ((size_t)lb * p.n_win + q0 + my_t) * p.n_q_heads + sg.g * p.group + (my_row - my_t * p.group);
        const size_t prow = (size_t)partial_slot((part * ctas) + cta, T0, sg.item_begin) * p.rows + my_row;
#pragma unroll 1
        for (int cc = 0; cc < D / 32; ++cc) {
          uint32_t o[32];
          tmem_ld_x32(oaddr + 32 * cc, o);
          tmem_ld_wait();
          if (!row_on) continue;
          if (complete) {
            uint4* const dst = reinterpret_cast<uint4*>(p.out + orow * D + 32 * cc);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              uint32_t w[4];
#pragma unroll
              for (int u = 0; u < 4; ++u)
                w[u] = pack_bf16x2(__uint_as_float(o[8 * k + 2 * u]) * inv, __uint_as_float(o[8 * k + 2 * u + 1]) * inv);
              dst[k] = make_uint4(w[0], w[1], w[2], w[3]);
            }
          } else {
            float4* const dst = reinterpret_cast<float4*>(p.ws_o + prow * D + 32 * cc);
#pragma unroll
            for (int k = 0; k < 8; ++k)
              dst[k] = make_float4(__uint_as_float(o[4 * k]) * inv, __uint_as_float(o[4 * k + 1]) * inv,
                                   __uint_as_float(o[4 * k + 2]) * inv, __uint_as_float(o[4 * k + 3]) * inv);
          }
        }
        if (row_on) {
          if (!complete) {
#pragma unroll
            for (int b = 0; b < D / 64; ++b) p.ws_lse[(size_t)b * p.lse_block + prow] = lse2;
          }
          else if (p.lse) p.lse[orow] = lse2 * kLn2;
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_o_empty + 8 * g);
      c.next_segment(prefix, p.batch, hkv);
    }
  softmax_done:
    if (!ok && p.d_status && my_row == 0) *p.d_status = SPECVLM_ERR_TIMEOUT;
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

template <int D, bool TREE>
static int32_t launch_pair_t(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const AttnTcParams& p,
                             int grid, cudaStream_t st) {
  return launch_tc_kernel<attn_pair_kernel<D, TREE>>(PairCfg<D>::TOTAL, tk, tv, tq, p, grid, st);
}

int32_t attn_pair_launch(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const AttnTcParams& p,
                         int head_dim, int grid, cudaStream_t st) {
  if (head_dim == 128)
    return p.parents ? launch_pair_t<128, true>(tk, tv, tq, p, grid, st) : launch_pair_t<128, false>(tk, tv, tq, p, grid, st);
  return p.parents ? launch_pair_t<64, true>(tk, tv, tq, p, grid, st) : launch_pair_t<64, false>(tk, tv, tq, p, grid, st);
}

}  // namespace specvlm
