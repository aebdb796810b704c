// Attention entry points (draft decode and verification) and the kernels for up to 16 query rows
// per KV head, i.e. draft decode: the GQA group's heads of one query token.
//
// With so few rows the step is a pure K/V stream (3.5 flop per cache byte at group 7): 64-token K
// and V tiles go HBM -> shared memory by 128-byte-swizzled tensor-map bulk copies
// (cp.async.bulk.tensor) through an mbarrier ring, four warps each score 16 tokens of a tile on
// m16n8k16 bf16 tiles with a private online softmax, and are merged once per item, i.e. per (layer, sequence, KV
// head).  An item has a CTA of its own where that is the fastest; else the CTAs work on slices of the list
// of all tiles.  Windows of more than 16 rows (verification) run on the tcgen05 kernels.
#include "attn_tc.cuh"

namespace specvlm {

// ---------------------------------------------------------------------------------------------
// One consumer warp's share of an item: 16 of a tile's 64 tokens, with a private running (max, sum, O).
// ---------------------------------------------------------------------------------------------
template <int D>
struct Rows16 {
  static constexpr int KSTEPS = D / 16;
  static constexpr int NT_O = D / 8;
  static constexpr int OPITCH = D + 8;            // fp32 pitch of the merge buffer
  uint32_t qf[KSTEPS][4];
  float o[NT_O][4];
  float m0, m1, l0, l1;
  int lim0, lim1;                                 // visible keys of the two rows this thread holds

  // P: AttnParams or AttnTcParams (n_q: query tokens of the window, lb: layer * batch + sequence)
  template <typename P>
  __device__ __forceinline__ void start(const P& p, int n_q, int rows, size_t lb, int g, int kv_len, int lane) {
    const int row0 = lane >> 2, row1 = row0 + 8, col = (lane & 3) * 2;
    const __nv_bfloat16* q0 = nullptr;
    const __nv_bfloat16* q1 = nullptr;
    lim0 = lim1 = 0;
    if (row0 < rows) {
      const int t = row0 / p.group, h = g * p.group + (row0 - t * p.group);
      q0 = p.q + ((lb * n_q + t) * p.n_q_heads + h) * D;
      lim0 = kv_len - n_q + t + 1;
    }
    if (row1 < rows) {
      const int t = row1 / p.group, h = g * p.group + (row1 - t * p.group);
      q1 = p.q + ((lb * n_q + t) * p.n_q_heads + h) * D;
      lim1 = kv_len - n_q + t + 1;
    }
#pragma unroll
    for (int ks = 0; ks < KSTEPS; ++ks) {
      qf[ks][0] = q0 ? *reinterpret_cast<const uint32_t*>(q0 + ks * 16 + col) : 0u;
      qf[ks][1] = q1 ? *reinterpret_cast<const uint32_t*>(q1 + ks * 16 + col) : 0u;
      qf[ks][2] = q0 ? *reinterpret_cast<const uint32_t*>(q0 + ks * 16 + 8 + col) : 0u;
      qf[ks][3] = q1 ? *reinterpret_cast<const uint32_t*>(q1 + ks * 16 + 8 + col) : 0u;
    }
#pragma unroll
    for (int nt = 0; nt < NT_O; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
    m0 = m1 = -INFINITY;
    l0 = l1 = 0.f;
  }

  // tile0: position of the tile's first token; vt: the V tile (generic address); cw: this warp's 16-token slice
  __device__ __forceinline__ void tile(uint32_t k_base, uint32_t v_base, uint8_t* vt, int tile0, int kv_len, float scale_log2,
                                       int cw, int lane) {
    const int col = (lane & 3) * 2;
    // per-lane ldmatrix row/chunk selectors
    const int mi = lane >> 3, r8 = lane & 7;
    const int k_tok = cw * 16 + (mi >> 1) * 8 + r8, k_chunk = mi & 1;   // K: non-transposed
    const int v_tok = cw * 16 + (mi & 1) * 8 + r8, v_chunk = mi >> 1;   // V: transposed
    const int tb = tile0 + cw * 16;                                      // first token of this warp's slice
    if (tb >= kv_len) return;
    if (tb + 16 > kv_len) {
      // rows past the end of the sequence hold whatever the page held: clear V there so that
      // a zero probability times a stale non-finite value cannot reach the accumulator
      const int first = kv_len - tile0;                                  // first invalid local row
      for (int t = first + (lane >> 3); t < cw * 16 + 16; t += 4) {
#pragma unroll
        for (int h = 0; h < D / 64; ++h)
          *reinterpret_cast<uint4*>(vt + h * (kTileTokens * 128) + t * 128 + (lane & 7) * 16) =
              make_uint4(0, 0, 0, 0);
      }
      fence_proxy_async();                                               // a copy may refill the slot later
      __syncwarp();
    }
    float sc[2][4];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < KSTEPS; ++ks) {
      uint32_t b0, b1, b2, b3;
      ldmatrix_x4(k_base + tile_offset<D>(k_tok, 2 * ks + k_chunk), b0, b1, b2, b3);
      mma_bf16_16816(sc[0], qf[ks], b0, b1);
      mma_bf16_16816(sc[1], qf[ks], b2, b3);
    }
    // scale, causal / length mask, running max
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int tok = tb + nt * 8 + col + (e & 1);
        const int lim = (e < 2) ? lim0 : lim1;
        const float v = tok < lim ? sc[nt][e] * scale_log2 : -INFINITY;
        sc[nt][e] = v;
        if (e < 2) mx0 = fmaxf(mx0, v); else mx1 = fmaxf(mx1, v);
      }
    }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);
    const float mu0 = mn0 == -INFINITY ? 0.f : mn0, mu1 = mn1 == -INFINITY ? 0.f : mn1;
    const float a0 = fast_exp2(m0 - mu0), a1 = fast_exp2(m1 - mu1);
    m0 = mn0;
    m1 = mn1;
    float ps0 = 0.f, ps1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      sc[nt][0] = fast_exp2(sc[nt][0] - mu0);
      sc[nt][1] = fast_exp2(sc[nt][1] - mu0);
      sc[nt][2] = fast_exp2(sc[nt][2] - mu1);
      sc[nt][3] = fast_exp2(sc[nt][3] - mu1);
      ps0 += sc[nt][0] + sc[nt][1];
      ps1 += sc[nt][2] + sc[nt][3];
    }
    l0 = l0 * a0 + ps0;
    l1 = l1 * a1 + ps1;
    uint32_t pa[4];
    pa[0] = pack_bf16x2(sc[0][0], sc[0][1]);
    pa[1] = pack_bf16x2(sc[0][2], sc[0][3]);
    pa[2] = pack_bf16x2(sc[1][0], sc[1][1]);
    pa[3] = pack_bf16x2(sc[1][2], sc[1][3]);
#pragma unroll
    for (int nt = 0; nt < NT_O; ++nt) {
      o[nt][0] *= a0;
      o[nt][1] *= a0;
      o[nt][2] *= a1;
      o[nt][3] *= a1;
    }
#pragma unroll
    for (int j = 0; j < D / 16; ++j) {
      uint32_t b0, b1, b2, b3;
      ldmatrix_x4_trans(v_base + tile_offset<D>(v_tok, 2 * j + v_chunk), b0, b1, b2, b3);
      mma_bf16_16816(o[2 * j], pa, b0, b1);
      mma_bf16_16816(o[2 * j + 1], pa, b2, b3);
    }
  }

  // this warp's partial to the merge buffer: o_sm [NW][16][OPITCH], m_sm and l_sm [NW][16]
  __device__ __forceinline__ void publish(float* o_sm, float* m_sm, float* l_sm, int rows, int warp, int lane) {
    const int row0 = lane >> 2, row1 = row0 + 8, col = (lane & 3) * 2;
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
    l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
    float* ow = o_sm + warp * 16 * OPITCH;
    // only the rows in use (7 of the 16 for the 7-head group of a decode step)
    if (row0 < rows) {
#pragma unroll
      for (int nt = 0; nt < NT_O; ++nt)
        *reinterpret_cast<float2*>(ow + row0 * OPITCH + nt * 8 + col) = make_float2(o[nt][0], o[nt][1]);
    }
    if (row1 < rows) {
#pragma unroll
      for (int nt = 0; nt < NT_O; ++nt)
        *reinterpret_cast<float2*>(ow + row1 * OPITCH + nt * 8 + col) = make_float2(o[nt][2], o[nt][3]);
    }
    if ((lane & 3) == 0) {
      m_sm[warp * 16 + row0] = m0;
      m_sm[warp * 16 + row1] = m1;
      l_sm[warp * 16 + row0] = l0;
      l_sm[warp * 16 + row1] = l1;
    }
  }
};

// The consumer warps' partials of row r, channels c .. c + 3, merged and normalised; returns the row's
// log-sum-exp (log2 units).  Every thread of the final pass derives its row's weights 2^(m_w - M) / den itself
// (16 shared loads and NW exponentials): cheaper than a separate weight phase behind two more barriers.
template <int D, int NW>
__device__ __forceinline__ float rows16_merge(const float* o_sm, const float* m_sm, const float* l_sm, int r, int c, float4& acc) {
  constexpr int OPITCH = Rows16<D>::OPITCH;
  float M = -INFINITY;
#pragma unroll
  for (int w = 0; w < NW; ++w) M = fmaxf(M, m_sm[w * 16 + r]);
  float den = 0.f;
  float wt[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    wt[w] = M != -INFINITY ? fast_exp2(m_sm[w * 16 + r] - M) : 0.f;
    den += l_sm[w * 16 + r] * wt[w];
  }
  const float inv = den > 0.f ? 1.f / den : 0.f;
  acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    const float f = wt[w] * inv;
    const float4 x = *reinterpret_cast<const float4*>(o_sm + (w * 16 + r) * OPITCH + c);
    acc.x += x.x * f;
    acc.y += x.y * f;
    acc.z += x.z * f;
    acc.w += x.w * f;
  }
  return den > 0.f ? M + log2f(den) : -INFINITY;
}

__device__ __forceinline__ void store_bf16x4(__nv_bfloat16* dst, const float4& v) {
  uint2 packed;
  packed.x = pack_bf16x2(v.x, v.y);
  packed.y = pack_bf16x2(v.z, v.w);
  *reinterpret_cast<uint2*>(dst) = packed;
}

constexpr int kMaxRows16Cluster = 8;       // the portable cluster size
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// By a consumer thread of a CTA that gives up (a wait expired): it stays, bounded, until the producer has gone and the last
// copies that it asked for have landed, since the CTA must not end under copies to its shared memory.  flags[0] is the abort
// flag, flags[1] the copies asked for once the producer has gone, -1 before.
template <int STAGES>
__device__ __forceinline__ void await_copies(uint32_t bar_full, volatile int* flags) {
  const uint64_t t0 = global_timer_ns();
  while (flags[1] < 0 && global_timer_ns() - t0 < kWaitLimitNs) {
  }
  const int issued = flags[1];
  for (int i = issued > STAGES ? issued - STAGES : 0; i < issued; ++i)
    while (!mbar_try_wait(bar_full + 8 * (i % STAGES), (i / STAGES) & 1) && global_timer_ns() - t0 < kWaitLimitNs) {
    }
}

// ---------------------------------------------------------------------------------------------
// One CTA per item.  4 consumer warps each own 16 of a tile's 64 tokens; they are merged once at the end.
// The last warp is the TMA producer.
// ---------------------------------------------------------------------------------------------
// NG consumer groups of 4 warps take alternate tiles (NG = 2 where an SM holds a single CTA, so
// that eight warps hide each other's latencies as two resident CTAs would).
// SPLIT: a cluster of n_cta CTAs per item, CTA r on tiles r, r + n_cta, ..; their results meet over distributed
// shared memory, each CTA folding its share of the output positions.  For a few short items, whose tiles one CTA would
// work through one after the other at 0.35 us each.
//
// The consumer warps of an item, or of a cluster's CTA.
template <int D, int STAGES, int NG, bool SPLIT>
__device__ __forceinline__ void rows16_consume(const AttnParams& p, uint8_t* smem, uint32_t base, volatile int* abort_flag,
                                               int kv_len, int n_my, int rank, int n_cta) {
  constexpr int TILE_BYTES = kTileTokens * D * 2, STAGE_BYTES = 2 * TILE_BYTES;
  constexpr int OPITCH = Rows16<D>::OPITCH;
  const uint32_t bar_full = base + STAGES * STAGE_BYTES, bar_empty = bar_full + 8 * STAGES;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = blockIdx.y, lb = blockIdx.z;
  const bool spec = p.block_table == nullptr;
  const int n_all = (kv_len + kTileTokens - 1) / kTileTokens;

  if (n_all == 0) {
    // An empty sequence: its outputs are zero, its LSE -inf.  The ring stays untouched: the tile that the producer
    // asked for before it knew the length may still be landing there, with whatever the cache rows hold.
    for (int idx = tid; idx < p.rows * (D / 8); idx += 128 * NG) {
      const int r = idx / (D / 8), c8 = idx - r * (D / 8);
      const int t = r / p.group, h = g * p.group + (r - t * p.group);
      const size_t orow = ((size_t)lb * p.n_q + t) * p.n_q_heads + h;
      *reinterpret_cast<uint4*>(p.out + orow * D + c8 * 8) = make_uint4(0, 0, 0, 0);
      if (p.lse && c8 == 0) p.lse[orow] = -INFINITY;
    }
    return;
  }
  const int cw = warp & 3, grp = warp >> 2;                           // token slice, consumer group
  Rows16<D> st;
  st.start(p, p.n_q, p.rows, lb, g, kv_len, lane);
  bool alive = true;
  // a CTA without a tile of its own: the one asked for before the length was known lands where the merge buffer will be
  if (SPLIT && n_my == 0 && spec && !mbar_wait(bar_full, 0, abort_flag)) alive = false;
  for (int i = grp; i < n_my; i += NG) {
    const int s = i % STAGES;
    if (!mbar_wait(bar_full + 8 * s, (i / STAGES) & 1, abort_flag)) {
      alive = false;
      break;
    }
    const uint32_t k_base = base + s * STAGE_BYTES;
    st.tile(k_base, k_base + TILE_BYTES, smem + s * STAGE_BYTES + TILE_BYTES, (i * n_cta + rank) * kTileTokens, kv_len,
            p.scale_log2, cw, lane);
    __syncwarp();
    if (lane == 0) mbar_arrive(bar_empty + 8 * s);
  }

  // test hook: the CTA that gives up although it has seen its tiles
  if (p.lost_cta == (int)((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x)) *abort_flag = 1;
  // ------------------------------------------------------------ merge the consumer warps' partials
  // (named barrier over the consumer threads; the producer warp has no part in it)
  asm volatile("bar.sync 1, %0;" ::"n"(128 * NG) : "memory");
  const bool gave_up = !alive || *abort_flag;   // a wait expired somewhere in this CTA (the flag tells all of it)
  // (the producer reports only the waits of its own, and it has none where the tiles fit the ring)
  if (gave_up && tid == 0 && p.d_status) *p.d_status = SPECVLM_ERR_TIMEOUT;
  if (!SPLIT && gave_up) {             // leave outputs alone
    if (tid == 0) await_copies<STAGES>(bar_full, abort_flag);
    return;
  }
  constexpr int NW = 4 * NG;                                           // consumer warps
  float* const o_sm = reinterpret_cast<float*>(smem);                  // [NW][16][OPITCH]
  float* const m_sm = o_sm + NW * 16 * OPITCH;                         // [NW][16]
  float* const l_sm = m_sm + NW * 16;                                  // [NW][16]
  st.publish(o_sm, m_sm, l_sm, p.rows, warp, lane);
  asm volatile("bar.sync 1, %0;" ::"n"(128 * NG) : "memory");
  if constexpr (SPLIT) {
    // This CTA's result, normalised, behind the merge buffer, and its log-sum-exps, for the whole cluster to read.  The
    // latter say whether the CTA gave up, and lie behind the ring, where no copy that was asked for before lands on them.
    float* const part_o = l_sm + NW * 16;                              // [16][D]
    float* const part_lse = reinterpret_cast<float*>(smem + STAGES * STAGE_BYTES + 16 * STAGES + 16);   // [16]
    for (int idx = tid; idx < p.rows * (D / 4); idx += 128 * NG) {
      const int r = idx / (D / 4), c = (idx - r * (D / 4)) * 4;
      float4 acc;
      const float lse2 = rows16_merge<D, NW>(o_sm, m_sm, l_sm, r, c, acc);
      *reinterpret_cast<float4*>(part_o + r * D + c) = acc;
      if (c == 0) part_lse[r] = gave_up ? __uint_as_float(kUnwritten) : lse2;
    }
    cluster_barrier();
    for (int idx = rank * 128 * NG + tid; idx < p.rows * (D / 4); idx += n_cta * 128 * NG) {
      const int r = idx / (D / 4), c = (idx - r * (D / 4)) * 4;
      float lse[kMaxRows16Cluster];
      float4 x[kMaxRows16Cluster];
#pragma unroll
      for (int k = 0; k < kMaxRows16Cluster; ++k) {
        lse[k] = -INFINITY;
        x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < n_cta) {
          lse[k] = ld_cluster_f32(cluster_map(smem_u32(part_lse + r), k));
          x[k] = ld_cluster_f32x4(cluster_map(smem_u32(part_o + r * D + c), k));
        }
      }
      float mm = -INFINITY, den = 0.f;
      bool lost = false;
#pragma unroll
      for (int k = 0; k < kMaxRows16Cluster; ++k) {
        lost |= unwritten(lse[k]);
        mm = fmaxf(mm, lse[k]);
      }
      if (lost) continue;                                              // a part is missing: leave the row alone
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < kMaxRows16Cluster; ++k) {
        const float w = lse[k] == -INFINITY ? 0.f : fast_exp2(lse[k] - mm);
        acc.x += w * x[k].x;
        acc.y += w * x[k].y;
        acc.z += w * x[k].z;
        acc.w += w * x[k].w;
        den += w;
      }
      const float inv = den > 0.f ? 1.f / den : 0.f;
      const int t = r / p.group, h = g * p.group + (r - t * p.group);
      const size_t orow = ((size_t)lb * p.n_q + t) * p.n_q_heads + h;
      store_bf16x4(p.out + orow * D + c, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
      if (p.lse && c == 0) p.lse[orow] = den > 0.f ? (mm + log2f(den)) * kLn2 : -INFINITY;
    }
    cluster_barrier();                                                 // nobody reads this CTA's shared memory any more
    if (gave_up && tid == 0) await_copies<STAGES>(bar_full, abort_flag);
    return;
  }
  for (int idx = tid; idx < p.rows * (D / 4); idx += 128 * NG) {
    const int r = idx / (D / 4), c = (idx - r * (D / 4)) * 4;
    float4 acc;
    const float lse2 = rows16_merge<D, NW>(o_sm, m_sm, l_sm, r, c, acc);
    const int t = r / p.group, h = g * p.group + (r - t * p.group);
    const size_t orow = ((size_t)lb * p.n_q + t) * p.n_q_heads + h;
    store_bf16x4(p.out + orow * D + c, acc);
    if (p.lse && c == 0) p.lse[orow] = lse2 * kLn2;
  }
}

// SPLIT: launched in clusters of gridDim.x CTAs per item, a number that the host's bound on the lengths gives.  A sequence of
// a few tiles is left to the first of them, since the hand-over would take longer (one layer, 4 items of d = 128 in a cache of
// 800 tokens, alone / by eight: 40 tokens 2.9 / 4.1 us, 200 3.9 / 4.1, 400 4.8 / 4.1; d = 64: 200 tokens 3.0 / 3.3, 400
// 3.8 / 3.3; by two, 36 items of d = 128: 200 tokens 4.1 / 4.5, 320 4.5 / 4.9, 400 5.2 / 5.1).  The producer serves both
// forms in one loop and the consumers have code of their own for each: the other ways round cost a cluster's full lengths
// 1 to 5 %.
constexpr int kSoloTiles = 4, kSoloTilesPair = 6;
// (CTAs per SM are as many as the ring allows; without that the compiler held d = 64 to 96 registers and spilled: 6 layers of
// 800 tokens, 24 items, 4.4 -> 4.2 us, 112 items of d = 128 and 755 tokens 9.83 -> 9.65)
template <int D, int STAGES, int NG, bool SPLIT>
__global__ void __launch_bounds__(32 * (4 * NG + 1), NG == 2 ? 1 : D == 64 ? 4 : 2)
attn_rows16_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                   const AttnParams p) {
  constexpr int TILE_BYTES = kTileTokens * D * 2;
  constexpr int STAGE_BYTES = 2 * TILE_BYTES;
  // A consumer group must see every phase of the ring slots it waits on: with the groups on
  // alternate tiles that holds only when a slot always belongs to the same group.  (A wait on a
  // phase two behind the barrier returns at once, the group then releases a slot it never read,
  // and the surplus arrival on the barrier is undefined behaviour: it faulted the kernel.)
  static_assert(STAGES % NG == 0, "ring depth must be a multiple of the number of consumer groups");

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* const smem = smem_raw + (base - raw_addr);
  const uint32_t bar_full = base + STAGES * STAGE_BYTES;
  const uint32_t bar_empty = bar_full + 8 * STAGES;
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(smem + STAGES * STAGE_BYTES + 16 * STAGES);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = blockIdx.y, lb = blockIdx.z;
  const int layer = lb / p.batch, b = lb - layer * p.batch;
  const int rank = SPLIT ? (int)blockIdx.x : 0, n_cta = SPLIT ? (int)gridDim.x : 1;

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 4);
    }
    abort_flag[0] = 0;
    abort_flag[1] = -1;                  // see await_copies
    mbar_fence_init();
  }
  if (tid == 32 * 4 * NG) {              // the producer's lane: descriptors are kernel parameters
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
  }
  __syncthreads();                       // the barriers are initialised
  pdl_launch_next();
  pdl_wait();

  // The first tile of a contiguous cache sits at a known place whatever the sequence's
  // length (rows past the cache's end are zero-filled by the copy): the producer asks for it
  // before the length has even been read, which takes a global-memory round trip off the start.
  const bool spec = p.block_table == nullptr;
  if (spec && tid == 32 * 4 * NG) {
    const uint64_t policy = l2_policy_evict_first();
    mbar_arrive_expect_tx(bar_full, STAGE_BYTES);
#pragma unroll
    for (int h = 0; h < D / 64; ++h) {
      tma_load_5d(base + h * (kTileTokens * 128), &tm_k, bar_full, h * 64, rank * kTileTokens, g, b, layer, policy);
      tma_load_5d(base + TILE_BYTES + h * (kTileTokens * 128), &tm_v, bar_full, h * 64, rank * kTileTokens, g, b, layer, policy);
    }
  }

  const int kv_len = clamp_len(p.seq_lens[b], p.max_seq_len);
  const int n_all = (kv_len + kTileTokens - 1) / kTileTokens;
  const bool solo = SPLIT && n_all <= (n_cta == 2 ? kSoloTilesPair : kSoloTiles);
  const int n_split = SPLIT ? (n_all + n_cta - 1 - rank) / n_cta : n_all;
  const int n_my = !solo ? n_split : rank == 0 ? n_all : 0;

  if (warp == 4 * NG) {
    // ------------------------------------------------------------------ producer
    if (lane == 0 && n_my == 0) {
      // an empty sequence, or a CTA without a part: nobody will consume the tile asked for above; stay until it has landed
      const uint64_t t0 = global_timer_ns();
      while (spec && !mbar_try_wait(bar_full, 0) && global_timer_ns() - t0 < kWaitLimitNs) {
      }
      abort_flag[1] = 0;
    }
    if (lane == 0 && n_my > 0) {
      const uint64_t policy = l2_policy_evict_first();
      const int tiles_per_block = p.block_tokens / kTileTokens;   // used only when paged
      int issued = spec ? 1 : 0;
      bool ok = true;
      for (int i = issued; i < n_my && ok; ++i) {
        const int s = i % STAGES;
        if (i >= STAGES) ok = mbar_wait(bar_empty + 8 * s, ((i / STAGES) - 1) & 1, abort_flag);
        if (!ok) break;
        const int t = solo ? i : i * n_cta + rank;
        int blk, tok;
        if (p.block_table) {
          blk = p.block_table[(size_t)b * p.max_blocks + t / tiles_per_block];
          tok = (t % tiles_per_block) * kTileTokens;
        } else {
          blk = b;
          tok = t * kTileTokens;
        }
        const uint32_t full = bar_full + 8 * s;
        mbar_arrive_expect_tx(full, STAGE_BYTES);
        const uint32_t dst = base + s * STAGE_BYTES;
#pragma unroll
        for (int h = 0; h < D / 64; ++h) {
          tma_load_5d(dst + h * (kTileTokens * 128), &tm_k, full, h * 64, tok, g, blk, layer, policy);
          tma_load_5d(dst + TILE_BYTES + h * (kTileTokens * 128), &tm_v, full, h * 64, tok, g, blk,
                      layer, policy);
        }
        issued = i + 1;
      }
      if (!ok) {
        // a wait expired: report, then stay until this CTA's copies in flight have landed
        if (p.d_status) *p.d_status = SPECVLM_ERR_TIMEOUT;
        const int first = issued > STAGES ? issued - STAGES : 0;
        for (int i = first; i < issued; ++i) {
          const uint64_t t0 = global_timer_ns();
          while (!mbar_try_wait(bar_full + 8 * (i % STAGES), (i / STAGES) & 1) &&
                 global_timer_ns() - t0 < kWaitLimitNs) {
          }
        }
      }
      abort_flag[1] = issued;
    }
    return;
  }

  if constexpr (SPLIT) {
    if (solo) {
      if (rank == 0) rows16_consume<D, STAGES, NG, false>(p, smem, base, abort_flag, kv_len, n_my, 0, 1);
      return;
    }
  }
  rows16_consume<D, STAGES, NG, SPLIT>(p, smem, base, abort_flag, kv_len, n_my, rank, n_cta);
}

// bar.sync 1 over n threads (whole warps) that also answers whether the predicate holds for all of them
__device__ __forceinline__ bool bar_and(bool pred, int n) {
  uint32_t all;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(all) : "r"((uint32_t)pred), "r"(n) : "memory");
  return all != 0;
}

// ---------------------------------------------------------------------------------------------
// The same on slices: a persistent CTA per SM streams a contiguous slice of the flat (layer, sequence, KV
// head, 64-token tile) list (attn_sched.h), whatever the items' number and lengths, so that every SM moves the
// same bytes; the producer runs ahead over item boundaries while the consumers merge and store an item, and
// items that a slice boundary cuts leave partial results for the merge kernel (attn_tc.cu).  It replaces a split
// of every item over the same number of CTAs with arrival counters (a memset, fences and a merge by one CTA):
// 1 layer of 6400 / 50 000 tokens 26.1 / 33.0 -> 8.6 / 21.4 us, 4 layers x 4 sequences of up to 12 800 tokens
// 99 -> 46.5 us (39 at the copy rate).
// ---------------------------------------------------------------------------------------------
template <int D>
struct SliceCfg {
  static constexpr int NG = 2;
  static constexpr int STAGES = D == 128 ? 4 : 8;
  static constexpr int TILE_BYTES = kTileTokens * D * 2;
  static constexpr int OFF_O = STAGES * 2 * TILE_BYTES;                          // merge buffer
  static constexpr int OFF_ML = OFF_O + 4 * NG * 16 * Rows16<D>::OPITCH * 4;
  static constexpr int OFF_BAR = OFF_ML + 2 * 4 * NG * 16 * 4;
  static constexpr int OFF_MISC = OFF_BAR + 16 * STAGES;
  static constexpr int OFF_PLAN = OFF_MISC + 16;
  static constexpr int OFF_PREFIX = OFF_PLAN + (kPlanBytes + 7) / 8 * 8;
  static constexpr int SMEM = OFF_PREFIX + (kSchedMaxBatch + 1) * 4 + 1024;
  static_assert(STAGES % NG == 0, "ring depth must be a multiple of the number of consumer groups");
  static_assert(SMEM <= 232448, "shared-memory plan does not fit");
};

template <int D>
__global__ void __launch_bounds__(32 * (4 * SliceCfg<D>::NG + 1), 1)
attn_rows16_slices_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                          const __grid_constant__ AttnTcParams p) {
  using C = SliceCfg<D>;
  constexpr int NG = C::NG, STAGES = C::STAGES, TILE_BYTES = C::TILE_BYTES, STAGE_BYTES = 2 * TILE_BYTES, NW = 4 * NG;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* const smem = smem_raw + (base - raw_addr);
  const uint32_t bar_full = base + C::OFF_BAR, bar_empty = bar_full + 8 * STAGES;
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC);
  CtaSlice* const slice = reinterpret_cast<CtaSlice*>(smem + C::OFF_PLAN);
  int* const prefix = reinterpret_cast<int*>(smem + C::OFF_PREFIX);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 4);
    }
    abort_flag[0] = 0;
    abort_flag[1] = -1;                  // see await_copies
    mbar_fence_init();
  }
  if (tid == 32 * NW) {
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
  }
  pdl_launch_next();
  pdl_wait();
  if (warp == 0) plan_slice<kTileTokens>(p, prefix, slice, blockIdx.x, gridDim.x, lane);
  if (warp > 0 && warp < NW) unwritten_parts(p, blockIdx.x, D, tid - 32, 32 * (NW - 1));
  __syncthreads();
  const int hkv = p.n_kv_heads, cta = blockIdx.x;
  const int64_t T0 = slice->begin, T1 = slice->end;

  if (warp == NW) {
    // ------------------------------------------------------------------ producer
    {
      const bool leader = elect_one();
      SliceCursor c;
      c.start(T0, T1, slice->first);
      const uint64_t policy = l2_policy_evict_first();
      const int tiles_per_block = p.block_table ? p.block_tokens / kTileTokens : 1;
      bool ok = true, told = false;
      int i = 0;
      for (; !c.done() && ok; ++i) {
        const int s = i % STAGES;
        if (i >= STAGES) ok = warp_wait(bar_empty + 8 * s, ((i / STAGES) - 1) & 1, abort_flag);
        if (!ok) break;
        const int t = c.sg.tile0 + c.j;
        int blk = c.sg.b, tok = t * kTileTokens;
        if (p.block_table) {
          blk = p.block_table[(size_t)c.sg.b * p.max_blocks + t / tiles_per_block];
          tok = (t % tiles_per_block) * kTileTokens;
        }
        const uint32_t full = bar_full + 8 * s, dst = base + s * STAGE_BYTES;
        if (leader) {
          mbar_arrive_expect_tx(full, STAGE_BYTES);
#pragma unroll
          for (int h = 0; h < D / 64; ++h) {
            tma_load_5d(dst + h * (kTileTokens * 128), &tm_k, full, h * 64, tok, c.sg.g, blk, c.sg.layer, policy);
            tma_load_5d(dst + TILE_BYTES + h * (kTileTokens * 128), &tm_v, full, h * 64, tok, c.sg.g, blk, c.sg.layer, policy);
          }
        }
        if (!told && i == STAGES - 1) {                     // the ring is full: time for the hand-over of a cut item
          if (leader) publish_cut_item(p, *slice, cta, cta, prefix);
          told = true;
        }
        c.next_tile(prefix, p.batch, hkv);
      }
      if (!told && leader) publish_cut_item(p, *slice, cta, cta, prefix);
      if (!ok) {
        // a wait expired: report, then stay until this CTA's copies in flight have landed
        if (p.d_status && leader) *p.d_status = SPECVLM_ERR_TIMEOUT;
        const uint64_t t0 = global_timer_ns();
        for (int k = i > STAGES ? i - STAGES : 0; k < i; ++k)
          while (!mbar_test_wait(bar_full + 8 * (k % STAGES), (k / STAGES) & 1) && global_timer_ns() - t0 < kWaitLimitNs) {
          }
      }
      if (leader) abort_flag[1] = i;
    }
    return;
  }

  // -------------------------------------------------------------------- consumers
  const int cw = warp & 3, grp = warp >> 2;                           // token slice, consumer group
  float* const o_sm = reinterpret_cast<float*>(smem + C::OFF_O);      // [NW][16][OPITCH]
  float* const m_sm = reinterpret_cast<float*>(smem + C::OFF_ML);     // [NW][16]
  float* const l_sm = m_sm + NW * 16;                                  // [NW][16]
  // sequences without any token: their outputs are zero, their LSE -inf
  if (slice->any_empty) {
    const int n_items = p.n_layers * p.batch * hkv;
    for (int item = cta; item < n_items; item += (int)gridDim.x) {
      const int lb = item / hkv, g = item - lb * hkv, b = lb % p.batch;
      if (prefix[b + 1] != prefix[b]) continue;
      for (int idx = tid; idx < p.rows * (D / 8); idx += 128 * NG) {
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
  bool alive = true;
  int i0 = 0;                                                          // slice index of the item's first tile
  while (!c.done()) {
    const Segment sg = c.sg;
    const int kv_len = clamp_len(p.seq_lens[sg.b], p.max_seq_len);
    const size_t lb = (size_t)sg.layer * p.batch + sg.b;
    Rows16<D> st;
    st.start(p, p.n_win, p.rows, lb, sg.g, kv_len, lane);
    for (int j = (grp + NG - i0 % NG) % NG; alive && j < sg.n_tiles; j += NG) {
      const int i = i0 + j, s = i % STAGES;
      if (!mbar_wait(bar_full + 8 * s, (i / STAGES) & 1, abort_flag)) {
        alive = false;
        break;
      }
      const uint32_t k_base = base + s * STAGE_BYTES;
      st.tile(k_base, k_base + TILE_BYTES, smem + s * STAGE_BYTES + TILE_BYTES, (sg.tile0 + j) * kTileTokens, kv_len,
              p.scale_log2, cw, lane);
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_empty + 8 * s);
    }
    // merge the consumer warps' partials; the first barrier also says that the previous item's have been read
    const bool complete = sg.tile0 == 0 && sg.n_tiles == sg.item_tiles;
    const int slot = partial_slot(cta, T0, sg.item_begin);
    // and whether every consumer has seen all its tiles: one answer for all threads, so that a row is stored whole or not at all
    const bool whole = bar_and(alive && cta != p.lost_cta, 128 * NG);
    if (!whole && tid == 0 && p.d_status) *p.d_status = SPECVLM_ERR_TIMEOUT;
    st.publish(o_sm, m_sm, l_sm, p.rows, warp, lane);
    asm volatile("bar.sync 1, %0;" ::"n"(128 * NG) : "memory");
    if (whole) {
      for (int idx = tid; idx < p.rows * (D / 4); idx += 128 * NG) {
        const int r = idx / (D / 4), ch = (idx - r * (D / 4)) * 4;
        float4 acc;
        const float lse2 = rows16_merge<D, NW>(o_sm, m_sm, l_sm, r, ch, acc);
        if (complete) {
          const int t = r / p.group, h = sg.g * p.group + (r - t * p.group);
          const size_t orow = (lb * p.n_win + t) * p.n_q_heads + h;
          store_bf16x4(p.out + orow * D + ch, acc);
          if (p.lse && ch == 0) p.lse[orow] = lse2 * kLn2;
        } else {
          const size_t prow = (size_t)slot * p.rows + r;
          *reinterpret_cast<float4*>(p.ws_o + prow * D + ch) = acc;
          if (ch % 64 == 0) p.ws_lse[(size_t)(ch / 64) * p.lse_block + prow] = lse2;
        }
      }
    }
    i0 += sg.n_tiles;
    c.next_segment(prefix, p.batch, hkv);
  }
  if (!alive && lane == 0) await_copies<STAGES>(bar_full, abort_flag);
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
// Test hook (specvlm_debug_set_attn_splits): 1 forces a CTA per item, n > 1 slices of about an n-th of a
// sequence each; 0 leaves the choice to the rule below.
static std::atomic<int> g_forced_splits{0};

constexpr int kRows16Max = 16;     // windows up to this many rows run on the 16-row kernels

// Time that one CTA takes for a tile, us.
static double rows16_tile_us(const specvlm_kv_t* kv) {
  return (kv->head_dim == 128 ? 0.35 : 0.25) * (kv->block_table ? 1.25 : 1.0);
}

// CTAs per item of a launch without slices: the number that is the fastest where every CTA has an SM of its own.  The
// hand-over costs 1.3 us: one layer of 4 items of 200 tokens 3.7 us with a CTA each, 4.3 with two; of 800 / 1600 / 3200
// tokens 7.0 / 11.3 / 20.1 with one (7.4 / 8.5 on slices from 1600) and 4.4 / 5.0 / 6.3 with eight.  Clusters do not use
// every SM of a GPC: 16 of eight CTAs no longer run side by side (4 layers of 800 tokens 7.3 -> 8.4), 24 of four do (2 layers
// x 3 sequences of 800 tokens 8.0 -> 5.4).
static int rows16_cluster(const specvlm_kv_t* kv, int64_t items, int64_t tiles) {
  if (g_forced_splits.load(std::memory_order_relaxed) == 1) return 1;
  int best = 1;
  double best_us = rows16_tile_us(kv) * tiles;
  for (int n = 2; n <= kMaxRows16Cluster; n *= 2) {
    const double us = 1.3 + rows16_tile_us(kv) * ((tiles + n - 1) / n);
    if (items * n <= (n == 2 ? 144 : n == 4 ? 96 : 64) && us < best_us) {
      best = n;
      best_us = us;
    }
  }
  return best;
}

// Whether slices are worth a workspace: estimated times in us, from the host's bound on the lengths, against a CTA per item.
static bool rows16_slices_beat_ctas(const specvlm_kv_t* kv, int32_t batch, int64_t items, int64_t tiles) {
  // A CTA per item: about 3 us around the tiles; while the items fit the SMs the longest one counts (one CTA takes 0.35 us
  // a tile at d = 128, a quarter more with a block table) or HBM does; beyond, rounds of two CTAs per SM at 0.75 us a tile,
  // or HBM with a last round that is partly empty.  Slices: 4.5 us with the merge kernel, the bytes, 2 us for every
  // item boundary of a CTA.  A batch is taken as ragged (slices balance it; so do many rounds): 0.85 of the bytes.
  // Slices have to win by 1.5 us: they cost a second launch.  Measured, 4 KV heads of d = 128, CTA per item / slices:
  // 1 layer of 1600 / 3200 / 6400 / 12 800 tokens 11.3 / 20.1 / 38.0 / 73.7 against 7.4 / 8.5 / 10.3 / 11.2; 20 layers of
  // 2560 / 5120 / 10 240 tokens 20.7 / 37.7 / 72.7 against 23.8 / 37.9 / 65.9; 28 layers of 640 / 1280 / 5120 tokens
  // 6.3 / 11.9 / 46.4 against 12.9 / 16.2 / 50.0; 28 layers x 4 ragged paged sequences of up to 640 / 1280 tokens
  // 18.1 / 34.0 against 28.1 / 41.4.
  const int64_t sms = sm_count();
  const double hbm = (double)items * tiles * (256.0 * kv->head_dim) / 6.65e6;
  const double ragged = batch > 1 ? 0.85 : 1.0;
  double per_item;
  if (items <= sms) {
    const double longest = rows16_tile_us(kv) * tiles;
    per_item = 3.0 + (longest > hbm ? longest : hbm);
  } else {
    const double rounds = (double)((items + 2 * sms - 1) / (2 * sms));
    const double stream = (1.0 + 0.2 / rounds) * ragged * hbm, serial = rounds * tiles * 0.75 * kv->head_dim / 128;
    per_item = 3.0 + (stream > serial ? stream : serial);
  }
  return 4.5 + ragged * hbm + 2.0 * (1.0 + (double)items / sms) + 1.5 < per_item;
}

// CTAs of a launch on slices, or 0 for a CTA (or a cluster) per item.  *scratch_ctas: the CTAs that the workspace has to
// have room for, 0 for none.  It does not depend on whether a cluster takes the slices' place: the choice between the two
// turns back and forth with the length, and a workspace sized for the longest sequences has to serve the shorter ones.
static int rows16_slices(const specvlm_kv_t* kv, int32_t batch, int* scratch_ctas) {
  const int64_t items = (int64_t)kv->n_layers * batch * kv->n_kv_heads;
  const int64_t tiles = (kv->max_seq_len + kTileTokens - 1) / kTileTokens, sms = sm_count();
  const int forced = g_forced_splits.load(std::memory_order_relaxed);
  *scratch_ctas = 0;
  if (batch > kSchedMaxBatch || forced == 1) return 0;
  if (forced > 1) {
    const int64_t n = items * (forced < tiles ? forced : tiles);
    return *scratch_ctas = (int)(n < 4 * sms ? n : 4 * sms);
  }
  if (!rows16_slices_beat_ctas(kv, batch, items, tiles)) return 0;
  *scratch_ctas = sched_scratch_ctas(items * tiles, (int)sms);
  const int n = rows16_cluster(kv, items, tiles);
  if (n > 1) {
    // A cluster per item, 3.9 us around its CTAs' tiles or the bytes, which half the SMs do not stream as well, against
    // slices, 6.5 us around the bytes (in pages 6) and more for many parts an item.  Measured, cluster / slices: 1 item
    // (d = 64) of 10 240 tokens 8.5 / 11.6; 12 items of 640 / 2560 / 10 240 4.9 / 7.3 / 18.5 against 7.0 / 8.3 / 16.4; 16 paged ones of 2560 / 5120 /
    // 10 240 8.3 / 13.4 / 23.9 against 9.0 / 10.8 / 15.7; 40 of 2560 / 10 240 / 20 480 11.3 / 38.8 / 75.5 against 14.2 / 37.3 /
    // 64.7; 64 of 1280 / 2560 / 5120 / 10 240 7.5 / 15.3 / 28.4 / 52.6 against 11.0 / 20.5 / 31.8 / 55.0; 72 ragged ones of up to
    // 1280 / 2560 / 10 240 7.5 / 11.3 / 47.2 against 12.9 / 16.1 / 48.3.
    const double hbm = (double)items * tiles * (256.0 * kv->head_dim) / 6.65e6, ragged = batch > 1 ? 0.85 : 1.0;
    const double longest = 1.08 * rows16_tile_us(kv) * ((tiles + n - 1) / n);
    const double parts = (double)(items * tiles < sms ? items * tiles : sms) / items;
    if ((kv->block_table ? 6.0 : 6.5) + ragged * hbm + 0.04 * parts >= 3.9 + (longest > 1.09 * hbm ? longest : 1.09 * hbm)) return 0;
  }
  const int even = sched_active_ctas(items * tiles, (int)sms);
  // slices that keep to item boundaries may use more CTAs: every item rounds its own up
  const int64_t aligned = items * sched_active_ctas(tiles, (int)sms);
  return aligned > even && items <= sms ? (int)(aligned < sms ? aligned : sms) : even;
}

static size_t rows16_scratch_bytes(const specvlm_kv_t* kv, int scratch_ctas, int rows) {
  return scratch_ctas == 0 ? 256 : SliceScratch(scratch_ctas, rows, kv->head_dim).bytes();
}
static size_t rows16_ws_bytes(const specvlm_kv_t* kv, int32_t batch, int rows) {
  int scratch_ctas;
  rows16_slices(kv, batch, &scratch_ctas);
  return rows16_scratch_bytes(kv, scratch_ctas, rows);
}

// tcgen05 path (attn_tc.cu)
size_t attn_tc_ws_bytes(const specvlm_kv_t* kv, int32_t batch, int rows, int group);
int32_t attn_tc_launch(const specvlm_kv_t* kv, const void* q, int32_t batch, int32_t n_q_heads, int32_t n_q,
                       float sm_scale, void* out, float* lse, void* ws, size_t ws_bytes, int32_t* d_status,
                       cudaStream_t st, const int32_t* tree_parents);

template <int D, int STAGES, int NG, bool SPLIT>
static int32_t launch_rows16_s(const CUtensorMap& tk, const CUtensorMap& tv, const AttnParams& p,
                               dim3 grid, cudaStream_t st) {
  constexpr int SMEM = STAGES * 2 * kTileTokens * D * 2 + 1024 + 16 * STAGES + 16 + (SPLIT ? 16 * 4 : 0);
  auto kern = attn_rows16_kernel<D, STAGES, NG, SPLIT>;
  static std::atomic<uint64_t> attr_done{0};
  if (!smem_attr_once(attr_done, reinterpret_cast<const void*>(kern), SMEM)) return SPECVLM_ERR_CUDA;
  return launch_clusters_after(kern, grid, (int)grid.x, dim3(32 * (4 * NG + 1)), (size_t)SMEM, st, tk, tv, p);
}

// Ring depth: 3 stages let two CTAs share an SM; a launch with no more CTAs than SMs would leave
// every SM with one CTA and 96 KB of copies in flight, too little to cover the HBM latency, so it
// takes 6 stages and two consumer groups instead.
template <int D>
static int32_t launch_rows16(const CUtensorMap& tk, const CUtensorMap& tv, const AttnParams& p,
                             dim3 grid, cudaStream_t st) {
  const int64_t ctas = (int64_t)grid.x * grid.y * grid.z;
  constexpr int kDeep = D == 128 ? 6 : 12;
  if (grid.x > 1) return launch_rows16_s<D, kDeep, 2, true>(tk, tv, p, grid, st);
  return ctas <= sm_count() ? launch_rows16_s<D, kDeep, 2, false>(tk, tv, p, grid, st)
                            : launch_rows16_s<D, 3, 1, false>(tk, tv, p, grid, st);
}

template <int D>
static int32_t launch_slices(const CUtensorMap& tk, const CUtensorMap& tv, const AttnTcParams& p, int ctas, cudaStream_t st) {
  using C = SliceCfg<D>;
  auto kern = attn_rows16_slices_kernel<D>;
  static std::atomic<uint64_t> attr_done{0};
  if (!smem_attr_once(attr_done, reinterpret_cast<const void*>(kern), C::SMEM)) return SPECVLM_ERR_CUDA;
  return launch_after(kern, dim3((unsigned)ctas), dim3(32 * (4 * C::NG + 1)), (size_t)C::SMEM, st, tk, tv, p);
}

// Test hook (specvlm_debug_attn_merge): one CTA's partial results as if it had given up, without a wait that expires.
__global__ void give_up_kernel(const __grid_constant__ AttnTcParams p, int gcta, int head_dim) {
  pdl_wait();
  unwritten_parts(p, gcta, head_dim, threadIdx.x, blockDim.x);
}

static int32_t attn_common(const specvlm_kv_t* kv, const void* q, int32_t batch, int32_t n_q_heads,
                           int32_t n_q, float sm_scale, void* out, float* lse, void* ws,
                           size_t ws_bytes, int32_t* d_status, void* stream, int lost_cta = -1, int32_t* n_ctas = nullptr) {
  int32_t rc = validate_kv(kv, batch, true);
  if (rc != SPECVLM_OK) return rc;
  if (!q || !out || n_q_heads < 1 || n_q < 1 || !(sm_scale > 0.f)) return SPECVLM_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(out)) return SPECVLM_ERR_INVALID_ARG;
  if (n_q_heads % kv->n_kv_heads != 0) return SPECVLM_ERR_INVALID_ARG;
  const int group = n_q_heads / kv->n_kv_heads;
  if (group > 16 || n_q > 9) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  const int rows = group * n_q;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (rows > kRows16Max)
    return attn_tc_launch(kv, q, batch, n_q_heads, n_q, sm_scale, out, lse, ws, ws_bytes, d_status, st, nullptr);

  const int64_t lb64 = (int64_t)kv->n_layers * batch;
  if (lb64 > 65535 || kv->n_kv_heads > 65535) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  CUtensorMap tk, tv;
  rc = encode_kv_map(&tk, kv, kv->k, kTileTokens);
  if (rc != SPECVLM_OK) return rc;
  rc = encode_kv_map(&tv, kv, kv->v, kTileTokens);
  if (rc != SPECVLM_OK) return rc;

  int scratch_ctas;
  const int ctas = rows16_slices(kv, batch, &scratch_ctas);
  if (scratch_ctas > 0) {
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return SPECVLM_ERR_INVALID_ARG;
    if (ws_bytes < rows16_scratch_bytes(kv, scratch_ctas, rows)) return SPECVLM_ERR_WORKSPACE_TOO_SMALL;
  }
  if (ctas > 0) {
    const SliceScratch sc(ctas, rows, kv->head_dim);
    AttnTcParams p = slice_params(kv, q, batch, n_q_heads, n_q, sm_scale, out, lse, d_status, 1, n_q, ws, sc);
    p.lost_cta = lost_cta;
    if (n_ctas) *n_ctas = ctas;
    rc = kv->head_dim == 128 ? launch_slices<128>(tk, tv, p, ctas, st) : launch_slices<64>(tk, tv, p, ctas, st);
    return rc != SPECVLM_OK ? rc : attn_merge_launch(p, kv->head_dim, ctas, st);
  }

  AttnParams p;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.out = static_cast<__nv_bfloat16*>(out);
  p.lse = lse;
  p.block_table = kv->block_table;
  p.seq_lens = kv->seq_lens;
  p.d_status = d_status;
  p.batch = batch;
  p.n_q = n_q;
  p.n_q_heads = n_q_heads;
  p.n_kv_heads = kv->n_kv_heads;
  p.group = group;
  p.rows = rows;
  p.max_blocks = kv->max_blocks;
  p.block_tokens = kv->block_tokens;
  p.max_seq_len = kv->max_seq_len;
  p.scale_log2 = sm_scale * kLog2e;
  p.lost_cta = lost_cta;

  const int n = rows16_cluster(kv, lb64 * kv->n_kv_heads, (kv->max_seq_len + kTileTokens - 1) / kTileTokens);
  dim3 grid((unsigned)n, (unsigned)kv->n_kv_heads, (unsigned)lb64);
  if (n_ctas) *n_ctas = (int32_t)(grid.x * grid.y * grid.z);
  return kv->head_dim == 128 ? launch_rows16<128>(tk, tv, p, grid, st) : launch_rows16<64>(tk, tv, p, grid, st);
}

}  // namespace specvlm

using namespace specvlm;

extern "C" void specvlm_debug_set_attn_splits(int32_t n_splits) {
  g_forced_splits.store(n_splits > 0 ? n_splits : 0, std::memory_order_relaxed);
}

extern "C" int32_t specvlm_debug_attn_merge(const specvlm_kv_t* kv, int32_t batch, int32_t n_q_heads, int32_t n_q,
                                            void* out, float* lse_or_null, void* ws, size_t ws_bytes, int32_t lost_cta,
                                            int32_t* n_ctas, void* stream) {
  const int32_t rc = validate_kv(kv, batch, true);
  if (rc != SPECVLM_OK) return rc;
  if (!out || !ws || !n_ctas || n_q_heads < 1 || n_q < 1 || n_q_heads % kv->n_kv_heads != 0) return SPECVLM_ERR_INVALID_ARG;
  const int group = n_q_heads / kv->n_kv_heads;
  if (group > 16 || n_q > 9 || batch > kSchedMaxBatch) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  int room;
  const SlicePlan pl = group * n_q > kRows16Max ? attn_tc_plan(kv, batch, group, n_q) : SlicePlan{rows16_slices(kv, batch, &room), 1, n_q};
  const int grid = pl.n_parts * pl.ctas;
  *n_ctas = grid;
  if (grid == 0) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  const SliceScratch sc(grid, pl.q_per * group, kv->head_dim);
  if (ws_bytes < sc.bytes()) return SPECVLM_ERR_WORKSPACE_TOO_SMALL;
  if (lost_cta >= grid) return SPECVLM_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const AttnTcParams p = slice_params(kv, nullptr, batch, n_q_heads, n_q, 1.f, out, lse_or_null, nullptr, pl.n_parts, pl.q_per, ws, sc);
  if (lost_cta >= 0) {
    const int32_t marked = launch_after(give_up_kernel, dim3(1), dim3(128), 0, st, p, lost_cta, kv->head_dim);
    if (marked != SPECVLM_OK) return marked;
  }
  return attn_merge_launch(p, kv->head_dim, pl.ctas, st);
}

extern "C" int32_t specvlm_debug_attn_give_up(const specvlm_kv_t* kv, const void* q, int32_t batch, int32_t n_q_heads, float sm_scale,
                                              void* out, float* lse_or_null, void* ws, size_t ws_bytes, int32_t lost_cta,
                                              int32_t* n_ctas, int32_t* d_status, void* stream) {
  if (!n_ctas) return SPECVLM_ERR_INVALID_ARG;
  return attn_common(kv, q, batch, n_q_heads, 1, sm_scale, out, lse_or_null, ws, ws_bytes, d_status, stream, lost_cta, n_ctas);
}

extern "C" size_t specvlm_attn_workspace_bytes(const specvlm_kv_t* kv, int32_t batch,
                                               int32_t n_q_heads, int32_t gamma) {
  if (!kv || batch < 1 || n_q_heads < 1 || gamma < 0 || kv->n_kv_heads < 1 ||
      n_q_heads % kv->n_kv_heads != 0 || kv->n_layers < 1 || kv->max_seq_len < 1)
    return 0;
  const int rows = (n_q_heads / kv->n_kv_heads) * (gamma + 1);
  if (n_q_heads / kv->n_kv_heads > 16 || gamma > 8) return 0;
  if (rows > kRows16Max) return batch <= kSchedMaxBatch ? attn_tc_ws_bytes(kv, batch, rows, n_q_heads / kv->n_kv_heads) : 0;
  return rows16_ws_bytes(kv, batch, rows);
}

extern "C" int32_t specvlm_draft_decode_attn(const specvlm_kv_t* kv, const void* q, int32_t batch,
                                             int32_t n_q_heads, float sm_scale, void* out,
                                             float* lse_or_null, void* ws, size_t ws_bytes,
                                             int32_t* d_status, void* stream) {
  NvtxRange nvtx_range(__func__);
  return attn_common(kv, q, batch, n_q_heads, 1, sm_scale, out, lse_or_null, ws, ws_bytes, d_status,
                     stream);
}

extern "C" int32_t specvlm_verify_attn(const specvlm_kv_t* kv, const void* q, int32_t batch,
                                       int32_t n_q_heads, int32_t gamma, float sm_scale, void* out,
                                       float* lse_or_null, void* ws, size_t ws_bytes,
                                       int32_t* d_status, void* stream) {
  NvtxRange nvtx_range(__func__);
  if (gamma < 0 || gamma > 8) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  return attn_common(kv, q, batch, n_q_heads, gamma + 1, sm_scale, out, lse_or_null, ws, ws_bytes,
                     d_status, stream);
}

extern "C" size_t specvlm_verify_tree_workspace_bytes(const specvlm_kv_t* kv, int32_t batch, int32_t n_q_heads,
                                                      int32_t n_nodes) {
  if (!kv || batch < 1 || batch > kSchedMaxBatch || n_q_heads < 1 || n_nodes < 1 || n_nodes > 64 ||
      kv->n_kv_heads < 1 || n_q_heads % kv->n_kv_heads != 0 || kv->n_layers < 1 || kv->max_seq_len < 1)
    return 0;
  const int rows = (n_q_heads / kv->n_kv_heads) * n_nodes;
  if (n_q_heads / kv->n_kv_heads > 16) return 0;
  return attn_tc_ws_bytes(kv, batch, rows, n_q_heads / kv->n_kv_heads);
}

extern "C" int32_t specvlm_verify_tree_attn(const specvlm_kv_t* kv, const void* q, const int32_t* parents,
                                            int32_t batch, int32_t n_q_heads, int32_t n_nodes, float sm_scale,
                                            void* out, float* lse_or_null, void* ws, size_t ws_bytes,
                                            int32_t* d_status, void* stream) {
  NvtxRange nvtx_range(__func__);
  int32_t rc = validate_kv(kv, batch, true);
  if (rc != SPECVLM_OK) return rc;
  if (!q || !out || !parents || n_q_heads < 1 || n_nodes < 1 || !(sm_scale > 0.f)) return SPECVLM_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(out) || n_q_heads % kv->n_kv_heads != 0) return SPECVLM_ERR_INVALID_ARG;
  const int group = n_q_heads / kv->n_kv_heads;
  if (group > 16 || n_nodes > 64) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  return attn_tc_launch(kv, q, batch, n_q_heads, n_nodes, sm_scale, out, lse_or_null, ws, ws_bytes, d_status,
                        static_cast<cudaStream_t>(stream), parents);
}
