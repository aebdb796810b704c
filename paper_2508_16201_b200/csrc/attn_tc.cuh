// Shared by the attention kernels that work on slices of the flat tile list (attn_tc.cu: windows of up to 128
// rows; attn_pair.cu: wider ones; attn.cu: up to 16 rows): launch parameters, tensor-memory access, the cold paths of
// the softmax loops and the hand-over of cut items to the merge kernel.
#pragma once
#include "attn.cuh"
#include "attn_sched.h"
#include "host_util.h"

namespace specvlm {

struct AttnTcParams {
  const __nv_bfloat16* q;     // [L][B][n_win][Hq][D] (the kernels of attn_tc.cu and attn_pair.cu read it through a tensor map)
  __nv_bfloat16* out;         // [L][B][n_win][Hq][D]
  float* lse;                 // [L][B][n_win][Hq] or null
  float* ws_o;                // partial results: [2 * grid][rows][D], normalised
  float* ws_lse;              // [D / 64][2 * grid][rows], log2 units: per 64-channel block, see unwritten_parts
  int4* ws_cut;               // [grid]: the cut item whose first part a CTA holds, see attn_merge_kernel
  const int32_t* block_table; // [B][max_blocks] or null
  const int32_t* seq_lens;    // [B]
  int32_t* d_status;
  const int32_t* parents;     // [B][n_win] parents of a draft tree's nodes (<= 64), or null: the window is a chain
  int32_t batch, n_layers, n_q_heads, n_kv_heads, group;
  int32_t n_win;              // tokens of the whole window
  int32_t n_parts, q_per;     // the window is cut into n_parts parts of q_per tokens (the last may be shorter)
  int32_t rows;               // rows of a full part = q_per * group (<= 128): the row pitch of the scratch slots
  int32_t max_blocks, block_tokens, max_seq_len;
  int32_t align;              // slices may keep to item boundaries (attn_sched.h): no more items than CTAs
  int32_t lse_block;          // floats from one 64-channel block's LSEs to the next one's
  float scale_log2;           // sm_scale * log2(e)
  int32_t lost_cta;           // test hook (attn.cu): the CTA that gives up as if a wait had expired; -1 as a rule
};

constexpr float kRescaleThreshold = 8.f;   // log2 units
constexpr int kMaxTreeNodes = 64;          // a window mask is one 64-bit word per node
constexpr int kBigTokens = 2 * kTileTokens;          // tokens per MMA tile
constexpr int kTcThreads = 384;
// setmaxnreg moves registers between the warps of a CTA inside the pool the CTA got at launch
// (threads x registers per thread as compiled: 384 x 168), and an increase blocks until the pool
// has them -- for ever, if the requests add up to more than the pool.  The launch code checks the
// sum against the compiled kernel's pool and refuses to launch otherwise.
constexpr int kRegsLight = 96, kRegsSoftmax = 200;
constexpr int kRegsNeeded = 128 * kRegsLight + 256 * kRegsSoftmax;

template <int N> __device__ __forceinline__ void setmaxnreg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N> __device__ __forceinline__ void setmaxnreg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// 16 TMEM lanes x 64 fp32 columns -> 32 registers per thread: registers 4j, 4j+1 hold lane
// (base + tid/4), columns 8j + 2(tid%4) + {0,1}; registers 4j+2, 4j+3 the same columns of lane
// (base + 8 + tid/4).
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_16x256b_x8(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float ldg_cg_f32(const float* p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ldg_cg_f32x4(const float* p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

__device__ __forceinline__ int clamp_len(int n, int max_len) { return n < 0 ? 0 : (n > max_len ? max_len : n); }

// Cold paths of the softmax loop, kept out of line: the loop's code has to stay small enough for
// the instruction cache (with the mask logic inline the 128-row variant ran 25 % slower, although
// only one or two tiles of an item ever need a mask).
//
// Tiles that overlap the window of new tokens: the invisible logits of this thread's two rows
// (a 16-lane half of S: rows lr and lr + 8, columns 8j + lc + {0, 1} of each 64-column block) are
// overwritten with -inf in tensor memory, so the loop itself knows no masks.  Visibility of key
// `tok` for the row of query token t: every key before the window, and inside the window the
// positions whose bit is set in the row's mask -- the token's ancestors and itself for a tree
// (a0, a1 = the rows' masks), positions up to t for a chain (a0, a1 = the rows' limits `lim`:
// key tok is visible when tok < lim).
template <bool TREE>
__device__ __noinline__ void mask_s_half(uint32_t saddr, int tile_tok0, int win0, int lc, uint64_t a0, uint64_t a1) {
  const uint64_t a[2] = {a0, a1};
#pragma unroll 1
  for (int c = 0; c < 2; ++c) {
    uint64_t mk[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if constexpr (TREE) {
        // 128 visibility bits of the tile: the keys before the window, then the row's window mask
        // at the window's offset in the tile
        const int sh = win0 - tile_tok0;                       // tile column of window position 0
        unsigned __int128 full = 0;
        if (a[e]) {
          if (sh > 0) full = sh >= 128 ? ~(unsigned __int128)0 : (((unsigned __int128)1 << sh) - 1);
          const unsigned __int128 w = a[e];
          full |= sh >= 0 ? (sh < 128 ? w << sh : (unsigned __int128)0)
                          : (sh > -64 ? w >> (-sh) : (unsigned __int128)0);
        }
        mk[e] = (uint64_t)(full >> (64 * c)) >> lc;
      } else {
        const int n_vis = (int)a[e] - tile_tok0 - 64 * c;       // visible columns of the block
        mk[e] = (n_vis <= 0 ? 0ull : (n_vis >= 64 ? ~0ull : ((1ull << n_vis) - 1ull))) >> lc;
      }
    }
    uint32_t v[32];
    tmem_ld_16x256b_x8(saddr + 64 * c, v);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (!((mk[(k >> 1) & 1] >> ((k >> 2) * 8 + (k & 1))) & 1ull)) v[k] = 0xff800000u;   // -inf
    tmem_st_16x256b_x8(saddr + 64 * c, v);
  }
  tmem_st_wait();
}

// The window mask of a draft tree's node t (another one in each lane), by a whole warp: bit w says that it attends window
// position w, itself and the nodes on its path to a root.  par[t] < t, -1 for a root; a node whose path breaks that rule
// sees itself only, and that is reported.  The parents sit in two registers of the warp, a step up is two shuffles:
// a launch of its own for the masks cost a tree call 2.2 us on the host and 1 us on the device.
static __device__ __noinline__ uint64_t tree_mask(const int32_t* par, int n_nodes, int t, int32_t* d_status) {
  const int lane = threadIdx.x & 31;
  const int lo = lane < n_nodes ? __ldcg(par + lane) : -1, hi = lane + 32 < n_nodes ? __ldcg(par + lane + 32) : -1;
  uint64_t a = 1ull << t;
  int cur = t;
  bool going = true;
#pragma unroll 1
  while (__any_sync(0xffffffffu, going)) {
    const int p0 = __shfl_sync(0xffffffffu, lo, cur & 31), p1 = __shfl_sync(0xffffffffu, hi, cur & 31);
    const int up = cur < 32 ? p0 : p1;
    if (!going) continue;
    if (up < 0) {
      going = false;
    } else if (up >= cur) {
      if (d_status) *d_status = SPECVLM_ERR_INVALID_ARG;
      a = 1ull << t;
      going = false;
    } else {
      a |= 1ull << up;
      cur = up;
    }
  }
  return a;
}
// The nodes of a sequence that no tile brings up (it has no token), for the report alone.
__device__ __forceinline__ void check_tree(const int32_t* par, int n_nodes, int lane, int32_t* d_status) {
  for (int t0 = 0; t0 < n_nodes; t0 += 32) tree_mask(par, n_nodes, t0 + lane < n_nodes ? t0 + lane : n_nodes - 1, d_status);
}

// A row maximum grew past the lazy-rescale threshold: the rows' O accumulators (16-lane half,
// d columns from oaddr on) are multiplied by f0 (row lr) and f1 (row lr + 8) in tensor memory.
template <int D>
__device__ __noinline__ void rescale_o_half(uint32_t oaddr, float f0, float f1) {
#pragma unroll 1
  for (int cc = 0; cc < D / 64; ++cc) {
    uint32_t o[32];
    tmem_ld_16x256b_x8(oaddr + cc * 64, o);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 32; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * (((k >> 1) & 1) ? f1 : f0));
    tmem_st_16x256b_x8(oaddr + cc * 64, o);
  }
  tmem_st_wait();
}

// Running sum of the tiles (of TILE tokens) per sequence, by one warp: prefix[b] = tiles of the sequences before b.
// Returns whether some sequence has no token.
template <int TILE>
__device__ __forceinline__ bool tile_prefix(const AttnTcParams& p, int* prefix, int lane) {
  int carry = 0;
  bool empty = false;
  for (int b0 = 0; b0 < p.batch; b0 += 32) {
    const int b = b0 + lane;
    int v = 0;
    if (b < p.batch) {
      v = (clamp_len(p.seq_lens[b], p.max_seq_len) + TILE - 1) / TILE;
      empty |= v == 0;
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, v, off);
      if (lane >= off) v += o;
    }
    if (b < p.batch) prefix[b + 1] = v + carry;
    carry += __shfl_sync(0xffffffffu, v, 31);
  }
  if (lane == 0) prefix[0] = 0;
  return __any_sync(0xffffffffu, empty);
}

// A CTA's slice of the flat tile list.
struct CtaSlice {
  int64_t total, begin, end;   // tiles of the list; the slice (empty: the CTA has no work)
  Segment first;               // the slice's first segment
  int n_active;                // CTAs with work, of slices of equal length
  int parts;                   // slices that keep to item boundaries: the CTAs of this one's item; 0 otherwise
  int any_empty;               // some sequence has no token
};
constexpr int kPlanBytes = (int)sizeof(CtaSlice) + (kSchedAlignedBatch + 1) * 4;   // with the CTAs per sequence behind it

// The plan of CTA `cta` of `ctas`, by one warp: the running sums of the tiles and the CTA's slice, to shared memory.
template <int TILE>
__device__ __forceinline__ void plan_slice(const AttnTcParams& p, int* prefix, CtaSlice* out, int cta, int ctas, int lane) {
  const bool empty = tile_prefix<TILE>(p, prefix, lane);
  __syncwarp();
  const int per_head = prefix[p.batch], lh = p.n_layers * p.n_kv_heads;
  const int64_t total = (int64_t)lh * per_head;
  int q = 0;
  int* const part_prefix = reinterpret_cast<int*>(out + 1);
  if (p.align && total > 0 && total < 0x7fffffff) {
    const int t = lane < p.batch ? prefix[lane + 1] - prefix[lane] : 0;
    const int q_first = aligned_q_first((int)total, ctas);
    int n = 0;
#pragma unroll
    for (int c = kSchedAlignedTries - 1; c >= 0; --c) {    // the first that fits is kept; sums of both, then one scan
      const int m = (int)((uint32_t)(t + q_first + c - 1) / (uint32_t)(q_first + c));
      if ((int64_t)lh * __reduce_add_sync(0xffffffffu, m) <= ctas) {
        q = q_first + c;
        n = m;
      }
    }
    if (q > 0) {
      if (p.batch > 1) {
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int o = __shfl_up_sync(0xffffffffu, n, off);
          if (lane >= off) n += o;
        }
      }
      part_prefix[lane + 1] = n;
      if (lane == 0) part_prefix[0] = 0;
    }
    __syncwarp();
  }
  if (lane == 0) {
    out->total = total;
    out->any_empty = empty ? 1 : 0;
    int64_t begin = 0, end = 0;
    int n_active = 1, parts = 0;
    Segment s = {};
    if (q > 0) {
      if (aligned_slice(cta, prefix, part_prefix, p.batch, p.n_layers, p.n_kv_heads, &s, &parts)) {
        begin = s.item_begin + s.tile0;
        end = begin + s.n_tiles;
      }
    } else if (total > 0) {
      n_active = sched_active_ctas(total, ctas);
      if (cta < n_active) {
        begin = slice_begin(cta, n_active, total);
        end = slice_begin(cta + 1, n_active, total);
        s = segment_at(begin, end, prefix, p.batch, p.n_kv_heads);
      }
    }
    out->begin = begin;
    out->end = end;
    out->first = s;
    out->n_active = n_active;
    out->parts = parts;
  }
}

// Which item, if any, this CTA's slice holds the first part of while a slice boundary cuts it: (layer *
// batch + sequence, KV head, scratch slot of the first part, number of parts), no parts if there is none.
// Written before any wait, so that the merge never reads a stale entry.
__device__ __forceinline__ void publish_cut_item(const AttnTcParams& p, const CtaSlice& sl, int cta, int gcta, const int* prefix) {
  int4 cut = make_int4(0, 0, 0, 0);
  if (sl.begin < sl.end && sl.end < sl.total) {
    const Segment s = segment_at(sl.end - 1, sl.end, prefix, p.batch, p.n_kv_heads);   // the item of the slice's last tile
    const int64_t item_end = s.item_begin + s.item_tiles;
    if (item_end > sl.end && s.item_begin >= sl.begin)
      cut = make_int4(s.layer * p.batch + s.b, s.g, partial_slot(gcta, sl.begin, s.item_begin),
                      sl.parts > 0 ? sl.parts : slice_owner(item_end - 1, sl.n_active, sl.total) - cta + 1);
  }
  p.ws_cut[gcta] = cut;
}

// A CTA that gives up (a wait expired) leaves partial results unwritten, and the merge must make nothing of what their
// slots hold.  So every CTA first fills the LSEs of its two slots with a bit pattern that no LSE has (a CTA stores -inf, a
// finite value or +inf), before the barrier behind its set-up, and the merge leaves a row alone that has such a part.  Where two
// groups of warps store a row's channels (attn_tc.cu at d = 128) one of them may give up where the other does not: each
// stores an LSE of its own with its 64-channel block.
constexpr uint32_t kUnwritten = 0xffffffffu;
__device__ __forceinline__ bool unwritten(float lse) { return __float_as_uint(lse) == kUnwritten; }
// by n_threads threads t = 0 ..
__device__ __forceinline__ void unwritten_parts(const AttnTcParams& p, int gcta, int head_dim, int t, int n_threads) {
  float* const slots = p.ws_lse + (size_t)2 * gcta * p.rows;
#pragma unroll 1
  for (int i = t; i < 2 * p.rows; i += n_threads) {
    slots[i] = __uint_as_float(kUnwritten);
    if (head_dim == 128) slots[p.lse_block + i] = __uint_as_float(kUnwritten);
  }
}

// attn_tc.cu: the merge of the items that slice boundaries cut, for a launch of n_parts sets of `ctas` CTAs
int32_t attn_merge_launch(const AttnTcParams& p, int head_dim, int ctas, cudaStream_t st);

// Scratch of a launch: partial results [2 * grid][rows][D], their LSEs, and the item that each CTA's slice cuts.
struct SliceScratch {
  int grid;
  size_t o_bytes, lse_bytes, cut_bytes;
  SliceScratch(int grid, int rows, int head_dim)
      : grid(grid),
        o_bytes(round_up((size_t)2 * grid * rows * head_dim * sizeof(float), 256)),
        lse_bytes(round_up((size_t)2 * grid * rows * (head_dim / 64) * sizeof(float), 256)),
        cut_bytes(round_up((size_t)grid * sizeof(int4), 256)) {}
  size_t bytes() const { return o_bytes + lse_bytes + cut_bytes; }
};

inline AttnTcParams slice_params(const specvlm_kv_t* kv, const void* q, int32_t batch, int32_t n_q_heads, int32_t n_q,
                                 float sm_scale, void* out, float* lse, int32_t* d_status, int n_parts, int q_per, void* ws,
                                 const SliceScratch& sc) {
  AttnTcParams p;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.out = static_cast<__nv_bfloat16*>(out);
  p.lse = lse;
  uint8_t* const w = static_cast<uint8_t*>(ws);
  p.ws_o = reinterpret_cast<float*>(w);
  p.ws_lse = reinterpret_cast<float*>(w + sc.o_bytes);
  p.ws_cut = reinterpret_cast<int4*>(w + sc.o_bytes + sc.lse_bytes);
  p.block_table = kv->block_table;
  p.seq_lens = kv->seq_lens;
  p.d_status = d_status;
  p.parents = nullptr;
  p.batch = batch;
  p.n_layers = kv->n_layers;
  p.n_q_heads = n_q_heads;
  p.n_kv_heads = kv->n_kv_heads;
  p.group = n_q_heads / kv->n_kv_heads;
  p.n_win = n_q;
  p.n_parts = n_parts;
  p.q_per = q_per;
  p.rows = q_per * p.group;
  p.max_blocks = kv->max_blocks;
  p.block_tokens = kv->block_tokens;
  p.max_seq_len = kv->max_seq_len;
  p.align = (int64_t)p.n_layers * batch * p.n_kv_heads <= sc.grid / n_parts && batch <= kSchedAlignedBatch;
  p.lse_block = 2 * sc.grid * p.rows;
  p.scale_log2 = sm_scale * kLog2e;
  p.lost_cta = -1;
  return p;
}

// How a launch on slices of a given window is laid out: `ctas` CTAs in each of n_parts sets (0: a CTA per item).
struct SlicePlan {
  int ctas, n_parts, q_per;
};
SlicePlan attn_tc_plan(const specvlm_kv_t* kv, int32_t batch, int32_t group, int32_t n_q);      // attn_tc.cu

// (a template of the kernel itself: kernels of one signature must not share the flag below)
template <auto kern>
static int32_t launch_tc_kernel(int smem, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq,
                                const AttnTcParams& p, int grid, cudaStream_t st) {
  // once per device and kernel: the opt-in shared-memory size, and the check that the compiled
  // kernel's register pool can satisfy the setmaxnreg requests (it never changes)
  static std::atomic<uint64_t> attr_done{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return SPECVLM_ERR_CUDA;
  if (!(attr_done.load(std::memory_order_acquire) & (1ull << (dev & 63)))) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) return SPECVLM_ERR_CUDA;
    if (fa.numRegs * kTcThreads < kRegsNeeded) return SPECVLM_ERR_CUDA;   // setmaxnreg could never be satisfied
    if (!smem_attr_once(attr_done, reinterpret_cast<const void*>(kern), smem)) return SPECVLM_ERR_CUDA;
  }
  return launch_after(kern, dim3((unsigned)grid), dim3(kTcThreads), (size_t)smem, st, tk, tv, tq, p);
}

}  // namespace specvlm
