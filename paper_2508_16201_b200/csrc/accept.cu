// Step 4c: greedy acceptance.  Kernel 1 streams the fp32 logits once (16-byte loads, all of a
// thread's loads in flight together) and leaves one (max, lowest index) candidate per (row, vocab
// chunk); kernel 2 finishes the argmax of the gamma+1 rows of a sequence and counts the leading
// draft tokens that equal it; its CTAs are scheduled while kernel 1 still runs (programmatic dependent
// launch), so the second launch costs no gap on the stream.
#include <mutex>

#include "common.cuh"
#include "host_util.h"

namespace specvlm {

constexpr int kAcceptThreads = 256;
constexpr int kAcceptVec = 8;                                      // float4 loads per thread, all issued up front
constexpr int kAcceptChunk = kAcceptThreads * kAcceptVec * 4;      // 8192 logits per CTA in kernel 1

struct Cand {
  float v;
  int32_t i;
};

// a is replaced by b when b is larger, or equal with a lower index
__device__ __forceinline__ void take_better(float& av, int& ai, float bv, int bi) {
  if (bv > av || (bv == av && bi < ai)) {
    av = bv;
    ai = bi;
  }
}

// The best of chunk `chunk` of the row at `base`, by a CTA; valid in thread 0.
__device__ __forceinline__ Cand chunk_best(const float* base, int vocab, int chunk) {
  const int lo = chunk * kAcceptChunk;
  const int hi = lo + kAcceptChunk < vocab ? lo + kAcceptChunk : vocab;
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  if (((reinterpret_cast<uintptr_t>(base + lo)) & 15u) == 0) {
    const int n4 = (hi - lo) >> 2;
    const float4* b4 = reinterpret_cast<const float4*>(base + lo);
    float4 x[kAcceptVec];
#pragma unroll
    for (int u = 0; u < kAcceptVec; ++u) {
      const int k = threadIdx.x + u * kAcceptThreads;
      x[u] = k < n4 ? __ldcs(b4 + k) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    }
#pragma unroll
    for (int u = 0; u < kAcceptVec; ++u) {
      const int i0 = lo + 4 * (threadIdx.x + u * kAcceptThreads);
      // ascending index with strict '>' keeps the lowest index among equals
      if (x[u].x > bv) { bv = x[u].x; bi = i0; }
      if (x[u].y > bv) { bv = x[u].y; bi = i0 + 1; }
      if (x[u].z > bv) { bv = x[u].z; bi = i0 + 2; }
      if (x[u].w > bv) { bv = x[u].w; bi = i0 + 3; }
    }
    for (int i = lo + 4 * n4 + threadIdx.x; i < hi; i += kAcceptThreads) take_better(bv, bi, base[i], i);
  } else {
    for (int i = lo + threadIdx.x; i < hi; i += kAcceptThreads) take_better(bv, bi, base[i], i);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
    take_better(bv, bi, ov, oi);
  }
  __shared__ float sv[kAcceptThreads / 32];
  __shared__ int si[kAcceptThreads / 32];
  if ((threadIdx.x & 31) == 0) {
    sv[threadIdx.x >> 5] = bv;
    si[threadIdx.x >> 5] = bi;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < kAcceptThreads / 32; ++w) take_better(bv, bi, sv[w], si[w]);
  return Cand{bv, bi};
}

__global__ void __launch_bounds__(kAcceptThreads)
accept_partial_kernel(const float* logits, int vocab, int n_chunks, Cand* __restrict__ part) {
  pdl_launch_next();
  pdl_wait();
  const int row = blockIdx.y, chunk = blockIdx.x;
  const Cand best = chunk_best(logits + (size_t)row * vocab, vocab, chunk);
  if (threadIdx.x == 0) part[(size_t)row * n_chunks + chunk] = best;
}

// A warp finishes the arg-max of a row of candidates (written by the grid before: read from L2); every lane has it.
__device__ __forceinline__ int row_argmax(const Cand* row, int n_chunks, int lane) {
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int c = lane; c < n_chunks; c += 32) {
    const int2 raw = __ldcg(reinterpret_cast<const int2*>(row + c));
    take_better(bv, bi, __int_as_float(raw.x), raw.y);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
    take_better(bv, bi, ov, oi);
  }
  return bi;
}

// The leading drafts that equal the rows' choices g_sm, by one thread.
__device__ __forceinline__ void match_drafts(const int* g_sm, const int32_t* draft, int b, int gamma, int32_t* accept_len,
                                             int32_t* next_token) {
  int n = 0;
  while (n < gamma && draft[(size_t)b * gamma + n] == g_sm[n]) ++n;
  accept_len[b] = n;
  next_token[b] = g_sm[n];
}

// The walk from the root to the child whose token is the choice at the current node, as long as there is one, by one
// thread.
__device__ __forceinline__ void walk_tree(const int* g_sm, const int32_t* node_tokens, const int32_t* parents, int b, int n_nodes,
                                          int32_t* accept_len, int32_t* next_token, int32_t* path) {
  const int32_t* tok = node_tokens + (size_t)b * n_nodes;
  const int32_t* par = parents + (size_t)b * n_nodes;
  int32_t* pth = path + (size_t)b * n_nodes;
  int cur = 0, n = 0;
  while (true) {
    int nxt = -1;
    for (int c = cur + 1; c < n_nodes; ++c)
      if (par[c] == cur && tok[c] == g_sm[cur]) {
        nxt = c;
        break;
      }
    if (nxt < 0) break;
    pth[n++] = nxt;
    cur = nxt;
  }
  for (int i = n; i < n_nodes; ++i) pth[i] = -1;
  accept_len[b] = n;
  next_token[b] = g_sm[cur];
}

// Both steps in one launch for a few short rows: a cluster of eight CTAs per sequence, a row each, whose choices go to
// the first CTA over distributed shared memory.  It saves the host a launch (6 rows of 1024 logits: 7.2 -> 3.7 us of host
// time) and the stream one while the clusters run side by side: device time, two launches / one, 6 rows of 1024 logits
// 2.87 / 2.26 us for one sequence, 2.98 / 2.58 for 16; 8 rows of 4096 3.18 / 2.95 for 24, 3.17 / 3.21 for 32, 3.59 / 3.94
// for 48; 1 row, seven of whose eight CTAs have none, 2.77 / 2.53 for 24, 2.77 / 3.84 for 64, 4.3 / 10.7 for 512.  With 8000
// logits a row, a whole chunk for a CTA, the device would take 4.1 us instead of 2.6.
// Up to 64 sequences the host's launch is longer than what the device loses, but in a graph.
constexpr int kAcceptSmallRows = 8, kAcceptSmallVocab = kAcceptChunk / 2, kAcceptSmallBatch = 24, kAcceptSmallBatchEager = 64;
static bool accept_small(int batch, int rows, int vocab, cudaStream_t st) {
  return rows <= kAcceptSmallRows && vocab <= kAcceptSmallVocab &&
         (batch <= kAcceptSmallBatch || (batch <= kAcceptSmallBatchEager && !being_captured(st)));
}
__global__ void __launch_bounds__(kAcceptThreads)
accept_small_kernel(const float* logits, int vocab, int rows, const int32_t* tokens, const int32_t* parents,
                    int32_t* __restrict__ accept_len, int32_t* __restrict__ next_token, int32_t* __restrict__ path,
                    int32_t* __restrict__ g_out) {
  __shared__ int g_sm[kAcceptSmallRows];
  const int b = blockIdx.x / kAcceptSmallRows, rank = blockIdx.x % kAcceptSmallRows;
  pdl_launch_next();
  pdl_wait();
  cluster_barrier();                       // every CTA of the cluster runs: the first one's shared memory may be written
  if (rank < rows) {
    const Cand best = chunk_best(logits + ((size_t)b * rows + rank) * vocab, vocab, 0);
    if (threadIdx.x == 0)
      asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(cluster_map(smem_u32(g_sm + rank), 0)), "r"(best.i) : "memory");
  }
  cluster_barrier();
  if (rank != 0) return;
  if (g_out && threadIdx.x < rows) g_out[(size_t)b * rows + threadIdx.x] = g_sm[threadIdx.x];
  if (threadIdx.x != 0) return;
  if (parents) walk_tree(g_sm, tokens, parents, b, rows, accept_len, next_token, path);
  else match_drafts(g_sm, tokens, b, rows - 1, accept_len, next_token);
}

// The finishing kernels do not release their successor early: CTAs of the next kernel would wait on the SMs that
// still stream logits (9 rows x 4 sequences 5.8 us a call, without 5.0; 9 x 16 15.6 and 15.2).
// one warp per (sequence, t); one CTA of (gamma+1) warps per sequence
__global__ void accept_finish_kernel(const Cand* part, int n_chunks,
                                     const int32_t* draft, int gamma,
                                     int32_t* __restrict__ accept_len, int32_t* __restrict__ next_token,
                                     int32_t* __restrict__ g_out) {
  __shared__ int g_sm[16];
  const int b = blockIdx.x, t = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();                            // kernel 1 has completed, its candidates are visible
  const int bi = row_argmax(part + ((size_t)b * (gamma + 1) + t) * n_chunks, n_chunks, lane);
  if (lane == 0) {
    g_sm[t] = bi;
    if (g_out) g_out[(size_t)b * (gamma + 1) + t] = bi;
  }
  __syncthreads();
  if (threadIdx.x == 0) match_drafts(g_sm, draft, b, gamma, accept_len, next_token);
}

// Tree drafting: one warp per node finishes its arg-max, then one thread walks the tree.
__global__ void accept_tree_finish_kernel(const Cand* part, int n_chunks,
                                          const int32_t* node_tokens,
                                          const int32_t* parents, int n_nodes,
                                          int32_t* __restrict__ accept_len, int32_t* __restrict__ next_token,
                                          int32_t* __restrict__ path, int32_t* __restrict__ g_out) {
  __shared__ int g_sm[64];
  const int b = blockIdx.x, lane = threadIdx.x & 31;
  pdl_wait();                            // kernel 1 has completed, its candidates are visible
  // a warp per node; with more than 32 nodes the warps take a second one each
  for (int t = threadIdx.x >> 5; t < n_nodes; t += blockDim.x >> 5) {
    const int bi = row_argmax(part + ((size_t)b * n_nodes + t) * n_chunks, n_chunks, lane);
    if (lane == 0) {
      g_sm[t] = bi;
      if (g_out) g_out[(size_t)b * n_nodes + t] = bi;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) walk_tree(g_sm, node_tokens, parents, b, n_nodes, accept_len, next_token, path);
}

// Built-in scratch of specvlm_accept_noalloc: room for kStaticCands (row, vocab chunk) candidates.
// Every GPU that loads the library holds these 128 KB until the process exits.
constexpr int kStaticCands = 16384;
static __device__ __align__(256) Cand g_accept_scratch[kStaticCands];

static int32_t launch_accept_small(const float* logits, int vocab, int batch, int rows, const int32_t* tokens,
                                   const int32_t* parents, int32_t* accept_len, int32_t* next_token, int32_t* path,
                                   int32_t* argmax, cudaStream_t st) {
  return launch_clusters_after(accept_small_kernel, dim3((unsigned)(batch * kAcceptSmallRows)), kAcceptSmallRows, dim3(kAcceptThreads), 0,
                               st, logits, vocab, rows, tokens, parents, accept_len, next_token, path, argmax);
}

}  // namespace specvlm

using namespace specvlm;

extern "C" size_t specvlm_accept_workspace_bytes(int32_t batch, int32_t gamma, int32_t vocab) {
  if (batch < 1 || gamma < 0 || vocab < 1) return 0;
  const size_t n_chunks = ((size_t)vocab + kAcceptChunk - 1) / kAcceptChunk;
  return round_up((size_t)batch * (gamma + 1) * n_chunks * sizeof(Cand), 256);
}

extern "C" int32_t specvlm_accept(const float* target_logits, const int32_t* draft_tokens,
                                  int32_t batch, int32_t gamma, int32_t vocab, int32_t* accept_len,
                                  int32_t* next_token, int32_t* target_argmax_or_null, void* ws,
                                  size_t ws_bytes, void* stream) {
  NvtxRange nvtx_range(__func__);
  if (!target_logits || !accept_len || !next_token || batch < 1 || gamma < 0 || vocab < 1 || !ws)
    return SPECVLM_ERR_INVALID_ARG;
  if (gamma > 0 && !draft_tokens) return SPECVLM_ERR_INVALID_ARG;
  if (gamma > 15) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  if ((int64_t)batch * (gamma + 1) > 65535) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  if ((reinterpret_cast<uintptr_t>(target_logits) & 3u) || (reinterpret_cast<uintptr_t>(ws) & 7u))
    return SPECVLM_ERR_INVALID_ARG;
  if (ws_bytes < specvlm_accept_workspace_bytes(batch, gamma, vocab)) return SPECVLM_ERR_WORKSPACE_TOO_SMALL;
  const int n_chunks = (vocab + kAcceptChunk - 1) / kAcceptChunk;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (accept_small(batch, gamma + 1, vocab, st))
    return launch_accept_small(target_logits, vocab, batch, gamma + 1, draft_tokens, nullptr, accept_len, next_token,
                               nullptr, target_argmax_or_null, st);
  Cand* part = static_cast<Cand*>(ws);
  int32_t rc = launch_after(accept_partial_kernel, dim3((unsigned)n_chunks, (unsigned)(batch * (gamma + 1))), dim3(kAcceptThreads), 0, st,
                            target_logits, vocab, n_chunks, part);
  if (rc != SPECVLM_OK) return rc;
  return launch_after(accept_finish_kernel, dim3((unsigned)batch), dim3(32u * (gamma + 1)), 0, st,
                          static_cast<const Cand*>(part), n_chunks, draft_tokens, gamma, accept_len, next_token,
                          target_argmax_or_null);
}

extern "C" int32_t specvlm_accept_noalloc(const float* target_logits, const int32_t* draft_tokens,
                                          int32_t batch, int32_t gamma, int32_t vocab, int32_t* accept_len,
                                          int32_t* next_token, int32_t* target_argmax_or_null, void* stream) {
  NvtxRange nvtx_range(__func__);
  if (!target_logits || !accept_len || !next_token || batch < 1 || gamma < 0 || vocab < 1)
    return SPECVLM_ERR_INVALID_ARG;
  if (gamma > 0 && !draft_tokens) return SPECVLM_ERR_INVALID_ARG;
  if (gamma > 15) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  if ((int64_t)batch * (gamma + 1) > 65535) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  if (reinterpret_cast<uintptr_t>(target_logits) & 3u) return SPECVLM_ERR_INVALID_ARG;
  const int n_chunks = (vocab + kAcceptChunk - 1) / kAcceptChunk;
  if ((int64_t)batch * (gamma + 1) * n_chunks > kStaticCands) return SPECVLM_ERR_TOO_LARGE;

  // Set-up, once per device: in host code the array's name is only a handle, the kernels need
  // the device address of this device's copy.
  constexpr int kMaxDevices = 64;
  static Cand* scratch_of[kMaxDevices] = {};
  static std::mutex mu;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SPECVLM_ERR_CUDA;
  Cand* part;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!scratch_of[dev]) {
      void* addr = nullptr;
      if (cudaGetSymbolAddress(&addr, g_accept_scratch) != cudaSuccess || !addr) return SPECVLM_ERR_CUDA;
      scratch_of[dev] = static_cast<Cand*>(addr);
    }
    part = scratch_of[dev];
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // every candidate slot that kernel 2 reads is written by kernel 1 of the same call first, so
  // nothing left over from an earlier call has to be cleared
  int32_t rc = launch_after(accept_partial_kernel, dim3((unsigned)n_chunks, (unsigned)(batch * (gamma + 1))), dim3(kAcceptThreads), 0, st,
                            target_logits, vocab, n_chunks, part);
  if (rc != SPECVLM_OK) return rc;
  return launch_after(accept_finish_kernel, dim3((unsigned)batch), dim3(32u * (gamma + 1)), 0, st,
                          static_cast<const Cand*>(part), n_chunks, draft_tokens, gamma, accept_len, next_token,
                          target_argmax_or_null);
}

extern "C" int32_t specvlm_accept_tree(const float* target_logits, const int32_t* node_tokens,
                                       const int32_t* parents, int32_t batch, int32_t n_nodes, int32_t vocab,
                                       int32_t* accept_len, int32_t* next_token, int32_t* path,
                                       int32_t* target_argmax_or_null, void* ws, size_t ws_bytes, void* stream) {
  NvtxRange nvtx_range(__func__);
  if (!target_logits || !node_tokens || !parents || !accept_len || !next_token || !path || !ws || batch < 1 ||
      n_nodes < 1 || vocab < 1)
    return SPECVLM_ERR_INVALID_ARG;
  if (n_nodes > 64 || (int64_t)batch * n_nodes > 65535) return SPECVLM_ERR_UNSUPPORTED_SHAPE;
  if ((reinterpret_cast<uintptr_t>(target_logits) & 3u) || (reinterpret_cast<uintptr_t>(ws) & 7u))
    return SPECVLM_ERR_INVALID_ARG;
  if (ws_bytes < specvlm_accept_workspace_bytes(batch, n_nodes - 1, vocab)) return SPECVLM_ERR_WORKSPACE_TOO_SMALL;
  const int n_chunks = (vocab + kAcceptChunk - 1) / kAcceptChunk;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (accept_small(batch, n_nodes, vocab, st))
    return launch_accept_small(target_logits, vocab, batch, n_nodes, node_tokens, parents, accept_len, next_token, path,
                               target_argmax_or_null, st);
  Cand* part = static_cast<Cand*>(ws);
  int32_t rc = launch_after(accept_partial_kernel, dim3((unsigned)n_chunks, (unsigned)(batch * n_nodes)), dim3(kAcceptThreads), 0, st,
                            target_logits, vocab, n_chunks, part);
  if (rc != SPECVLM_OK) return rc;
  return launch_after(accept_tree_finish_kernel, dim3((unsigned)batch), dim3(32u * (n_nodes < 32 ? n_nodes : 32)), 0, st,
                          static_cast<const Cand*>(part), n_chunks, node_tokens, parents, n_nodes, accept_len,
                          next_token, path, target_argmax_or_null);
}
