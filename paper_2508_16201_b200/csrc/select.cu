// Steps 1b + 2: Stage I top-k retention and Stage II spatially uniform reduction.  One cluster of up
// to eight CTAs per sequence; every thread keeps its share of the keys in registers.
//   1. radix select (8 bits a pass, most significant first) finds the k1-th largest key T and how
//      many keys equal to T belong to the top-k1; a pass ends the descent early when its digit's keys
//      are wanted whole;
//   2. ordered scans give the rank of each key equal to T among its equals, so ties go to the lower
//      index, and the number of unselected tokens before each token and before each frame;
//   3. the Stage-II pick test is integer arithmetic per token, and so is a kept token's place in
//      the output: (selected tokens before it) + (picks before it), both closed forms of the
//      unselected count, so no third scan is needed.
// Everything is deterministic: no atomics decide an output.
//
// Top-P mode (Eq. 6): the Stage-I count is the shortest prefix of the ranking whose cumulative
// score reaches lambda_r of the total.  The same radix descent runs on score mass instead of
// counts, and ends at the very key and tie count that the selection needs.  Masses are the scores
// truncated to multiples of 2^-36 (capped at 1) and summed as integers, lambda_r is in
// thousandths: integer sums do not depend on the order of the additions, so the count is a
// function of the scores alone.
//
// What bounds it is latency: a pass is a shared-memory histogram, one exchange over the cluster
// and a scan; the keys' range is found first so that a pass spreads them over all its digits (with
// fixed digits the leading byte of a request's scores takes two or three values, and the atomics
// collide: 10 % to 25 % slower).  6272 scores of a 32-frame video: 19.4 us with one CTA that walked the keys in
// shared memory, 8.5 us now (Top-P 27.8 -> 12.3); 50 176 scores of a 256-frame video: 84 -> 18.6 us
// (Top-P 154.5 -> 24.4); 16 sequences of 6272: 19.8 -> 10.8 us.
#include <cooperative_groups.h>

#include "common.cuh"
#include "host_util.h"

namespace specvlm {

namespace cg = cooperative_groups;

constexpr int kSelThreads = 512;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelMaxCluster = 8;      // the portable cluster size
constexpr int kSelMaxKeys = 14;        // keys per thread: 8 x 512 x 14 = 57 344 tokens
constexpr int kSelMaxFrames = 1024;
constexpr int kSelCopies = 8;          // interleaved copies of a histogram bin: lanes with equal digits spread over them
constexpr int kSelMaxBatch = 64;
constexpr int kTopPFracBits = 36;

// score mass of a key (keys of non-negative floats are their bits with the top bit set)
__device__ __forceinline__ unsigned long long key_mass(uint32_t key) {
  const double a = (double)__uint_as_float(key & 0x7fffffffu) * (double)(1ull << kTopPFracBits);
  const unsigned long long one = 1ull << kTopPFracBits;
  return a >= (double)one ? one : (unsigned long long)a;
}

struct SelSeq {
  int32_t score_off, n_frames, k1, k_total, kept_off;
  int32_t lambda_pm;                   // >= 0: Top-P mode, k1 is computed; < 0: k1 as given
  int32_t seq_index;                   // position in the batch (random selector's counter word)
};

// Philox-4x32, 10 rounds (Salmon et al., SC'11), first output word: the counter-based generator
// of the random selector
__device__ __forceinline__ uint32_t philox4x32_10_word0(uint32_t c0, uint32_t c1, uint32_t k0, uint32_t k1) {
  uint32_t c2 = 0u, c3 = 0u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c0;
}
struct SelParams {
  const float* scores;
  int32_t* kept_idx;
  int32_t* k1_out;                     // [batch] Stage-I counts or null
  int32_t tokens_per_frame;
  int32_t k1_out_base;                 // index of seq[0] in k1_out
  int32_t random_keys;                 // 1: rank Philox keys instead of scores
  uint32_t seed_lo, seed_hi;
  SelSeq seq[kSelMaxBatch];
};

// Shared-memory plan of a CTA (dynamic).  The received histograms are double-buffered by pass, so
// one cluster barrier per pass is enough.
struct SelSmem {
  uint32_t hist[3][256 * kSelCopies];                      // counts, low and high mass pieces: all zero between passes
  uint32_t rcount[2][kSelMaxCluster][256];                 // every CTA's counts of the pass, by digit
  unsigned long long rmass[2][kSelMaxCluster][256];        // ... and masses (Top-P descent)
  uint32_t wmin[kSelWarps], wmax[kSelWarps];
  uint32_t rmin[kSelMaxCluster], rmax[kSelMaxCluster];     // every CTA's smallest and largest key
  unsigned long long wmass[8];                             // warp totals of a scan
  unsigned long long mass_above;
  int wcount[kSelWarps];
  int digit, count, same;                                  // result of a pass's scan
  int less[kSelMaxCluster], equal[kSelMaxCluster];         // every CTA's keys below and equal to the threshold
  int cf[kSelMaxFrames + 1];                                        // unselected tokens before each frame
  uint32_t quota[kSelMaxFrames + 1];                                // Stage-II picks before each frame
};

// One pass of the descent over the live keys [base, base + (n_digits << shift)), n_digits <= 256: into the CTA's histogram, the
// histogram to every CTA of the cluster, and the scan of the summed bins from 255 down.  Leaves in sm.digit the digit
// at which the running count reaches `want` (or, with MASS, 1000 x the running mass reaches `want`);
// through sm.count the count (and sm.mass_above the mass) of the larger digits, through sm.same the
// count of that digit's keys.  Every CTA does the same scan.  FIRST (with MASS): `want` is the
// fraction in thousandths and becomes that fraction of the total mass; a total of zero leaves sm.digit at -1.
template <int KEYS, bool MASS, bool FIRST>
__device__ __forceinline__ void sel_pass(SelSmem& sm, cg::cluster_group& cluster, const uint32_t (&key)[KEYS],
                                         uint32_t valid, uint32_t base, uint32_t n_digits, int shift, int parity, unsigned long long& want,
                                         unsigned long long above, int n_above) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_cta = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int copy = lane & (kSelCopies - 1);
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    const uint32_t digit = (key[i] - base) >> shift;        // (a key below base wraps round to a large digit)
    if (((valid >> i) & 1u) && digit < n_digits) {
      const uint32_t at = digit * kSelCopies + copy;
      atomicAdd(&sm.hist[0][at], 1u);
      if (MASS) {
        // 64-bit sums as two pieces of 18 bits: a CTA's at most 7168 keys keep each sum below 2^32
        const unsigned long long q = key_mass(key[i]);
        atomicAdd(&sm.hist[1][at], (uint32_t)q & 0x3ffffu);
        atomicAdd(&sm.hist[2][at], (uint32_t)(q >> 18));
      }
    }
  }
  if (FIRST && tid == 0) sm.digit = -1;
  __syncthreads();
  if (tid < 256) {
    auto take = [&](int which) {
      uint4* const h = reinterpret_cast<uint4*>(&sm.hist[which][tid * kSelCopies]);
      const uint4 a = h[0], b = h[1];
      h[0] = h[1] = make_uint4(0u, 0u, 0u, 0u);            // ready for the next pass
      return (unsigned long long)a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
    };
    const uint32_t n = (uint32_t)take(0);
    unsigned long long m = 0ull;
    if (MASS) m = take(1) + (take(2) << 18);
#pragma unroll
    for (int c = 0; c < kSelMaxCluster; ++c) {
      if (c < n_cta) {
        *cluster.map_shared_rank(&sm.rcount[parity][rank][tid], c) = n;
        if (MASS) *cluster.map_shared_rank(&sm.rmass[parity][rank][tid], c) = m;
      }
    }
  }
  cluster.sync();
  // thread t holds digit 255 - t: an inclusive scan over the threads is a scan from the top digit down
  int n = 0, n_incl = 0;
  unsigned long long m = 0ull, m_incl = 0ull;
  if (tid < 256) {
    const int d = 255 - tid;
#pragma unroll
    for (int c = 0; c < kSelMaxCluster; ++c) {
      if (c < n_cta) {
        n += (int)sm.rcount[parity][c][d];
        if (MASS) m += sm.rmass[parity][c][d];
      }
    }
    n_incl = n;
    m_incl = m;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int vn = __shfl_up_sync(0xffffffffu, n_incl, off);
      const unsigned long long vm = MASS ? __shfl_up_sync(0xffffffffu, m_incl, off) : 0ull;
      if (lane >= off) {
        n_incl += vn;
        m_incl += vm;
      }
    }
    if (lane == 31) {
      sm.wcount[warp] = n_incl;
      if (MASS) sm.wmass[warp] = m_incl;
    }
  }
  __syncthreads();
  if (FIRST) {
    unsigned long long total = 0ull;
#pragma unroll
    for (int w = 0; w < 8; ++w) total += sm.wmass[w];
    want *= total;
  }
  if (tid < 256) {
    int n_before = n_above + n_incl - n;                    // live keys with larger digits, and all before them
    unsigned long long m_before = above + m_incl - m;
#pragma unroll
    for (int w = 0; w < 7; ++w) {
      if (w < warp) {
        n_before += sm.wcount[w];
        if (MASS) m_before += sm.wmass[w];
      }
    }
    const bool here = MASS ? 1000ull * m_before < want && 1000ull * (m_before + m) >= want
                           : (unsigned long long)n_before < want && (unsigned long long)(n_before + n) >= want;
    if (here) {
      sm.digit = 255 - tid;
      sm.count = n_before;
      sm.mass_above = m_before;
      sm.same = n;
    }
  }
  __syncthreads();
}

// KEYS: keys per thread (an upper bound of the launch's).  Token j of the sequence belongs to CTA, warp,
// round i and lane in that order of significance, so the order of tokens is the order of ballots.
template <int KEYS>
__global__ void __launch_bounds__(kSelThreads, KEYS <= 6 ? 2 : 1) select_kernel(const __grid_constant__ SelParams p) {
  extern __shared__ __align__(16) uint8_t sel_smem[];
  SelSmem& sm = *reinterpret_cast<SelSmem*>(sel_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int n_cta = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int seq = blockIdx.x / n_cta;
  const SelSeq sq = p.seq[seq];
  const int T = p.tokens_per_frame, F = sq.n_frames, n_v = F * T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k_total = sq.k_total;
  int k1 = sq.k1;
  const int n_keys = (n_v + n_cta * kSelThreads - 1) / (n_cta * kSelThreads);
  const int j0 = (rank * kSelWarps + warp) * 32 * n_keys + lane;   // this thread's tokens: j0 + 32 i

  pdl_launch_next();
  for (int i = tid; i < 3 * 256 * kSelCopies / 4; i += kSelThreads)
    reinterpret_cast<uint4*>(&sm.hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
  pdl_wait();
  // order-preserving map float -> uint32 (larger float <=> larger key)
  uint32_t key[KEYS];
  uint32_t valid = 0u;
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    const int j = j0 + 32 * i;
    key[i] = 0u;
    if (i < n_keys && j < n_v) {
      valid |= 1u << i;
      if (p.random_keys) {
        // random selector: the key of token j is the top 24 bits of a Philox word, as an fp32 value
        const float r = (float)(philox4x32_10_word0((uint32_t)j, (uint32_t)sq.seq_index, p.seed_lo, p.seed_hi) >> 8);
        key[i] = __float_as_uint(r) | 0x80000000u;
      } else {
        const uint32_t u = __float_as_uint(__ldcg(p.scores + sq.score_off + j));
        key[i] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
      }
    }
  }

  uint32_t thr = 0u;                   // selected: keys above thr, and the first k_rem keys equal to it
  int k_rem = 0;
  int parity = 0;
  bool have_thr = false;

  // ---- the keys' range: the first pass then spreads them over its 256 digits (the leading bits of
  // the scores of one request are nearly all the same, and its atomics would collide)
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    if ((valid >> i) & 1u) {
      kmin = min(kmin, key[i]);
      kmax = max(kmax, key[i]);
    }
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) {
    sm.wmin[warp] = kmin;
    sm.wmax[warp] = kmax;
  }
  cluster.sync();                      // every CTA of the cluster runs: its shared memory may be written
  if (tid < n_cta) {
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) {
      kmin = min(kmin, sm.wmin[w]);
      kmax = max(kmax, sm.wmax[w]);
    }
    *cluster.map_shared_rank(&sm.rmin[rank], tid) = kmin;
    *cluster.map_shared_rank(&sm.rmax[rank], tid) = kmax;
  }
  cluster.sync();
#pragma unroll
  for (int c = 0; c < kSelMaxCluster; ++c) {
    if (c < n_cta) {
      kmin = min(kmin, sm.rmin[c]);
      kmax = max(kmax, sm.rmax[c]);
    }
  }
  const int top_shift = max(0, 24 - __clz((kmax - kmin) | 1u));   // (kmax - kmin) >> top_shift < 256

  // ---- 0. Top-P: the Stage-I count from the score mass
  if (sq.lambda_pm >= 0) {
    int c = 0;
    unsigned long long target = (unsigned long long)sq.lambda_pm;      // x total mass after the first pass
    if (target > 0ull) {
      uint32_t base = kmin;
      int shift = top_shift;
      sel_pass<KEYS, true, true>(sm, cluster, key, valid, base, 256u, shift, parity, target, 0ull, 0);
      parity ^= 1;
      if (sm.digit >= 0) {
        base += (uint32_t)sm.digit << shift;
        // a digit with a single key is that key: its lower bits need no look
        while (shift > 0 && sm.same > 1) {
          const uint32_t n_digits = shift >= 8 ? 256u : 1u << shift;
          shift = max(0, shift - 8);
          const int n_above = sm.count;    // count and mass of the keys ranked before every live key
          const unsigned long long above = sm.mass_above;
          sel_pass<KEYS, true, false>(sm, cluster, key, valid, base, n_digits, shift, parity, target, above,
                                      n_above);
          base += (uint32_t)sm.digit << shift;
          parity ^= 1;
        }
        if (sm.same == 1) {
          c = sm.count + 1;
          thr = base - 1u;                 // (base > 0: the keys of scores that have a mass are large)
          k_rem = 0;
        } else {
          // every key equal to base carries the same mass: take as many as still needed
          const unsigned long long q = key_mass(base);
          const unsigned long long need = target - 1000ull * sm.mass_above;      // > 0: that mass alone does not reach
          const unsigned long long e = (need + 1000ull * q - 1ull) / (1000ull * q);
          c = sm.count + (int)e;
          thr = base;
          k_rem = (int)e;
        }
        have_thr = c <= k_total;           // the descent has found the c-th largest key on its way
      }
    }
    k1 = c < k_total ? c : k_total;
    if (rank == 0 && tid == 0 && p.k1_out) p.k1_out[seq + p.k1_out_base] = k1;
  }

  // ---- 1. radix select of the k1-th largest key
  if (k1 > 0 && !have_thr) {
    uint32_t base = kmin;
    uint32_t n_digits = 256u;
    int shift = top_shift, n_above = 0;
    unsigned long long want = (unsigned long long)k1;
    while (true) {
      sel_pass<KEYS, false, false>(sm, cluster, key, valid, base, n_digits, shift, parity, want, 0ull, n_above);
      base += (uint32_t)sm.digit << shift;
      n_above = sm.count;
      parity ^= 1;
      thr = base;
      k_rem = k1 - n_above;                // wanted among the live keys
      if (k_rem == sm.same) {              // all of them: no need to look at the lower bits
        thr = base - 1u;
        k_rem = 0;
        if (base == 0u) {
          thr = 0u;
          k_rem = n_v;
        }
        break;
      }
      if (shift == 0) break;
      n_digits = shift >= 8 ? 256u : 1u << shift;
      shift = max(0, shift - 8);
    }
  }

  // ---- 2. counts below and at the threshold, over the cluster
  int n_less = 0, n_eq = 0;
  {
    __syncthreads();                       // sm.wcount is still read by the scans above
#pragma unroll
    for (int i = 0; i < KEYS; ++i) {
      if (i < n_keys) {
        const bool ok = (valid >> i) & 1u;
        n_eq += __popc(__ballot_sync(0xffffffffu, ok && k1 > 0 && key[i] == thr));
        n_less += __popc(__ballot_sync(0xffffffffu, ok && (k1 <= 0 || key[i] < thr)));
      }
    }
    if (lane == 0) {                       // a warp's two counts in one word: at most 448 tokens each
      sm.wcount[warp] = (n_less << 16) | n_eq;
    }
    __syncthreads();
    if (tid < n_cta) {
      int l = 0, e = 0;
#pragma unroll
      for (int w = 0; w < kSelWarps; ++w) {
        l += sm.wcount[w] >> 16;
        e += sm.wcount[w] & 0xffff;
      }
      *cluster.map_shared_rank(&sm.less[rank], tid) = l;
      *cluster.map_shared_rank(&sm.equal[rank], tid) = e;
    }
    cluster.sync();
  }
  // keys equal to the threshold before this warp, and unselected tokens before it (and in all)
  int eq_rank = 0, run = 0, m_total = 0;
  {
    int e_all = 0, l_all = 0;
#pragma unroll
    for (int c = 0; c < kSelMaxCluster; ++c) {
      const int ec = c < n_cta ? sm.equal[c] : 0, lc = c < n_cta ? sm.less[c] : 0;
      if (c < rank) {
        eq_rank += ec;
        run += lc;
      }
      e_all += ec;
      l_all += lc;
    }
#pragma unroll
    for (int w = 0; w < kSelWarps - 1; ++w) {
      if (w < warp) {
        run += sm.wcount[w] >> 16;
        eq_rank += sm.wcount[w] & 0xffff;
      }
    }
    run += max(0, eq_rank - k_rem);        // ties past the k_rem-th stay unselected
    m_total = l_all + max(0, e_all - k_rem);
  }
  // ---- per token: selected?, and the unselected tokens before it; the same before each frame
  uint32_t sel_bits = 0u;
  int before[KEYS];
  const uint32_t below = (1u << lane) - 1u;
  const int f0 = j0 < n_v ? j0 / T : 0;    // frame of the thread's first token; later ones count up from it
  {
    int f = f0, f_end = (f0 + 1) * T;      // (n_v + 32 fits an int)
#pragma unroll
    for (int i = 0; i < KEYS; ++i) {
      before[i] = 0;
      if (i < n_keys) {
        const bool ok = (valid >> i) & 1u;
        const bool eq = ok && k1 > 0 && key[i] == thr;
        const uint32_t eqs = __ballot_sync(0xffffffffu, eq);
        const bool sel = ok && k1 > 0 && (key[i] > thr || (eq && eq_rank + __popc(eqs & below) < k_rem));
        eq_rank += __popc(eqs);
        const uint32_t uns = __ballot_sync(0xffffffffu, ok && !sel);
        before[i] = run + __popc(uns & below);
        run += __popc(uns);
        if (sel) sel_bits |= 1u << i;
        if (ok) {
          const int j = j0 + 32 * i;
          while (j >= f_end) {
            ++f;
            f_end += T;
          }
          if (j == f_end - T)
            for (int c = 0; c < n_cta; ++c) *cluster.map_shared_rank(&sm.cf[f], c) = before[i];
        }
      }
    }
  }
  if (tid == 0) sm.cf[F] = m_total;
  cluster.sync();                          // the last access to another CTA's shared memory is complete
  // ---- 3. Stage II pick test and the kept tokens' places
  // All products below stay under 2^32: counts are at most n_v <= 57 344 tokens.
  const uint32_t n_u = (uint32_t)(k_total - k1);
  if (n_u > 0u) {                          // then m_total >= n_u > 0
    for (int f = tid; f <= F; f += kSelThreads) sm.quota[f] = ((uint32_t)sm.cf[f] * n_u) / (uint32_t)m_total;
    __syncthreads();
  }
  int32_t* const out = p.kept_idx + sq.kept_off;
  int f = f0, f_end = (f0 + 1) * T, f_have = -1;
  uint32_t c0 = 0u, c_f = 0u, q0 = 0u, n_f = 0u;
  float ratio = 0.f;
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    if (!((valid >> i) & 1u)) continue;
    const bool sel = (sel_bits >> i) & 1u;
    const int j = j0 + 32 * i;
    uint32_t picks = 0u;                   // Stage-II picks among the tokens before this one
    bool keep = sel;
    if (n_u > 0u) {
      while (j >= f_end) {
        ++f;
        f_end += T;
      }
      if (f != f_have) {
        f_have = f;
        c0 = (uint32_t)sm.cf[f];
        c_f = (uint32_t)sm.cf[f + 1] - c0;
        q0 = sm.quota[f];
        n_f = sm.quota[f + 1] - q0;
        ratio = __fdividef((float)n_f, (float)max(c_f, 1u));
      }
      picks = q0;
      if (n_f > 0u) {
        // The picks of a frame have ranks floor(t c_f / n_f): t = ceil(r n_f / c_f) of them lie below
        // rank r.  The quotient in fp32 is within one of it (t <= 57 344, relative error below 2^-20)
        // and is set right by exact products; one integer division per token cost a third of the kernel.
        const uint32_t r = (uint32_t)before[i] - c0, rn = r * n_f;
        uint32_t t = (uint32_t)((float)r * ratio);
        if (t * c_f < rn) ++t;
        if (t * c_f < rn) ++t;
        if (t > 0u && (t - 1u) * c_f >= rn) --t;
        picks += min(t, n_f);
        if (!sel) keep = t < n_f && t * c_f < rn + n_f;    // floor(t c_f / n_f) == r (t c_f >= r n_f holds)
      }
    }
    if (keep) out[(uint32_t)(j - before[i]) + picks] = j;
  }
}

// window / frame selectors: closed-form index lists, one CTA per sequence
struct RangeParams {
  int32_t* kept_idx;
  int32_t* kept_n_out;
  int32_t mode, tokens_per_frame, batch0;
  int32_t n_frames[kSelMaxBatch], k_total[kSelMaxBatch], kept_off[kSelMaxBatch];
};

__global__ void baseline_ranges_kernel(const __grid_constant__ RangeParams p) {
  pdl_launch_next();
  pdl_wait();
  const int i = blockIdx.x;
  const int F = p.n_frames[i], T = p.tokens_per_frame, K = p.k_total[i], n_v = F * T;
  int32_t* out = p.kept_idx + p.kept_off[i];
  int n = K;
  if (p.mode == SPECVLM_SEL_FRAMES) {
    const int nf = K / T;                       // whole frames that fit the budget
    n = nf * T;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      const int fi = j / T;
      out[j] = (int)(((long long)fi * F) / nf) * T + (j - fi * T);
    }
  } else {
    const int start = p.mode == SPECVLM_SEL_WINDOW_FRONT ? 0 : (p.mode == SPECVLM_SEL_WINDOW_END ? n_v - K : (n_v - K) / 2);
    for (int j = threadIdx.x; j < n; j += blockDim.x) out[j] = start + j;
  }
  if (threadIdx.x == 0 && p.kept_n_out) p.kept_n_out[p.batch0 + i] = n;
}

template <int KEYS>
static int32_t launch_select(const SelParams& p, int n_seq, int n_cta, cudaStream_t st) {
  static std::atomic<uint64_t> attr_done{0};
  if (!smem_attr_once(attr_done, reinterpret_cast<const void*>(select_kernel<KEYS>), (int)sizeof(SelSmem)))
    return SPECVLM_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_seq * n_cta));
  cfg.blockDim = dim3(kSelThreads);
  cfg.dynamicSmemBytes = sizeof(SelSmem);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)n_cta;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, select_kernel<KEYS>, p) != cudaSuccess) return SPECVLM_ERR_CUDA;
  return launch_status();
}

// CTAs per sequence.  More CTAs mean fewer keys per thread but a dearer exchange per pass.  One
// sequence, 1 / 2 / 4 / 8 CTAs: 784 tokens 7.3 / 6.8 / 7.1 / 7.6 us (Top-P 8.8 / 8.4 / 9.0 / 10.2),
// 1568 tokens 9.3 / 7.6 / 7.2 / 7.6, 3136 tokens 11.4 / 8.6 / 6.9 / 6.5, 6272 tokens 17.2 / 12.8 / 10.0 / 8.5,
// 25 088 tokens - / - / 18.0 / 14.3.  Above 6 x 8 x 512 tokens a CTA fills an SM, and more than
// about a dozen clusters of eight no longer run side by side: 16 sequences of 25 088 tokens take
// 26.6 us with eight CTAs each, 19.6 us with four (which hold up to 4 x 7168).
static int select_cluster(int64_t max_tokens, int n_seq) {
  if (max_tokens <= 2048) return 2;
  if (n_seq > 12 && max_tokens > 6 * kSelMaxCluster * kSelThreads && max_tokens <= 4 * kSelMaxKeys * kSelThreads) return 4;
  return kSelMaxCluster;
}

static int32_t select_common(const float* scores, const int32_t* video_cu, const int32_t* n_frames,
                             int32_t tokens_per_frame, const int32_t* k_stage1, const int32_t* lambda_permille,
                             const int32_t* k_total, const int32_t* kept_cu, int32_t batch, int32_t* kept_idx,
                             int32_t* k1_out, void* stream, bool random_keys = false, uint64_t seed = 0) {
  if ((!scores && !random_keys) || !video_cu || !n_frames || (!k_stage1 && !lambda_permille) || !k_total || !kept_cu || !kept_idx ||
      batch < 1 || tokens_per_frame < 1)
    return SPECVLM_ERR_INVALID_ARG;
  int64_t max_tokens = 0;
  for (int b = 0; b < batch; ++b) {
    const int64_t n_v = (int64_t)n_frames[b] * tokens_per_frame;
    if (n_frames[b] < 1 || n_frames[b] > kSelMaxFrames || n_v > kSelMaxCluster * kSelThreads * kSelMaxKeys)
      return SPECVLM_ERR_UNSUPPORTED_SHAPE;
    if (k_total[b] < 0 || k_total[b] > n_v) return SPECVLM_ERR_INVALID_ARG;
    if (lambda_permille) {
      if (lambda_permille[b] < 0 || lambda_permille[b] > 1000) return SPECVLM_ERR_INVALID_ARG;
    } else if (k_stage1[b] < 0 || k_stage1[b] > k_total[b]) {
      return SPECVLM_ERR_INVALID_ARG;
    }
    if ((!random_keys && video_cu[b + 1] - video_cu[b] < n_v) || kept_cu[b + 1] - kept_cu[b] < k_total[b])
      return SPECVLM_ERR_INVALID_ARG;
    if (n_v > max_tokens) max_tokens = n_v;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int n_cta = select_cluster(max_tokens, batch < kSelMaxBatch ? batch : kSelMaxBatch);
  SelParams p;
  p.scores = scores;
  p.kept_idx = kept_idx;
  p.k1_out = k1_out;
  p.tokens_per_frame = tokens_per_frame;
  p.random_keys = random_keys ? 1 : 0;
  p.seed_lo = (uint32_t)(seed & 0xffffffffu);
  p.seed_hi = (uint32_t)(seed >> 32);
  for (int b0 = 0; b0 < batch; b0 += kSelMaxBatch) {
    const int nb = batch - b0 < kSelMaxBatch ? batch - b0 : kSelMaxBatch;
    p.k1_out_base = b0;
    for (int i = 0; i < nb; ++i) {
      const int b = b0 + i;
      p.seq[i] = SelSeq{video_cu[b], n_frames[b], lambda_permille ? 0 : k_stage1[b], k_total[b], kept_cu[b],
                        lambda_permille ? lambda_permille[b] : -1, b};
    }
    const int32_t rc = max_tokens <= 2 * n_cta * kSelThreads   ? launch_select<2>(p, nb, n_cta, st)
                       : max_tokens <= 6 * n_cta * kSelThreads ? launch_select<6>(p, nb, n_cta, st)
                                                               : launch_select<kSelMaxKeys>(p, nb, n_cta, st);
    if (rc != SPECVLM_OK) return rc;
  }
  return SPECVLM_OK;
}

}  // namespace specvlm

using namespace specvlm;

extern "C" int32_t specvlm_select(const float* scores, const int32_t* video_cu, const int32_t* n_frames,
                                  int32_t tokens_per_frame, const int32_t* k_stage1,
                                  const int32_t* k_total, const int32_t* kept_cu, int32_t batch,
                                  int32_t* kept_idx, int32_t* d_status, void* stream) {
  NvtxRange nvtx_range(__func__);
  (void)d_status;
  if (!k_stage1) return SPECVLM_ERR_INVALID_ARG;
  return select_common(scores, video_cu, n_frames, tokens_per_frame, k_stage1, nullptr, k_total, kept_cu, batch,
                       kept_idx, nullptr, stream);
}

extern "C" int32_t specvlm_select_top_p(const float* scores, const int32_t* video_cu, const int32_t* n_frames,
                                        int32_t tokens_per_frame, const int32_t* lambda_permille,
                                        const int32_t* k_total, const int32_t* kept_cu, int32_t batch,
                                        int32_t* kept_idx, int32_t* k_stage1_out_or_null, int32_t* d_status,
                                        void* stream) {
  NvtxRange nvtx_range(__func__);
  (void)d_status;
  if (!lambda_permille) return SPECVLM_ERR_INVALID_ARG;
  return select_common(scores, video_cu, n_frames, tokens_per_frame, nullptr, lambda_permille, k_total, kept_cu,
                       batch, kept_idx, k_stage1_out_or_null, stream);
}

extern "C" int32_t specvlm_select_baseline(int32_t mode, uint64_t seed, const int32_t* n_frames,
                                           int32_t tokens_per_frame, const int32_t* k_total,
                                           const int32_t* kept_cu, int32_t batch, int32_t* kept_idx,
                                           int32_t* kept_n_out_or_null, void* stream) {
  NvtxRange nvtx_range(__func__);
  if (!n_frames || !k_total || !kept_cu || !kept_idx || batch < 1 || tokens_per_frame < 1)
    return SPECVLM_ERR_INVALID_ARG;
  if (mode < SPECVLM_SEL_WINDOW_FRONT || mode > SPECVLM_SEL_RANDOM) return SPECVLM_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (mode == SPECVLM_SEL_RANDOM) {
    // the k_total largest Philox keys: the selection kernel with keys in place of scores and
    // Stage I taking the whole budget
    int32_t rc = select_common(nullptr, kept_cu /*unused*/, n_frames, tokens_per_frame, k_total, nullptr, k_total,
                               kept_cu, batch, kept_idx, nullptr, stream, true, seed);
    if (rc != SPECVLM_OK || !kept_n_out_or_null) return rc;
    return cudaMemcpyAsync(kept_n_out_or_null, k_total, (size_t)batch * sizeof(int32_t), cudaMemcpyHostToDevice, st) ==
                   cudaSuccess
               ? SPECVLM_OK
               : SPECVLM_ERR_CUDA;
  }
  RangeParams p;
  p.kept_idx = kept_idx;
  p.kept_n_out = kept_n_out_or_null;
  p.mode = mode;
  p.tokens_per_frame = tokens_per_frame;
  for (int b0 = 0; b0 < batch; b0 += kSelMaxBatch) {
    const int nb = batch - b0 < kSelMaxBatch ? batch - b0 : kSelMaxBatch;
    p.batch0 = b0;
    for (int i = 0; i < nb; ++i) {
      const int b = b0 + i;
      const int64_t n_v = (int64_t)n_frames[b] * tokens_per_frame;
      if (n_frames[b] < 1 || n_v > 0x7fffffff || k_total[b] < 0 || k_total[b] > n_v ||
          kept_cu[b + 1] - kept_cu[b] < k_total[b])
        return SPECVLM_ERR_INVALID_ARG;
      p.n_frames[i] = n_frames[b];
      p.k_total[i] = k_total[b];
      p.kept_off[i] = kept_cu[b];
    }
    const int32_t rc = launch_after(baseline_ranges_kernel, dim3((unsigned)nb), dim3(256), 0, st, p);
    if (rc != SPECVLM_OK) return rc;
  }
  return SPECVLM_OK;
}
