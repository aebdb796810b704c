// Work partition of the persistent attention kernel.  Plain C++ (no CUDA types) so that the same
// functions run on the device and in a host unit test.
//
// An "item" is one (layer, sequence, KV head); it owns ceil(seq_len / 64) K/V tiles.  All tiles of
// all items form one flat list ordered by (layer, sequence, KV head, tile).  CTA c of n streams the
// contiguous slice [slice_begin(c), slice_begin(c + 1)) of that list, so every CTA moves the same
// number of tiles (+-1) and an item is cut only where a slice boundary falls inside it.  A CTA's
// slice is a sequence of "segments" (maximal runs inside one item); only its first and its last
// segment can be partial, which bounds the scratch memory to two partial results per CTA.
// Where the items are fewer than the CTAs the slices keep to item boundaries instead (aligned_slice): one
// segment a CTA, the tiles as even as the items allow.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define SPECVLM_HD __host__ __device__ __forceinline__
#else
#define SPECVLM_HD inline
#endif

namespace specvlm {

constexpr int kSchedMaxBatch = 127;     // sequences per call (their tile counts live in shared memory)
constexpr int kSchedMinTilesPerCta = 2;   // below this a slice is not worth a CTA of its own (a tile per softmax group)

// Number of CTAs that get a non-empty slice.
SPECVLM_HD int sched_active_ctas(int64_t total_tiles, int grid) {
  int64_t n = (total_tiles + kSchedMinTilesPerCta - 1) / kSchedMinTilesPerCta;
  if (n > grid) n = grid;
  if (n < 1) n = 1;
  return (int)n;
}

SPECVLM_HD int64_t slice_begin(int c, int n_active, int64_t total_tiles) {
  return (int64_t)c * total_tiles / n_active;
}

// The CTA whose slice holds flat tile f (0 <= f < total_tiles).
SPECVLM_HD int slice_owner(int64_t f, int n_active, int64_t total_tiles) {
  return (int)(((f + 1) * n_active - 1) / total_tiles);
}

struct Segment {
  int layer, b, g;        // the item
  int item;               // (layer * batch + b) * n_kv_heads + g
  int tile0;              // first tile of the segment inside the item
  int n_tiles;            // tiles of the segment
  int item_tiles;         // tiles of the whole item
  int64_t item_begin;     // flat index of the item's first tile
};

// Locates flat tile f and cuts the segment at `slice_end`.  prefix[b] = tiles of sequences < b
// (prefix[batch] = tiles of one KV head of one layer); every sequence holding f has >= 1 tile.
SPECVLM_HD Segment segment_at(int64_t f, int64_t slice_end, const int* prefix, int batch, int n_kv_heads) {
  Segment s;
  const int64_t per_layer = (int64_t)n_kv_heads * prefix[batch];
  s.layer = (int)(f / per_layer);
  const int64_t rem = f - (int64_t)s.layer * per_layer;
  int lo = 0, hi = batch - 1;             // last b with n_kv_heads * prefix[b] <= rem
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((int64_t)n_kv_heads * prefix[mid] <= rem) lo = mid; else hi = mid - 1;
  }
  s.b = lo;
  s.item_tiles = prefix[lo + 1] - prefix[lo];
  const int64_t rem2 = rem - (int64_t)n_kv_heads * prefix[lo];
  s.g = (int)(rem2 / s.item_tiles);
  s.tile0 = (int)(rem2 - (int64_t)s.g * s.item_tiles);
  s.item = (s.layer * batch + s.b) * n_kv_heads + s.g;
  s.item_begin = f - s.tile0;
  int64_t n = s.item_tiles - s.tile0;
  if (n > slice_end - f) n = slice_end - f;
  s.n_tiles = (int)n;
  return s;
}

// CTAs that a caller's scratch has room for, of a launch of up to total_tiles tiles on at most `grid`.  Slices that keep to
// item boundaries take up to items * ceil(t / 2) CTAs for items of t tiles, at most twice the even split's; whether they are
// used depends on how the tiles fall on items.  The room depends on the number of tiles alone and never falls as it rises,
// so that a workspace sized for the longest sequences and the largest batch serves every shorter and smaller call.
SPECVLM_HD int sched_scratch_ctas(int64_t total_tiles, int grid) {
  const int even = sched_active_ctas(total_tiles, grid);
  return 2 * even < grid ? 2 * even : grid;
}

// Where the items are fewer than the CTAs, slices that keep to item boundaries: an item of t tiles gets ceil(t / q)
// CTAs of its own, as equal as its tiles allow.  No CTA then works on two items, one after the other (with a few tiles a
// CTA the second one's hand-over is as long as its tiles).  part_prefix[b] = CTAs of one KV head of the sequences < b.
// The arithmetic is in 32 bits (it is on the way to the first tile): total < 2^31.
constexpr int kSchedAlignedBatch = 32;
constexpr int kSchedAlignedTries = 2;     // q from the smallest that could fit; more tiles a CTA are not worth it

// Tiles a CTA from which to look for such a split.
SPECVLM_HD int aligned_q_first(int total_tiles, int grid) {
  const int q = (int)(((uint32_t)total_tiles + (uint32_t)grid - 1u) / (uint32_t)grid);
  return q > kSchedMinTilesPerCta ? q : kSchedMinTilesPerCta;
}

// The slice of CTA c, one segment, and its item's CTAs in `parts`; false if c has no work.
SPECVLM_HD bool aligned_slice(int c, const int* prefix, const int* part_prefix, int batch, int n_layers, int n_kv_heads,
                              Segment* s, int* parts) {
  const int per_layer = n_kv_heads * part_prefix[batch];
  if (per_layer == 0 || c >= n_layers * per_layer) return false;
  const int layer = n_layers == 1 ? 0 : (int)((uint32_t)c / (uint32_t)per_layer), rem = c - layer * per_layer;
  int lo = 0, hi = batch - 1;             // last b with n_kv_heads * part_prefix[b] <= rem
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (n_kv_heads * part_prefix[mid] <= rem) lo = mid; else hi = mid - 1;
  }
  const int n = part_prefix[lo + 1] - part_prefix[lo], t = prefix[lo + 1] - prefix[lo];
  const int rem2 = rem - n_kv_heads * part_prefix[lo], g = (int)((uint32_t)rem2 / (uint32_t)n), part = rem2 - g * n;
  s->layer = layer;
  s->b = lo;
  s->g = g;
  s->item = (layer * batch + lo) * n_kv_heads + g;
  s->item_tiles = t;
  s->item_begin = (int64_t)n_kv_heads * ((int64_t)layer * prefix[batch] + prefix[lo]) + (int64_t)g * t;
  // part * t / n and (part + 1) * t / n: the first t % n parts' worth of remainders falls evenly
  const int base = (int)((uint32_t)t / (uint32_t)n), rest = t - base * n;
  s->tile0 = part * base + (int)((uint32_t)(part * rest) / (uint32_t)n);
  s->n_tiles = (part + 1) * base + (int)((uint32_t)((part + 1) * rest) / (uint32_t)n) - s->tile0;
  *parts = n;
  return true;
}

// Scratch slot of the partial result that CTA c holds for the item starting at flat tile item_begin:
// slot 2c when the item is the first segment of c's slice, 2c + 1 otherwise (then it is the last).
SPECVLM_HD int partial_slot(int c, int64_t cta_slice_begin, int64_t item_begin) {
  return cta_slice_begin >= item_begin ? 2 * c : 2 * c + 1;
}

// Walks a CTA's slice segment by segment, in flat order.  (Taking the item that the slice end cuts
// first, so that the merges of cut items happen early, was measured slower: the partial results'
// stores and fences then wait behind the full-rate K/V streams of the other CTAs.)
struct SliceCursor {
  int64_t f, end;
  Segment sg;
  int j;          // tile inside the current segment
  int seg_idx;    // segments entered so far - 1
  SPECVLM_HD void start(int64_t begin, int64_t end_, const int* prefix, int batch, int hkv) {
    f = begin;
    end = end_;
    j = 0;
    seg_idx = 0;
    if (f < end) sg = segment_at(f, end, prefix, batch, hkv);
  }
  // the same with the slice's first segment at hand
  SPECVLM_HD void start(int64_t begin, int64_t end_, const Segment& first) {
    f = begin;
    end = end_;
    j = 0;
    seg_idx = 0;
    sg = first;
  }
  SPECVLM_HD bool done() const { return f >= end; }
  SPECVLM_HD bool last_of_segment() const { return j == sg.n_tiles - 1; }
  SPECVLM_HD void next_tile(const int* prefix, int batch, int hkv) {
    ++f;
    if (++j == sg.n_tiles) next_segment(prefix, batch, hkv);
  }
  SPECVLM_HD void next_segment(const int* prefix, int batch, int hkv) {
    f = sg.item_begin + sg.tile0 + sg.n_tiles;
    j = 0;
    ++seg_idx;
    if (f < end) sg = segment_at(f, end, prefix, batch, hkv);
  }
};

}  // namespace specvlm
