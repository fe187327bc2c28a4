// Label-segmented adjacency: besides the id-sorted rows, the library keeps
// every row ordered by (neighbour label, neighbour id), so the neighbours of a
// vertex with one label form one contiguous, id-sorted segment.
#pragma once

#include "kernels.cuh"

namespace gsm {

// The segment of label l in a row [b, e) of at most 254 entries, from the
// neighbour label counts (none of them saturated): its start is the sum of the
// counts of the labels before l.  The counts of a vertex are whole 8-byte
// words (nlc_stride), loaded together, so the lookup is one load deep; two
// binary searches of the labels are 2 log2(e - b).
__device__ __forceinline__ int2 counted_segment(const GraphDev &g, int32_t x, int32_t l,
                                                int32_t b) {
  const uint2 *row = reinterpret_cast<const uint2 *>(g.nlc + (int64_t)x * g.nlc_stride);
  uint32_t before = 0, own = 0;
  for (int32_t w = 0; w <= l >> 3; ++w) {
    uint2 c = __ldg(row + w);
    if (w == l >> 3) {  // keep the bytes before l's
      const uint32_t byte = l & 7;
      own = ((byte < 4 ? c.x : c.y) >> (8 * (byte & 3))) & 0xffu;
      c.x = byte >= 4 ? c.x : c.x & ((1u << (8 * byte)) - 1u);
      c.y = byte >= 4 ? c.y & ((1u << (8 * (byte - 4))) - 1u) : 0u;
    }
    before = __dp4a(c.x, 0x01010101u, before);
    before = __dp4a(c.y, 0x01010101u, before);
  }
  return make_int2(b + (int32_t)before, b + (int32_t)(before + own));
}
constexpr int32_t kCountedRow = 254;

// [first, second) = the neighbours of x with label l (rows of lcol are
// ordered by (label, id), so they are one contiguous, id-sorted segment): from
// a hub's segment table, the neighbour label counts of a short row, or two
// binary searches.
__device__ __forceinline__ int2 label_segment(const GraphDev &g, int32_t x, int32_t l) {
  if (g.num_labels > 1 && g.hub_seg) {  // a hub: its segment table
    const int32_t h = __ldg(g.hub + x);
    if (h >= 0) {
      const int32_t *t = g.hub_seg + (size_t)h * (g.num_labels + 1) + l;
      return make_int2(__ldg(t), __ldg(t + 1));
    }
  }
  const int32_t b = __ldg(g.rp + x), e = __ldg(g.rp + x + 1);
  if (g.num_labels == 1) return make_int2(b, e);
  if (g.nlc && e - b <= kCountedRow) return counted_segment(g, x, l, b);
  int32_t lo = b, len = e - b;  // first entry with label >= l
  while (len > 0) {
    const int32_t half = len >> 1;
    if (__ldg(g.llab + lo + half) < l) {
      lo += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  int32_t hi = lo;
  len = e - lo;  // first entry with label > l
  while (len > 0) {
    const int32_t half = len >> 1;
    if (__ldg(g.llab + hi + half) <= l) {
      hi += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  return make_int2(lo, hi);
}

// The part of an id-sorted segment of lcol with ids in [lo, hi).
__device__ __forceinline__ int2 cut_segment(const GraphDev &g, int2 seg, int32_t lo, int32_t hi) {
  int32_t a = seg.x, len = lo > 0 ? seg.y - seg.x : 0;
  while (len > 0) {
    const int32_t half = len >> 1;
    if (__ldg(g.lcol + a + half) < lo) {
      a += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  if (hi >= g.n) return make_int2(a, seg.y);
  int32_t b = a;
  len = seg.y - a;
  while (len > 0) {
    const int32_t half = len >> 1;
    if (__ldg(g.lcol + b + half) < hi) {
      b += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  return make_int2(a, b);
}

// Is y (label ly) in x's row?  One binary search on the (label, id) order: the
// part that can hold y is halved with its longer side kept, so that its length
// does not depend on what was read: a load, a compare and an add a step (the
// 5-cycle listing of R-MAT 20 spends half its instructions here: 1,834 ->
// 1,721 us with the same form in group_contains).
__device__ __forceinline__ bool row_search(const GraphDev &g, int32_t lo, int32_t e, int32_t ly,
                                           int32_t y) {
  int32_t len = e - lo;
  if (len <= 0) return false;
  if (g.num_labels == 1) {  // one label: a plain search of the id-sorted row
    while (len > 1) {
      const int32_t half = len >> 1;
      if (__ldg(g.lcol + lo + half - 1) < y) lo += half;
      len -= half;
    }
    return __ldg(g.lcol + lo) == y;
  }
  while (len > 1) {
    const int32_t half = len >> 1;
    const int32_t ml = __ldg(g.llab + lo + half - 1);
    if (ml < ly || (ml == ly && __ldg(g.lcol + lo + half - 1) < y)) lo += half;
    len -= half;
  }
  return __ldg(g.llab + lo) == ly && __ldg(g.lcol + lo) == y;
}

__device__ __forceinline__ bool hub_bit(const GraphDev &g, int32_t h, int32_t v) {
  return (__ldg(g.hub_bits + (size_t)h * g.hub_words + (v >> 5)) >> (v & 31)) & 1u;
}

// Is w (label l) in the row [b, e) of x, no hub, when x is asked about few
// candidates in a row (at most kFewCandidates)?  Then x's row does not come to
// stay in L1, a search of n entries reads log2(n) random L2 sectors, and their
// rate bounds the level: one bit of w's bitmap when w is a hub, else the
// search of the shorter of the two rows (adjacency is symmetric).  The last
// level of a 5-cycle listing on R-MAT 20 (4 candidates a row, mostly hubs)
// went from 3.9 to 2.0 ms for 67 M checks; taken for all rows, the triangle
// count (146 candidates a row) went from 20.8 to 31.1 ms, hence the line.
constexpr int32_t kFewCandidates = 16;
constexpr int32_t kLongRow = 32;  // entries: up to a line of 128 bytes one side is as good
__device__ __forceinline__ bool row_contains_few(const GraphDev &g, int32_t x, int32_t b,
                                                 int32_t e, int32_t l, int32_t w) {
  if (g.hub) {
    const int32_t h = __ldg(g.hub + w);
    if (h >= 0) return hub_bit(g, h, x);
  }
  if (e - b > kLongRow) {
    const int32_t wb = __ldg(g.rp + w), we = __ldg(g.rp + w + 1);
    if (we - wb < e - b) return row_search(g, wb, we, __ldg(g.lab + x), x);
  }
  return row_search(g, b, e, l, w);
}

// Is w (label l) a neighbour of x?  One bit of x's adjacency bitmap when x is
// a hub, else a binary search of x's row (few: row_contains_few).
__device__ __forceinline__ bool row_contains_l(const GraphDev &g, int32_t x, int32_t l, int32_t w,
                                               bool few = false) {
  if (!GSM_IN_BOUNDS(g.dbg, x >= 0 && x < g.n, kDbgNeighbour)) return false;
  if (g.hub) {
    const int32_t h = __ldg(g.hub + x);
    if (h >= 0) return hub_bit(g, h, w);
  }
  const int32_t b = __ldg(g.rp + x), e = __ldg(g.rp + x + 1);
  return few && !g.hub_lo ? row_contains_few(g, x, b, e, l, w) : row_search(g, b, e, l, w);
}

}  // namespace gsm
