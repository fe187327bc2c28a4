// Device helpers of the verification kernels (extend count, write, single
// pass): tile row staging, the candidate check and the row writer.
#pragma once

#include <type_traits>

#include "kernels.cuh"
#include "segments.cuh"

namespace gsm {

__device__ __forceinline__ bool bitmap_has(const uint32_t *__restrict__ bm, int32_t v) {
  return (__ldg(bm + (v >> 5)) >> (v & 31)) & 1u;
}

// Inside one launch every index is 32-bit: candidates are numbered locally
// from wa (a launch covers fewer than 2^30), rows and frontier elements stay
// below 2^31 (the host code chunks frontiers to that), only output addresses of
// the final rows are 64-bit.
//
// A tile's rows [r0, r0+span): their work offsets, relative to wa, are staged
// in shared memory when they fit (span <= tile items: always, unless rows
// without work pile up); items then find their row by binary search there,
// otherwise in the global offsets.
struct TileRows {
  int32_t r0;
  int32_t span;
  bool staged;
};

__device__ __forceinline__ TileRows stage_rows(const int64_t *__restrict__ woff,
                                               const int32_t *__restrict__ tile_row, int64_t wa,
                                               int32_t tile_items, int32_t *s_woff,
                                               int32_t tile) {
  TileRows t;
  t.r0 = tile_row[tile];
  t.span = tile_row[tile + 1] + 1 - t.r0;
  t.staged = t.span <= tile_items;
  if (t.staged)
    for (int32_t j = threadIdx.x; j <= t.span; j += blockDim.x)
      s_woff[j] = (int32_t)(woff[t.r0 + j] - wa);
  __syncthreads();
  return t;
}

// Row of local item x and the local offset where that row's candidates start.
__device__ __forceinline__ int32_t item_row(const TileRows &t, const int32_t *s_woff,
                                            const int64_t *__restrict__ woff, int64_t wa,
                                            int32_t x, int32_t *row_start) {
  int32_t lo = 0, hi = t.span;  // largest j in [0, span) with offset(r0+j) <= x
  if (t.staged) {
    while (hi - lo > 1) {
      const int32_t mid = (lo + hi) >> 1;
      if (s_woff[mid] <= x) lo = mid; else hi = mid;
    }
    *row_start = s_woff[lo];
  } else {
    while (hi - lo > 1) {
      const int32_t mid = (lo + hi) >> 1;
      if (woff[t.r0 + mid] - wa <= x) lo = mid; else hi = mid;
    }
    *row_start = (int32_t)(woff[t.r0 + lo] - wa);
  }
  return t.r0 + lo;
}

// From row r0 + rr, whose candidates end at re <= x, to the row of item x, and
// where its candidates start and end.  Mostly the next; rows without work are
// stepped over (kSteps rows), longer runs by a search: bounds cut off a row's
// segment leave runs of millions (counting the 5-cycles of two low roots of
// R-MAT 20, whose symmetry orders two vertices, one thread stepped through
// most of 6.5 M rows: 237 ms, 0.56 with the search).
template <int kSteps = 4>
__device__ __forceinline__ void next_row(const TileRows &t, const int32_t *s_woff,
                                         const int64_t *__restrict__ woff, int64_t wa, int32_t x,
                                         int32_t *rr, int32_t *rs, int32_t *re) {
  auto offset = [&](int32_t j) { return t.staged ? s_woff[j] : (int32_t)(woff[t.r0 + j] - wa); };
  for (int32_t step = 0; step < kSteps; ++step) {
    ++*rr;
    *rs = *re;
    *re = offset(*rr + 1);
    if (x < *re) return;
  }
  int32_t lo = *rr + 1, hi = t.span;  // (the tile's last item lies before offset(span))
  while (hi - lo > 1) {
    const int32_t mid = (lo + hi) >> 1;
    if (offset(mid) <= x) lo = mid; else hi = mid;
  }
  *rr = lo;
  *rs = offset(lo);
  *re = offset(lo + 1);
}

// A row extended by one vertex at position i.
template <typename Row>
struct ExtendedRow {
  const Row &row;
  int32_t i, w;
  __device__ __forceinline__ int32_t operator()(int c) const { return c == i ? w : row(c); }
};

// Position c of row r of a column-major frontier (leading dimension ld).
struct ColumnRow {
  const int32_t *__restrict__ F;
  int32_t ld, r;
  __device__ __forceinline__ int32_t operator()(int c) const { return F[c * ld + r]; }
};

// Index of the parent row a written row comes from (for the sink's prefix
// ranks); -1 where the row type has none.
__device__ __forceinline__ int32_t parent_index(const ColumnRow &r) { return r.r; }
template <typename Row>
__device__ __forceinline__ int32_t parent_index(const Row &) {
  return -1;
}

// The checks of Sec. 3.2 verification that need no adjacency search, for
// candidate w of a partial embedding (row(c) = the image of pi_c): label +
// signature (bitmap of C(pi_i)) and injectivity against same-label,
// non-adjacent positions (the bounds of the new vertex were cut off its
// segment with the pivot).  A null bitmap: the segment's entries are all
// candidates.  Desc is a
// level description with the fields of LevelDesc used here (the single-query
// LevelDesc or the batched form's BatchLevel).
template <typename Desc, typename Row>
__device__ __forceinline__ bool check_local(const Desc &d, const Row &row, int32_t w) {
  if (d.bitmap && !bitmap_has(d.bitmap, w)) return false;
  for (int t = 0; t < d.ninj; ++t)
    if (row(d.inj[t]) == w) return false;
  return true;
}

// The whole one-step check: check_local plus the presence of every query
// edge to a mapped neighbour other than the pivot (row_contains_l; few: the
// row has at most kFewCandidates candidates).
template <typename Desc, typename Row>
__device__ __forceinline__ bool check_candidate(const GraphDev &g, const Desc &d,
                                                const Row &row, int32_t w, int slot,
                                                bool few) {
  if (!check_local(d, row, w)) return false;
  for (int b = 0; b < d.nb; ++b) {
    if (b == slot) continue;
    if (!row_contains_l(g, row(d.bpos[b]), d.lab, w, few)) return false;
  }
  return true;
}

// check_candidate that also adds to *probe_bytes 4 * ceil(log2 deg(x)) for
// every non-tree edge check it makes against a mapped vertex x (the bytes a
// binary search of x's row reads; the check itself may be one bitmap probe).
template <typename Desc, typename Row>
__device__ __forceinline__ bool check_candidate_probes(const GraphDev &g, const Desc &d,
                                                       const Row &row, int32_t w, int slot,
                                                       bool few, uint32_t *probe_bytes) {
  if (!check_local(d, row, w)) return false;
  for (int b = 0; b < d.nb; ++b) {
    if (b == slot) continue;
    const int32_t x = row(d.bpos[b]);
    const int32_t deg = __ldg(g.rp + x + 1) - __ldg(g.rp + x);
    *probe_bytes += deg > 1 ? 4u * (32u - __clz((uint32_t)(deg - 1))) : 0u;
    if (!row_contains_l(g, x, d.lab, w, few)) return false;
  }
  return true;
}

// The images of the leaves for one core embedding (row(c) = the image of core
// position c): the product over the groups (LeafDesc), 0 if a leaf has none.
// part(l, v) receives the partial products (l leaves placed); *over is set
// when the number exceeds 64 bits.  kLeaves: an upper bound of the leaves.
template <int kLeaves, typename Row, typename Part>
__device__ __forceinline__ unsigned long long leaf_number(const GraphDev &g, const LeafDesc &leaf,
                                                          const Row &row, bool *over,
                                                          const Part &part) {
  unsigned long long v = 1;
  bool big = false;
  int32_t a = 0;
  constexpr int kUnroll = kLeaves <= 3 ? kLeaves : 1;
#pragma unroll kUnroll
  for (int l = 0; l < kLeaves; ++l) {
    if (l >= leaf.nleaves) break;
    if (l == 0 || leaf.of[l] != leaf.of[l - 1]) {
      const LeafGroup &gr = leaf.grp[leaf.of[l]];
      const int32_t x = row(gr.pos);
      int2 seg = label_segment(g, x, gr.lab);
      if (gr.lo > 0 || gr.hi < g.n) seg = cut_segment(g, seg, gr.lo, gr.hi);
      a = seg.y - seg.x;
      for (uint32_t m = gr.in_mask; m; m &= m - 1) {
        const int32_t y = row(__ffs(m) - 1);
        a -= y >= gr.lo && y < gr.hi;
      }
      for (uint32_t m = gr.chk_mask; m && a > 0; m &= m - 1) {
        const int32_t y = row(__ffs(m) - 1);
        if (y >= gr.lo && y < gr.hi && row_contains_l(g, x, gr.lab, y)) --a;
      }
    } else {
      --a;
    }
    part(l, v);
    if (a <= 0) return 0;
    big = big || __umul64hi(v, (unsigned long long)a);
    v *= (unsigned long long)a;
  }
  *over = *over || big;
  return v;
}

// One thread's sums of the leaf numbers of core embeddings.
template <int kLeaves>
struct LeafSums {
  unsigned long long lo = 0, hi = 0;  // of the numbers' 32-bit halves
  unsigned long long part[kLeaves] = {};  // partial embeddings with l leaves placed
  bool over = false;

  template <typename Row>
  __device__ __forceinline__ void add(const GraphDev &g, const LeafDesc &leaf, const Row &row) {
    const unsigned long long v = leaf_number<kLeaves>(
        g, leaf, row, &over, [&](int l, unsigned long long x) { part[l] += x; });
    lo += (uint32_t)v;
    hi += v >> 32;
  }

  // Adds the warp's sums into the count's words (all lanes call it).
  __device__ __forceinline__ void flush(const LeafDesc &leaf, unsigned long long *total) {
    constexpr unsigned kAll = 0xffffffffu;
    const bool first = (threadIdx.x & 31) == 0;
    auto sum = [&](unsigned long long v, unsigned long long *to) {
#pragma unroll
      for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
      if (first && v) atomicAdd(to, v);
      return v;
    };
    // (a warp's own sums of fewer than 2^31 halves of 32 bits do not wrap)
    const double v = (double)sum(lo, total) + 4294967296.0 * (double)sum(hi, total + 1);
    if (first && v >= kCountSmall) atomicAdd((double *)(total + kCountApprox), v);
    if (__any_sync(kAll, over) && first) atomicOr(total + 2, 1ull);
#pragma unroll
    for (int l = 0; l < kLeaves; ++l)
      if (l < leaf.nleaves) sum(part[l], total + 3 + l);
  }
};

// Entries of w's (label, id)-ordered row scanned at most per group by the
// 2-look-ahead before it gives up (and keeps the candidate).
constexpr int32_t kLaScan = 64;

// The k-look-ahead of Sec. 3.2 for a candidate w of pi_i that passed the
// level's checks: does the partial embedding extended by w still leave room
// for the query neighbours of pi_i placed later?  For every label group t of
// those neighbours:
//   1-look-ahead: w keeps at least la_need[t] neighbours with the label that
//   are not in the row (its label segment, minus the mapped neighbours of
//   pi_i, which are adjacent to w, minus the other same-label row vertices
//   adjacent to w), since an embedding maps the group to distinct unused
//   neighbours of w;
//   2-look-ahead: at least la_need[t] of those unused neighbours are
//   candidates of some query vertex of the group (checked over the first
//   kLaScan entries of the segment; a longer segment is not pruned).
// Both conditions hold for every embedding that extends the row, so pruning
// on them never changes the result.
template <typename Row>
__device__ __forceinline__ bool lookahead_ok(const GraphDev &g, const LevelDesc &d,
                                             const Row &row, int32_t w) {
  for (int t = 0; t < d.nla; ++t) {
    const int2 seg = label_segment(g, w, d.la_lab[t]);
    int32_t avail = seg.y - seg.x - d.la_known[t];
    for (uint32_t m = d.la_pos[t]; m; m &= m - 1) {
      const int32_t x = row(__ffs(m) - 1);
      // x carries the label, so it is in w's row iff it is in the segment
      int32_t lo = seg.x, len = seg.y - seg.x;
      while (len > 0) {
        const int32_t half = len >> 1;
        if (__ldg(g.lcol + lo + half) < x) {
          lo += half + 1;
          len -= half + 1;
        } else {
          len = half;
        }
      }
      if (lo < seg.y && __ldg(g.lcol + lo) == x) --avail;
    }
    if (avail < d.la_need[t]) return false;
    if (d.la >= 2) {
      const int32_t end = min(seg.y, seg.x + kLaScan);
      int32_t found = 0;
      for (int32_t e = seg.x; e < end && found < d.la_need[t]; ++e) {
        const int32_t x = __ldg(g.lcol + e);
        bool cand = false;
        for (uint32_t u = d.la_uq[t]; u && !cand; u &= u - 1)
          cand = bitmap_has(d.cand + (size_t)(__ffs(u) - 1) * d.n_words, x);
        if (!cand) continue;
        bool used = false;  // a row vertex (only same-label positions can be)
        for (int c = 0; c < d.i && !used; ++c) used = row(c) == x;
        if (!used) ++found;
      }
      if (found < d.la_need[t] && end == seg.y) return false;
    }
  }
  return true;
}

// The check of one row's candidates for 1 to 3 mapped neighbours, at most two
// injectivity tests and no look-ahead: what it needs of the row is loaded once
// per row and kept in registers, with where the other neighbours' adjacency is.  The last level of
// a 5-cycle listing on R-MAT 20 (67 M candidates, four a row) went from 2.00 to
// 1.67 ms with it, the distinct 4-cliques of R-MAT 16 from 11.3 to 9.8 ms.
template <int kNb>
struct RowCheck {
  static constexpr int kOthers = kNb > 1 ? kNb - 1 : 1;
  int32_t inj0 = -1, inj1 = -1;  // same-label images
  // the neighbours besides the pivot: row [b, e), or, of a hub, e = -1 and b =
  // its bitmap's index
  int32_t b[kOthers], e[kOthers];

  __device__ __forceinline__ void load(const GraphDev &g, const LevelDesc &d,
                                       const ColumnRow &row, int slot) {
    if (d.ninj > 0) inj0 = row(d.inj[0]);
    if (d.ninj > 1) inj1 = row(d.inj[1]);
    if constexpr (kNb > 1) {
#pragma unroll
      for (int o = 0; o < kOthers; ++o) {
        const int32_t x = row(d.bpos[o + (o >= slot)]);
        b[o] = e[o] = 0;
        if (!GSM_IN_BOUNDS(g.dbg, x >= 0 && x < g.n, kDbgNeighbour)) continue;
        const int32_t h = g.hub ? __ldg(g.hub + x) : -1;
        if (h >= 0) {
          b[o] = h;
          e[o] = -1;
        } else {
          b[o] = __ldg(g.rp + x);
          e[o] = __ldg(g.rp + x + 1);
        }
      }
    }
  }

  __device__ __forceinline__ bool ok(const GraphDev &g, const LevelDesc &d, int32_t w) const {
    if (w == inj0 || w == inj1) return false;
    if (d.bitmap && !bitmap_has(d.bitmap, w)) return false;
    if constexpr (kNb > 1) {
#pragma unroll
      for (int o = 0; o < kOthers; ++o)
        if (!(e[o] < 0 ? hub_bit(g, b[o], w) : row_search(g, b[o], e[o], d.lab, w))) return false;
    }
    return true;
  }
};

// How a level's launch checks its candidates.
//   kCheckAny      every shape: check_candidate and the look-ahead, one
//                  candidate after the other, the row read again for each;
//                  kCheckAnyFew: also from the candidate's side
//                  (row_contains_few), with the candidates loaded together
//   kCheckWide, kCheckWideFew: the same two in CTAs of more than 256 threads
//   kCheckRow + n  n = 1..3 mapped neighbours, at most two injectivity tests,
//                  no look-ahead: RowCheck
//   kCheckGroup+n  the same shapes, n = 2, 3: the loads of a thread's four
//                  candidates are issued together, stage by stage -- candidate
//                  bitmap, images of the row, hub indexes, adjacency words, and
//                  the steps of the binary searches
// A check is a chain of dependent loads.  With few candidates a row they miss
// L1 and the chains' latency bounds the level: grouped, the last level of a
// 5-cycle listing on R-MAT 20 (four candidates a row) took 1.46 instead of
// 1.67 ms; 1.17 with searches that compare ids alone and halve by length
// (the listing 1,981 -> 1,834 -> 1,721 us).  With many, the row's adjacency stays in L1 and the grouped form's
// registers cost more warps than it gains: ordered triangles of R-MAT 20 (146
// a row) 24.1 against 19.9 ms, 4-cliques of R-MAT 16 12.5 against 9.8 ms.
// Hence grouped up to kFewCandidates candidates a row on average.  The forms for
// every shape go by the same line: one candidate after the other with eight CTAs
// an SM counts the 6-cliques of R-MAT 15 with three labels in 44.3 ms, four
// loaded together and looked at from both sides, at four CTAs, in 57.4.
constexpr int kCheckWideFew = -3, kCheckWide = -2, kCheckAnyFew = -1, kCheckAny = 0, kCheckRow = 0,
              kCheckGroup = 3;
constexpr int kMaxRowCheck = 3;

// Which of the `alive` pairs are edges: w[j] (label lab_of(j)) in the row of
// x[j].  row_contains_l of four pairs, their loads issued together; few (bit
// j): see row_contains_few.
template <typename Lab>
__device__ __forceinline__ uint32_t group_contains(const GraphDev &g,
                                                   const int32_t (&x)[kItemsPerThread],
                                                   const int32_t (&w)[kItemsPerThread],
                                                   const Lab &lab_of, uint32_t alive,
                                                   uint32_t few) {
  constexpr int kN = kItemsPerThread;
  uint32_t open = alive;  // pairs no bitmap has decided
  if (g.hub) {
    int32_t h[kN];
    uint32_t word[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) h[j] = (alive >> j) & 1u ? __ldg(g.hub + x[j]) : -1;
    uint32_t rev = 0;  // taken from the candidate's bitmap
#pragma unroll
    for (int j = 0; j < kN; ++j)
      if (h[j] < 0 && (alive & few) >> j & 1u) {
        h[j] = __ldg(g.hub + w[j]);
        rev |= 1u << j;
      }
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const int32_t v = (rev >> j) & 1u ? x[j] : w[j];
      word[j] = h[j] >= 0 ? __ldg(g.hub_bits + (size_t)h[j] * g.hub_words + (v >> 5)) >> (v & 31)
                          : 0u;
    }
#pragma unroll
    for (int j = 0; j < kN; ++j)
      if (h[j] >= 0) {
        open &= ~(1u << j);
        if (!(word[j] & 1u)) alive &= ~(1u << j);
      }
  }
  if (!open) return alive;
  // binary searches, step by step together
  int32_t lo[kN], len[kN], end[kN], key[kN], lab[kN];
#pragma unroll
  for (int j = 0; j < kN; ++j) {
    const bool on = (open >> j) & 1u;
    lo[j] = on ? __ldg(g.rp + x[j]) : 0;
    end[j] = on ? __ldg(g.rp + x[j] + 1) : 0;
    key[j] = w[j];
    lab[j] = lab_of(j);
  }
#pragma unroll
  for (int j = 0; j < kN; ++j) {
    if ((few & open) >> j & 1u && end[j] - lo[j] > kLongRow) {
      const int32_t wb = __ldg(g.rp + w[j]), we = __ldg(g.rp + w[j] + 1);
      if (we - wb < end[j] - lo[j]) {  // the candidate's row is shorter: x in it
        lo[j] = wb;
        end[j] = we;
        key[j] = x[j];
        lab[j] = __ldg(g.lab + x[j]);
      }
    }
    len[j] = end[j] - lo[j];
    if (len[j] <= 0) {  // an empty row, or none to search
      if ((open >> j) & 1u) alive &= ~(1u << j);
      open &= ~(1u << j);
      len[j] = 0;
    }
  }
  // The part [lo, lo + len) that can hold the key is halved with its longer
  // side kept, so that its length does not depend on what was read: a step is a
  // load, a compare and an add, and the longest of the four rows counts the
  // steps for all.
  const bool one = g.num_labels == 1;
  int32_t longest = len[0];
#pragma unroll
  for (int j = 1; j < kN; ++j) longest = max(longest, len[j]);
  auto search = [&](auto plain) {  // plain: one label, ids alone order a row
    for (; longest > 1; longest -= longest >> 1) {
      int32_t v[kN], m[kN];
#pragma unroll
      for (int j = 0; j < kN; ++j) {
        const int32_t half = len[j] >> 1;
        v[j] = half > 0 ? __ldg(g.lcol + lo[j] + half - 1) : key[j];
        if constexpr (!decltype(plain)::value)
          m[j] = half > 0 ? __ldg(g.llab + lo[j] + half - 1) : lab[j];
      }
#pragma unroll
      for (int j = 0; j < kN; ++j) {
        const int32_t half = len[j] >> 1;
        bool below = v[j] < key[j];
        if constexpr (!decltype(plain)::value)
          below = m[j] < lab[j] || (m[j] == lab[j] && below);
        if (below) lo[j] += half;
        len[j] -= half;
      }
    }
    int32_t v[kN], m[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      v[j] = (open >> j) & 1u ? __ldg(g.lcol + lo[j]) : key[j];
      if constexpr (!decltype(plain)::value)
        m[j] = (open >> j) & 1u ? __ldg(g.llab + lo[j]) : lab[j];
    }
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      bool in = v[j] == key[j];
      if constexpr (!decltype(plain)::value) in = in && m[j] == lab[j];
      if (!in) alive &= ~(1u << j);
    }
  };
  if (one)
    search(std::true_type{});
  else
    search(std::false_type{});
  return alive;
}

// The candidates x = xb .. xb + 3 of one thread, below x1: returns a bit for
// each that passes the level's checks; rj, wj: their rows and vertices.
// kProbes (kCheckAny only): adds the checks' probe bytes to *probe_bytes.
// kSteps (kCheckAny, kCheckWide): next_row's.
template <int kCheck, bool kProbes = false, int kSteps = 4>
__device__ __forceinline__ uint32_t check_group(
    const GraphDev &g, const LevelDesc &d, const int32_t *__restrict__ F, int32_t ld,
    const TileRows &t, const int32_t *s_woff, const int64_t *__restrict__ woff, int64_t wa,
    const int32_t *__restrict__ pstart, const uint8_t *__restrict__ pslot, int32_t xb, int32_t x1,
    int32_t (&rj)[kItemsPerThread], int32_t (&wj)[kItemsPerThread],
    uint32_t *probe_bytes = nullptr) {
  constexpr int kN = kItemsPerThread;
  constexpr int kNb = kCheck > kCheckGroup ? kCheck - kCheckGroup : 0;
  int32_t rs;
  int32_t r = item_row(t, s_woff, woff, wa, xb, &rs);
  int32_t rr = r - t.r0;
  int32_t re = t.staged ? s_woff[rr + 1] : (int32_t)(woff[r + 1] - wa);
  int32_t pst = pstart[r], slot = pslot[r];
  if constexpr (kCheck > kCheckRow && kCheck <= kCheckRow + kMaxRowCheck) {
    RowCheck<kCheck - kCheckRow> check;
    check.load(g, d, ColumnRow{F, ld, r}, slot);
    uint32_t bits = 0;
#pragma unroll
    for (int j = 0; j < kN; ++j) {  // (rj, wj: only of candidates that pass)
      const int32_t x = xb + j;
      if (x >= x1) break;
      if (x >= re) {
        next_row(t, s_woff, woff, wa, x, &rr, &rs, &re);
        r = t.r0 + rr;
        pst = pstart[r];
        slot = pslot[r];
        check.load(g, d, ColumnRow{F, ld, r}, slot);
      }
      if (!GSM_IN_BOUNDS(g.dbg, pst + (x - rs) >= 0 && pst + (x - rs) < g.nnz, kDbgCandidate) ||
          !GSM_IN_BOUNDS(g.dbg, r >= 0 && r < ld, kDbgRow))
        continue;
      const int32_t w = __ldg(g.lcol + pst + (x - rs));
      rj[j] = r;
      wj[j] = w;
      if (check.ok(g, d, w)) bits |= 1u << j;
    }
    return bits;
  }
  if constexpr (kCheck == kCheckAny || kCheck == kCheckWide) {  // (rj, wj: as above)
    uint32_t bits = 0;
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const int32_t x = xb + j;
      if (x >= x1) break;
      if (x >= re) {
        next_row<kSteps>(t, s_woff, woff, wa, x, &rr, &rs, &re);
        r = t.r0 + rr;
        pst = pstart[r];
        slot = pslot[r];
      }
      if (!GSM_IN_BOUNDS(g.dbg, pst + (x - rs) >= 0 && pst + (x - rs) < g.nnz, kDbgCandidate) ||
          !GSM_IN_BOUNDS(g.dbg, r >= 0 && r < ld, kDbgRow))
        continue;
      const int32_t w = __ldg(g.lcol + pst + (x - rs));
      rj[j] = r;
      wj[j] = w;
      const ColumnRow row{F, ld, r};
      bool ok;
      if constexpr (kProbes)
        ok = check_candidate_probes(g, d, row, w, slot, false, probe_bytes);
      else
        ok = check_candidate(g, d, row, w, slot, false);
      if (ok && (!d.la || lookahead_ok(g, d, row, w))) bits |= 1u << j;
    }
    return bits;
  }
  int32_t at[kN], sj[kN];
  uint32_t alive = 0, few = 0;
#pragma unroll
  for (int j = 0; j < kN; ++j) {
    const int32_t x = xb + j;
    if (x < x1) {
      if (x >= re) {
        next_row(t, s_woff, woff, wa, x, &rr, &rs, &re);
        r = t.r0 + rr;
        pst = pstart[r];
        slot = pslot[r];
      }
      if (GSM_IN_BOUNDS(g.dbg, pst + (x - rs) >= 0 && pst + (x - rs) < g.nnz, kDbgCandidate) &&
          GSM_IN_BOUNDS(g.dbg, r >= 0 && r < ld, kDbgRow))
        alive |= 1u << j;
      if (re - rs <= kFewCandidates) few |= 1u << j;
    }
    rj[j] = r;
    sj[j] = slot;
    at[j] = pst + (x - rs);
  }
  if (g.hub_lo) few = 0;  // bitmaps that do not cover the mapped neighbours
  if constexpr (kCheck < kCheckAny) {
#pragma unroll
    for (int j = 0; j < kN; ++j) wj[j] = (alive >> j) & 1u ? __ldg(g.lcol + at[j]) : 0;
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      if (!((alive >> j) & 1u)) continue;
      const ColumnRow row{F, ld, rj[j]};
      bool ok;
      if constexpr (kProbes)
        ok = check_candidate_probes(g, d, row, wj[j], sj[j], (few >> j) & 1u, probe_bytes);
      else
        ok = check_candidate(g, d, row, wj[j], sj[j], (few >> j) & 1u);
      if (!ok || (d.la && !lookahead_ok(g, d, row, wj[j]))) alive &= ~(1u << j);
    }
    return alive;
  }
  // what depends on the row alone is loaded beside the candidates
  int32_t x[kNb > 1 ? kNb - 1 : 1][kN], y[2][kN];
#pragma unroll
  for (int j = 0; j < kN; ++j) wj[j] = (alive >> j) & 1u ? __ldg(g.lcol + at[j]) : 0;
#pragma unroll
  for (int o = 0; o + 1 < kNb; ++o)
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      x[o][j] = (alive >> j) & 1u ? F[d.bpos[o + (o >= sj[j])] * ld + rj[j]] : 0;
      if (!GSM_IN_BOUNDS(g.dbg, x[o][j] >= 0 && x[o][j] < g.n, kDbgNeighbour)) {
        alive &= ~(1u << j);
        x[o][j] = 0;
      }
    }
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int j = 0; j < kN; ++j)
      y[t][j] = t < d.ninj && (alive >> j) & 1u ? F[d.inj[t] * ld + rj[j]] : -1;
  if (d.bitmap) {
    uint32_t word[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j)
      word[j] = (alive >> j) & 1u ? __ldg(d.bitmap + (wj[j] >> 5)) : 0u;
#pragma unroll
    for (int j = 0; j < kN; ++j)
      if (!((word[j] >> (wj[j] & 31)) & 1u)) alive &= ~(1u << j);
  }
#pragma unroll
  for (int j = 0; j < kN; ++j)
    if (y[0][j] == wj[j] || y[1][j] == wj[j]) alive &= ~(1u << j);
#pragma unroll
  for (int o = 0; o + 1 < kNb; ++o)  // neighbours besides the pivot
    alive = group_contains(g, x[o], wj, [&](int) { return d.lab; }, alive, few);
  return alive;
}

// Writes the partial embedding `src` (src(c) = image of pi_c, c < d.i)
// extended by w as output row `row` of the sink (see RowSink): position c goes
// to column d.out_col[c], w to d.out_col[d.i].
template <int kMode, typename Row>
__device__ __forceinline__ void put_row(const RowSink &sink, const LevelDesc &d, const Row &src,
                                        int32_t w, int64_t row) {
  const int32_t i = d.i;
  if (kMode == kSinkColumns) {
    int32_t *o = (int32_t *)sink.out + row;
    for (int c = 0; c < i; ++c) o[d.out_col[c] * sink.ld] = src(c);
    o[d.out_col[i] * sink.ld] = w;
  } else if (kMode == kSinkRows) {
    int32_t *o = (int32_t *)sink.out + row * sink.k;
    for (int c = 0; c < i; ++c) o[d.out_col[c]] = src(c);
    o[d.out_col[i]] = w;
  } else if (sink.nw <= 2) {
    // packed key of one or two words: column j occupies bits
    // [(k-1-j)*b, (k-j)*b); each column is read once and or-ed into the
    // word(s) it overlaps
    uint64_t *o = (uint64_t *)sink.out + row;
    uint64_t w0 = 0, w1 = 0;
    for (int c = 0; c <= i; ++c) {
      const uint64_t v = (uint32_t)(c < i ? src(c) : w);
      const int32_t p = (sink.k - 1 - d.out_col[c]) * sink.bits;
      if (p >= 64) {
        w1 |= v << (p - 64);
      } else {
        w0 |= v << p;
        if (p + sink.bits > 64) w1 |= v >> (64 - p);
      }
    }
    if (sink.rank) {
      const int32_t pr = parent_index(src);
      if (pr >= 0) {
        const uint64_t v = (uint32_t)__ldg(sink.rank + pr);
        const int32_t p = sink.rank_pos;
        if (p >= 64) {
          w1 |= v << (p - 64);
        } else {
          w0 |= v << p;
          if (p > 32) w1 |= v >> (64 - p);
        }
      }
    }
    o[0] = w0;
    if (sink.nw == 2) o[sink.ld] = w1;
  } else {
    // packed key: column j occupies bits [(k-1-j)*b, (k-j)*b); word t
    // collects the columns that overlap bits [64t, 64t+64)
    uint64_t *o = (uint64_t *)sink.out + row;
    for (int t = 0; t < sink.nw; ++t) {
      uint64_t kw = 0;
      for (int c = 0; c <= i; ++c) {
        const uint64_t v = (uint32_t)(c < i ? src(c) : w);
        const int32_t lo = (sink.k - 1 - d.out_col[c]) * sink.bits - 64 * t;
        if (lo >= 0 && lo < 64)
          kw |= v << lo;
        else if (lo < 0 && lo + sink.bits > 0)
          kw |= v >> (-lo);
      }
      o[t * sink.ld] = kw;
    }
  }
}

__device__ __forceinline__ unsigned long long load_relaxed(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}


// Exclusive rank of this thread's c items among the block's (threads in
// order) and the block total; s_warp holds 33 ints; contains two barriers.
__device__ __forceinline__ int32_t block_rank(int32_t c, int32_t *s_warp, int32_t *total) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(kAll, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int nwarps = blockDim.x >> 5;
    const int32_t v = lane < nwarps ? s_warp[lane] : 0;
    int32_t wi = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(kAll, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < nwarps) s_warp[lane] = wi - v;
    if (lane == 31) s_warp[32] = wi;
  }
  __syncthreads();
  *total = s_warp[32];
  return incl - c + s_warp[warp];
}

// Decoupled look-back, in two halves so that a CTA can verify its next tile
// between them.  lookback_publish: tile `tile` has T survivors; tile 0
// publishes its inclusive prefix, every other tile its own count, and the
// level total (word tiles + 1) gains T.  Any thread may call it.
__device__ __forceinline__ void lookback_publish(unsigned long long *lookback, int32_t tile,
                                                 int32_t tiles, unsigned long long T) {
  atomicExch(lookback + tile, (tile == 0 ? kLbInclusive : kLbAggregate) | T);
  if (T) atomicAdd(lookback + tiles + 1, T);
}

// lookback_resolve, run by one whole warp after lookback_publish: reads the
// published words of the 32 preceding tiles at a time (lane l: tile
// window_end - l) until one holds an inclusive prefix, publishes the tile's
// own inclusive prefix, and returns the number of survivors of all earlier
// tiles in every lane.  A wait longer than spin_limit polls sets word
// tiles + 2 and returns the (smaller) sum found so far, so every row the
// caller writes stays inside the level's reserved output.  publish = false
// keeps the tile's word unwritten (fault injection: later tiles wait on it).
__device__ __forceinline__ unsigned long long lookback_resolve(unsigned long long *lookback,
                                                               int32_t tile, int32_t tiles,
                                                               unsigned long long T, int lane,
                                                               int32_t spin_limit,
                                                               bool publish = true) {
  constexpr unsigned kAll = 0xffffffffu;
  if (tile == 0) return 0;
  unsigned long long prefix = 0;
  int32_t window_end = tile - 1;
  int32_t polls = 0;
  bool gave_up = false;
  while (true) {
    const int32_t j = window_end - lane;
    unsigned long long st = j >= 0 ? load_relaxed(lookback + j) : kLbInclusive;
    unsigned long long flag = st & ~kLbValue;
    // wait until every tile of the window has published
    while (__any_sync(kAll, flag == 0)) {
      if (++polls > spin_limit) {
        gave_up = true;
        break;
      }
      __nanosleep(32);
      if (flag == 0) {
        st = load_relaxed(lookback + j);
        flag = st & ~kLbValue;
      }
    }
    if (gave_up) break;
    const uint32_t has_prefix = __ballot_sync(kAll, flag == kLbInclusive);
    // tiles up to the nearest inclusive prefix (the lowest such lane)
    const int32_t stop = has_prefix ? __ffs(has_prefix) - 1 : 31;
    unsigned long long v = lane <= stop ? (st & kLbValue) : 0;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
    prefix += v;
    if (has_prefix) break;
    window_end -= 32;
  }
  if (lane == 0) {
    if (gave_up) atomicExch(lookback + tiles + 2, 1ull);
    if (publish) atomicExch(lookback + tile, kLbInclusive | (prefix + T));
  }
  return prefix;
}

// Both halves at once (the tile waits for its prefix right after counting);
// publish = false: as above, and the total gains T all the same.
__device__ __forceinline__ unsigned long long lookback_prefix(unsigned long long *lookback,
                                                              int32_t tile, int32_t tiles,
                                                              unsigned long long T, int lane,
                                                              int32_t spin_limit,
                                                              bool publish = true) {
  if (lane == 0) {
    if (publish)
      lookback_publish(lookback, tile, tiles, T);
    else if (T)
      atomicAdd(lookback + tiles + 1, T);
  }
  __syncwarp();
  return lookback_resolve(lookback, tile, tiles, T, lane, spin_limit, publish);
}

}  // namespace gsm
