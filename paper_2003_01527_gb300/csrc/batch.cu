// Batched form: many query graphs against one resident data graph, all
// levels of all queries issued as one fixed sequence of persistent kernels
// (captured once as a CUDA graph by the host driver).
//
// The queries advance together, one verification level per step (Sec. 3.2,
// Algorithm 1), over one concatenated frontier whose rows carry the index of
// their query ("segment").  No kernel needs a size from the host: every
// launch has a fixed grid and reads the sizes of its step (rows, candidates,
// tiles, survivors) from device memory, so the whole sequence runs without a
// host synchronisation.  Buffers have fixed capacities; a step that would
// exceed them sets an overflow flag, produces nothing further, and the host
// reruns the batch on the single-query path.
#include <algorithm>
#include <cstddef>

#include "batch.h"
#include "filter_body.cuh"
#include "segments.cuh"
#include "verify.cuh"

namespace gsm {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---- set-up, filter and level 1

// Zeroes what the batch adds up in: the step sizes, the overflow flag, the
// counts and the list's look-back words.
__global__ void __launch_bounds__(256) k_b_init(BatchStep *state, int32_t *overflow,
                                                unsigned long long *counts, int64_t ncounts,
                                                unsigned long long *lb_list, int64_t lb_words) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t j = t; j <= kMaxK; j += stride) state[j] = BatchStep{0, 0, 0, 0, 0, 0, 0};
  for (int64_t j = t; j < ncounts; j += stride) counts[j] = 0;
  for (int64_t j = t; j < lb_words; j += stride) lb_list[j] = 0;
  if (t == 0) *overflow = 0;
}

__global__ void __launch_bounds__(256) k_b_filter(GraphDev g, const FilterDesc *__restrict__ fds,
                                                  uint32_t *const *__restrict__ bm_out,
                                                  unsigned long long *__restrict__ sizes) {
  __shared__ FilterDesc s_d;
  const int32_t q = blockIdx.y;
  for (int j = threadIdx.x; j < (int)(sizeof(FilterDesc) / 4); j += blockDim.x)
    reinterpret_cast<int32_t *>(&s_d)[j] = reinterpret_cast<const int32_t *>(fds + q)[j];
  __syncthreads();
  if (s_d.k == 0) return;  // padding slot of a bucketed batch
  filter_warps(g, s_d, bm_out[q], sizes + (int64_t)q * kMaxK,
               ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
               ((int64_t)gridDim.x * blockDim.x) >> 5);
}

// The same from the graph's bitmaps (a thread per word, a CTA row per query).
template <int kV>
__global__ void __launch_bounds__(256) k_b_filter_bits(GraphDev g,
                                                       const FilterDesc *__restrict__ fds,
                                                       uint32_t *const *__restrict__ bm_out,
                                                       unsigned long long *__restrict__ sizes) {
  __shared__ FilterDesc s_d;
  const int32_t q = blockIdx.y;
  for (int j = threadIdx.x; j < (int)(sizeof(FilterDesc) / 4); j += blockDim.x)
    reinterpret_cast<int32_t *>(&s_d)[j] = reinterpret_cast<const int32_t *>(fds + q)[j];
  __syncthreads();
  filter_words<kV>(g, s_d, bm_out[q], sizes ? sizes + (int64_t)q * kMaxK : nullptr, 0, 1);
}

// ---- counts, and what the last CTA of a kernel does

// One thread's sum of the numbers of one query's whole embeddings (halves of
// 32 bits), added to the query's two count words when the query changes.
struct BatchSum {
  int32_t q = -1;
  unsigned long long lo = 0, hi = 0;
  __device__ __forceinline__ void add(int32_t query, unsigned long long v,
                                      unsigned long long *counts) {
    if (query != q) {
      put(counts);
      q = query;
    }
    lo += (uint32_t)v;
    hi += v >> 32;
  }
  __device__ __forceinline__ void put(unsigned long long *counts) {
    if (lo) atomicAdd(counts + 2 * (int64_t)q, lo);
    if (hi) atomicAdd(counts + 2 * (int64_t)q + 1, hi);
    lo = hi = 0;
  }
  // All lanes of the warp: one atomic for the warp when its lanes sum one
  // query (most tiles hold rows of one query), else one per lane.
  __device__ __forceinline__ void flush(unsigned long long *counts) {
    const bool has = lo || hi;
    const uint32_t m = __ballot_sync(kFull, has);
    if (!m) return;
    const int32_t q0 = __shfl_sync(kFull, q, __ffs(m) - 1);
    if (__all_sync(kFull, !has || q == q0)) {
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        lo += __shfl_xor_sync(kFull, lo, o);
        hi += __shfl_xor_sync(kFull, hi, o);
      }
      q = q0;
      if ((threadIdx.x & 31) == 0) put(counts);
      lo = hi = 0;
    } else {
      put(counts);
    }
  }
};

// The number of query `bq`'s embeddings with this core row.
template <typename Row>
__device__ __forceinline__ unsigned long long core_number(const GraphDev &g, const BatchQuery &bq,
                                                          const Row &row, bool *over) {
  if (bq.leaf.nleaves == 0) return 1;
  return leaf_number<kMaxK>(g, bq.leaf, row, over, [](int, unsigned long long) {});
}

// True in every thread of the CTA that finishes last (lb: the kernel's
// look-back words; the counter of finished CTAs is word tiles + 3).  One
// barrier; the CTA's earlier atomics are ordered before its count.
__device__ __forceinline__ bool last_cta(unsigned long long *lb, int64_t tiles) {
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(lb + tiles + 3, 1ull) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  return s_last;
}

__device__ __forceinline__ void zero_words(unsigned long long *p, int64_t n) {
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) p[j] = 0;
}

// Rows of a level go into arrays of this leading dimension: as many as there
// are candidates, at most what the frontier holds (more survivors are an
// overflow).
__device__ __forceinline__ int64_t level_ld(int64_t most, int32_t width, int64_t cap_rows,
                                            int64_t cap_elems) {
  return min(most, min(cap_rows, cap_elems / width));
}

// Level 1 of every query: its candidate list for pi_0, queries in batch order.
// Tiles of kBatchListTile root-bitmap words (only words inside the root's
// restriction are numbered: list_off); a tile's rows start where the
// look-back says.  Queries whose core is one vertex are counted here.  The
// last CTA sets the level's size and zeroes the next kernel's look-back words.
__global__ void __launch_bounds__(256) k_b_list(GraphDev g, const BatchQuery *__restrict__ qs,
                                                int32_t nq, const int64_t *__restrict__ list_off,
                                                BatchStep *state, int64_t cap,
                                                int32_t *__restrict__ F,
                                                int32_t *__restrict__ rseg,
                                                unsigned long long *counts,
                                                unsigned long long *lb,
                                                unsigned long long *lb_pivot, int32_t spin_limit,
                                                int32_t stall_tile, int32_t *overflow) {
  constexpr int kWords = kBatchListTile / 256;  // of a thread, consecutive
  __shared__ int32_t s_warp[33];
  __shared__ int32_t s_tile, s_q;
  __shared__ unsigned long long s_prefix;
  const int64_t words = list_off[nq];
  const int32_t tiles = (int32_t)((words + kBatchListTile - 1) / kBatchListTile);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool over = false;
  for (;;) {
    if (threadIdx.x == 0) {
      const int32_t tile = (int32_t)atomicAdd(lb + tiles, 1ull);
      int32_t lo = 0, len = nq;  // last query whose words start at or before the tile
      while (len > 1) {
        const int32_t half = len >> 1;
        if (list_off[lo + half] <= (int64_t)tile * kBatchListTile) lo += half;
        len -= half;
      }
      s_tile = tile;
      s_q = lo;
    }
    __syncthreads();
    const int32_t tile = s_tile;
    if (tile >= tiles) break;  // uniform across the block
    int32_t q = s_q;
    uint32_t word[kWords];
    int32_t qw[kWords], vw[kWords];
    int32_t c = 0;
    BatchSum sum;
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      const int64_t i = (int64_t)tile * kBatchListTile + threadIdx.x * kWords + j;
      word[j] = 0;
      if (i >= words) continue;
      while (list_off[q + 1] <= i) ++q;
      const BatchQuery &bq = qs[q];
      const int32_t w = bq.word0 + (int32_t)(i - list_off[q]);
      uint32_t x = __ldg(bq.root_bitmap + w);
      if (bq.kc == 1) {
        for (; x; x &= x - 1) {
          const int32_t v = w * 32 + __ffs(x) - 1;
          sum.add(q, core_number(g, bq, [&](int) { return v; }, &over), counts);
        }
      }
      word[j] = x;
      qw[j] = q;
      vw[j] = w * 32;
      c += __popc(x);
    }
    sum.flush(counts);
    int32_t T;
    const int32_t rank = block_rank(c, s_warp, &T);
    if (warp == 0) {
      const unsigned long long p = lookback_prefix(lb, tile, tiles, (unsigned long long)T, lane,
                                                   spin_limit, tile != stall_tile);
      if (lane == 0) s_prefix = p;
    }
    __syncthreads();
    int64_t pos = (int64_t)s_prefix + rank;
#pragma unroll
    for (int j = 0; j < kWords; ++j)
      for (uint32_t x = word[j]; x; x &= x - 1, ++pos)
        if (pos < cap) {
          F[pos] = vw[j] + __ffs(x) - 1;
          rseg[pos] = qw[j];
        }
    __syncthreads();  // the shared words are reused by the next tile
  }
  if (over) *overflow = kBatchOverflow;  // past 64 bits: the single-query path reports it
  if (!last_cta(lb, tiles)) return;
  const int64_t R = (int64_t)atomicAdd(lb + tiles + 1, 0ull);
  const bool late = atomicAdd(lb + tiles + 2, 0ull) != 0;
  const bool ok = !late && R <= cap;
  if (threadIdx.x == 0) {
    if (late) *overflow = kBatchTimeout;
    else if (!ok) *overflow = kBatchOverflow;
    state[1].R = ok ? R : 0;
    state[1].ld = R;
  }
  zero_words(lb_pivot, (ok ? (R + kBatchPivotTile - 1) / kBatchPivotTile : 0) + kLbExtra);
}

// ---- one step: level i -> i+1 (frontier rows of width i, column-major,
// leading dimension state[i].ld)

// Pivot choice of every row and scan of the rows' candidate counts: tiles of
// kBatchPivotTile rows, a row per thread.  A row also writes itself into
// tile_row for every level tile that starts among its candidates.  The last
// CTA sets the step's candidates, tiles and next leading dimension, and
// zeroes the level's look-back words.
__global__ void __launch_bounds__(256) k_b_pivot_scan(
    GraphDev g, const BatchQuery *__restrict__ qs, int32_t i, BatchStep *state,
    const int32_t *__restrict__ F, const int32_t *__restrict__ rseg,
    int32_t *__restrict__ pstart, uint8_t *__restrict__ pslot, int64_t *__restrict__ woff,
    int32_t *__restrict__ tile_row, int32_t tile_items, int64_t cap_rows, int64_t cap_elems,
    int64_t cap_items, unsigned long long *lb, unsigned long long *lb_level, int32_t spin_limit,
    int32_t stall_tile, int32_t *overflow) {
  __shared__ int64_t s_warp[33];
  __shared__ int32_t s_tile;
  __shared__ unsigned long long s_prefix;
  const int64_t R = state[i].R, ld = state[i].ld;
  const int32_t tiles = (int32_t)((R + kBatchPivotTile - 1) / kBatchPivotTile);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t max_tiles = (cap_items + tile_items - 1) / tile_items;  // entries of tile_row
  for (;;) {
    if (threadIdx.x == 0) s_tile = (int32_t)atomicAdd(lb + tiles, 1ull);
    __syncthreads();
    const int32_t tile = s_tile;
    if (tile >= tiles) break;  // uniform across the block
    const int64_t r = tile * kBatchPivotTile + threadIdx.x;
    int32_t best = 0;
    if (r < R) {
      const BatchLevel &L = qs[rseg[r]].lv[i];
      int32_t best_start = 0, best_slot = 0, lo = L.rlo;
      best = 0x7fffffff;
      for (int t = 0; t < L.ngt; ++t) lo = max(lo, F[L.gt[t] * ld + r] + 1);
      for (int b = 0; b < L.nb; ++b) {
        const int32_t x = F[L.bpos[b] * ld + r];
        int2 seg = label_segment(g, x, L.lab);  // only pi_i's label can match
        if (L.cut) seg = cut_segment(g, seg, lo, L.rhi);
        if (seg.y - seg.x < best) {
          best = seg.y - seg.x;
          best_start = seg.x;
          best_slot = b;
        }
      }
      pstart[r] = best_start;
      pslot[r] = (uint8_t)best_slot;
    }
    // exclusive scan over the tile
    int64_t incl = best;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const int64_t v = lane < 8 ? s_warp[lane] : 0;
      int64_t vi = v;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, vi, o);
        if (lane >= o) vi += y;
      }
      if (lane < 8) s_warp[lane] = vi - v;
      const unsigned long long T = (unsigned long long)__shfl_sync(kFull, vi, 7);
      const unsigned long long p =
          lookback_prefix(lb, tile, tiles, T, lane, spin_limit, tile != stall_tile);
      if (lane == 0) s_prefix = p;
    }
    __syncthreads();
    if (r < R) {
      const int64_t s = (int64_t)s_prefix + s_warp[warp] + incl - best, e = s + best;
      woff[r] = s;
      if (best > 0)
        for (int64_t t = (s + tile_items - 1) / tile_items; t * tile_items < e && t < max_tiles;
             ++t)
          tile_row[t] = (int32_t)r;
    }
    __syncthreads();  // the shared words are reused by the next tile
  }
  if (!last_cta(lb, tiles)) return;
  const int64_t W = (int64_t)atomicAdd(lb + tiles + 1, 0ull);
  const bool late = atomicAdd(lb + tiles + 2, 0ull) != 0;
  const bool ok = !late && W <= cap_items;
  const int64_t level_tiles = ok ? (W + tile_items - 1) / tile_items : 0;
  if (threadIdx.x == 0) {
    if (late) *overflow = kBatchTimeout;
    else if (!ok) *overflow = kBatchOverflow;
    woff[R] = W;
    state[i].W = ok ? W : 0;
    state[i].tiles = level_tiles;
    if (level_tiles > 0) tile_row[level_tiles] = (int32_t)(R - 1);
    state[i + 1].ld = level_ld(W, i + 1, cap_rows, cap_elems);
  }
  zero_words(lb_level, level_tiles + kLbExtra);
}

// check_candidate of a thread's four candidates (w[j] of row r[j], a row of
// query q[j], pivot slot s[j]; `alive`: which of them there are), their loads
// issued together, stage by stage, as in the single-query path's grouped form:
// a batch's levels are short, and a check is a chain of dependent loads.
__device__ __forceinline__ uint32_t b_check_group(
    const GraphDev &g, const BatchQuery *__restrict__ qs, int32_t i,
    const int32_t *__restrict__ F, int32_t ld, const int32_t (&r)[kItemsPerThread],
    const int32_t (&q)[kItemsPerThread], const int32_t (&s)[kItemsPerThread],
    const int32_t (&w)[kItemsPerThread], uint32_t alive, uint32_t few) {
  constexpr int kN = kItemsPerThread;
  int32_t lab[kN];
  int nb = 0, ninj = 0;
  {
    const uint32_t *bm[kN];
    uint32_t word[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const BatchLevel &L = qs[q[j]].lv[i];
      const bool on = (alive >> j) & 1u;
      bm[j] = on ? L.bitmap : nullptr;
      lab[j] = L.lab;
      nb = max(nb, on ? (int)L.nb : 0);
      ninj = max(ninj, on ? (int)L.ninj : 0);
    }
#pragma unroll
    for (int j = 0; j < kN; ++j) word[j] = bm[j] ? __ldg(bm[j] + (w[j] >> 5)) : ~0u;
#pragma unroll
    for (int j = 0; j < kN; ++j)
      if (!((word[j] >> (w[j] & 31)) & 1u)) alive &= ~(1u << j);
  }
  for (int t = 0; t < ninj; ++t) {
    int32_t y[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const BatchLevel &L = qs[q[j]].lv[i];
      y[j] = (alive >> j) & 1u && t < L.ninj ? F[L.inj[t] * ld + r[j]] : -1;
    }
#pragma unroll
    for (int j = 0; j < kN; ++j)
      if (y[j] == w[j]) alive &= ~(1u << j);
  }
  for (int o = 0; o + 1 < nb && alive; ++o) {  // neighbours besides the pivot
    int32_t x[kN];
    uint32_t now = 0;  // candidates with this many neighbours
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const BatchLevel &L = qs[q[j]].lv[i];
      x[j] = 0;
      if ((alive >> j) & 1u && o + 1 < L.nb) {
        x[j] = F[L.bpos[o + (o >= s[j])] * ld + r[j]];
        now |= 1u << j;
      }
    }
    alive &= ~now | group_contains(g, x, w, [&](int j) { return lab[j]; }, now, few);
  }
  return alive;
}

// Verification and write pass of one step, in one launch: tiles by ticket; a
// tile's survivors are ranked, kept in one of two shared buffers and written
// after the CTA has verified its next tile, when the look-back has its prefix
// (the single-query path's k_extend_fused).
// Survivors of a query at its last level are counted (times their leaf
// numbers), and for a query that lists its rows written to the result arena;
// the others become rows of the next level.  Both ranks travel in one
// look-back word (30 bits each: a level has fewer than 2^30 candidates).
// Thread t of a tile takes the 4 consecutive candidates 4t .. 4t+3.
//
// Bound by latency at these sizes (thousands of candidates a level): one
// launch and a look-back replace the count pass, two three-kernel scans, two
// one-thread kernels and two write passes of the step.  256 counted queries on
// R-MAT 18 take 21 launches instead of 116 and 1,000 us instead of 1,250; 48
// listed ones 21 instead of 160, and 1,820 us instead of 2,160.
constexpr int kPackBits = 30;
constexpr unsigned long long kPackMask = (1ull << kPackBits) - 1;

template <int kMaxThreads>
__global__ void __launch_bounds__(kMaxThreads, kMaxThreads == 256 ? 4 : 1) k_b_level(
    GraphDev g, const BatchQuery *__restrict__ qs, int32_t i, BatchStep *state,
    const int32_t *__restrict__ F, const int32_t *__restrict__ rseg,
    const int32_t *__restrict__ pstart, const uint8_t *__restrict__ pslot,
    const int64_t *__restrict__ woff, const int32_t *__restrict__ tile_row, int64_t cap_rows,
    int64_t cap_elems, int64_t cap_final, unsigned long long *counts, int32_t *__restrict__ Fn,
    int32_t *__restrict__ rseg_n, int32_t *__restrict__ final_rows, unsigned long long *lb,
    unsigned long long *lb_pivot, int32_t spin_limit, int32_t stall_tile, int32_t *overflow) {
  static_assert(kItemsPerThread == 4, "four candidates per thread");
  extern __shared__ int32_t smem[];
  __shared__ int32_t s_tile;
  __shared__ int32_t s_warp[33];
  __shared__ unsigned long long s_prefix;
  const int32_t ld = (int32_t)state[i].ld, W = (int32_t)state[i].W;
  const int32_t tiles = (int32_t)state[i].tiles;
  const int64_t ldn = state[i + 1].ld, FB = state[i].FB;
  const int32_t B = blockDim.x;
  const int32_t tile_items = B * kItemsPerThread;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t *s_woff = smem;
  int32_t *s_pairs = s_woff + tile_items + 4;  // 2 buffers of tile_items (row, vertex) pairs
  int32_t pend = -1, pend_T = 0, buf = 0;
  const int32_t width = i + 1;
  bool over = false;

  // T packs the tile's survivors: next rows in the low half (pairs from the
  // front of the buffer), result rows in the high half (pairs from its end)
  auto finish = [&](int32_t tile, int32_t T, int32_t pb) {
    const int32_t tn = T & 0xffff, tf = (int32_t)((uint32_t)T >> 16);
    if (warp == 0) {
      const unsigned long long p = lookback_resolve(
          lb, tile, tiles, ((unsigned long long)tf << kPackBits) | (unsigned long long)tn, lane,
          spin_limit, tile != stall_tile);
      if (lane == 0) s_prefix = p;
    }
    __syncthreads();
    const int32_t *pairs = s_pairs + pb * 2 * tile_items;
    const int64_t pn = (int64_t)(s_prefix & kPackMask), pf = (int64_t)(s_prefix >> kPackBits);
    for (int32_t x = threadIdx.x; x < tn; x += B) {
      const int32_t r = pairs[2 * x];
      const int64_t pos = pn + x;
      if (pos >= ldn) continue;  // over capacity: reported below
      for (int c = 0; c < i; ++c) Fn[c * ldn + pos] = F[c * ld + r];
      Fn[i * ldn + pos] = pairs[2 * x + 1];
      rseg_n[pos] = rseg[r];
    }
    for (int32_t x = threadIdx.x; x < tf; x += B) {
      const int32_t *pr = pairs + 2 * (tile_items - 1 - x);
      const int32_t r = pr[0];
      const int64_t at = FB + (pf + x) * width;
      if (at + width > cap_final) continue;  // over capacity: reported below
      const int8_t *oc = qs[rseg[r]].out_col;
      int32_t *dst = final_rows + at;
      for (int c = 0; c < i; ++c) dst[oc[c]] = F[c * ld + r];
      dst[oc[i]] = pr[1];
    }
  };

  for (;;) {
    if (threadIdx.x == 0) s_tile = (int32_t)atomicAdd(lb + tiles, 1ull);
    __syncthreads();
    const int32_t tile = s_tile;
    if (tile >= tiles) break;  // uniform across the block
    const int32_t x0 = tile * tile_items, x1 = min(x0 + tile_items, W);
    const TileRows t = stage_rows(woff, tile_row, 0, tile_items, s_woff, tile);
    const int32_t xb = x0 + warp * 128 + lane * kItemsPerThread;
    constexpr int kN = kItemsPerThread;
    uint32_t bits = 0, fbits = 0;
    int32_t rj[kN], wj[kN];
    BatchSum sum;
    if (xb < x1) {
      int32_t rs;
      int32_t r = item_row(t, s_woff, woff, 0, xb, &rs);
      int32_t rr = r - t.r0;
      int32_t re = t.staged ? s_woff[rr + 1] : (int32_t)woff[r + 1];
      int32_t q = rseg[r], pst = pstart[r], slot = pslot[r];
      int32_t qj[kN], sj[kN], at[kN];
      uint32_t alive = 0, few = 0;
#pragma unroll
      for (int j = 0; j < kN; ++j) {
        const int32_t x = xb + j;
        if (x < x1) {
          if (x >= re) {
            next_row(t, s_woff, woff, 0, x, &rr, &rs, &re);
            r = t.r0 + rr;
            q = rseg[r];
            pst = pstart[r];
            slot = pslot[r];
          }
          alive |= 1u << j;
          if (re - rs <= kFewCandidates) few |= 1u << j;
        }
        rj[j] = r;
        qj[j] = q;
        sj[j] = slot;
        at[j] = pst + (x - rs);
      }
#pragma unroll
      for (int j = 0; j < kN; ++j) wj[j] = (alive >> j) & 1u ? __ldg(g.lcol + at[j]) : 0;
      alive = b_check_group(g, qs, i, F, ld, rj, qj, sj, wj, alive, few);
#pragma unroll
      for (int j = 0; j < kN; ++j) {
        if (!((alive >> j) & 1u)) continue;
        const BatchQuery &bq = qs[qj[j]];
        if (i != bq.kc - 1) {
          bits |= 1u << j;
        } else {
          const ColumnRow row{F, ld, rj[j]};
          sum.add(qj[j], core_number(g, bq, ExtendedRow<ColumnRow>{row, i, wj[j]}, &over), counts);
          if (bq.enumerate) fbits |= 1u << j;
        }
      }
    }
    sum.flush(counts);
    int32_t T;
    const int32_t rank = block_rank(__popc(bits) | (__popc(fbits) << 16), s_warp, &T);
    {
      int32_t *s_pair = s_pairs + buf * 2 * tile_items;
      int32_t qn = rank & 0xffff, qf = (int32_t)((uint32_t)rank >> 16);
#pragma unroll
      for (int j = 0; j < kItemsPerThread; ++j) {
        if (!(((bits | fbits) >> j) & 1u)) continue;
        const int32_t at = (bits >> j) & 1u ? qn++ : tile_items - 1 - qf++;
        s_pair[2 * at] = rj[j];
        s_pair[2 * at + 1] = wj[j];
      }
    }
    if (threadIdx.x == 0 && tile != stall_tile)
      lookback_publish(lb, tile, tiles,
                       ((unsigned long long)((uint32_t)T >> 16) << kPackBits) |
                           (unsigned long long)(T & 0xffff));
    __syncthreads();
    if (pend >= 0) finish(pend, pend_T, buf ^ 1);
    pend = tile;
    pend_T = T;
    buf ^= 1;
  }
  if (pend >= 0) finish(pend, pend_T, buf ^ 1);
  if (over) *overflow = kBatchOverflow;  // past 64 bits: the single-query path reports it
  if (!last_cta(lb, tiles)) return;
  const unsigned long long total = atomicAdd(lb + tiles + 1, 0ull);
  const bool late = atomicAdd(lb + tiles + 2, 0ull) != 0;
  const int64_t S = (int64_t)(total & kPackMask), FS = (int64_t)(total >> kPackBits);
  const bool rows_ok = !late && S <= cap_rows && S * width <= cap_elems;
  const bool final_ok = !late && FB + FS * width <= cap_final;
  const int64_t Rn = rows_ok ? S : 0;
  if (threadIdx.x == 0) {
    if (late) *overflow = kBatchTimeout;
    else if (!rows_ok || !final_ok) *overflow = kBatchOverflow;
    state[i].S = S;
    state[i].FS = final_ok ? FS : 0;
    state[i + 1].R = Rn;
    state[i + 1].FB = FB + (final_ok ? FS * width : 0);
  }
  zero_words(lb_pivot, (Rn + kBatchPivotTile - 1) / kBatchPivotTile + kLbExtra);
}

}  // namespace

void launch_filter_many(const GraphDev &g, const FilterDesc *fds, uint32_t *const *bm_out,
                        unsigned long long *sizes, int32_t nq, int32_t n_words,
                        cudaStream_t s) {
  if (nq <= 0) return;
  if (sizes) cudaMemsetAsync(sizes, 0, sizeof(unsigned long long) * nq * kMaxK, s);
  if (g.thr && n_words > 0) {
    const dim3 grid(filter_grid(n_words), nq);
    if (n_words % 4 == 0)
      k_b_filter_bits<4><<<grid, 256, 0, s>>>(g, fds, bm_out, sizes);
    else
      k_b_filter_bits<1><<<grid, 256, 0, s>>>(g, fds, bm_out, sizes);
    return;
  }
  const int gx = (int)std::min<int64_t>((n_words + 7) / 8, 128);
  k_b_filter<<<dim3(std::max(gx, 1), nq), 256, 0, s>>>(g, fds, bm_out, sizes);
}

namespace {
size_t level_smem(int32_t block) {
  return sizeof(int32_t) * ((size_t)block * kItemsPerThread * 5 + 4);
}
}  // namespace

void batch_setup() {
  cudaFuncSetAttribute(k_b_level<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)level_smem(1024));
}

int batch_enqueue(const GraphDev &g, const BatchArgs &a, cudaStream_t s) {
  const int32_t B = a.block, G = a.grid;
  const int32_t tile_items = B * kItemsPerThread;
  const int64_t list_tiles = ((int64_t)a.nq * a.n_words + kBatchListTile - 1) / kBatchListTile;
  k_b_init<<<(unsigned)std::min<int64_t>((list_tiles + 2 * a.nq) / 256 + 1, G), 256, 0, s>>>(
      a.state, a.overflow, a.counts, 2 * (int64_t)a.nq, a.lb_list, list_tiles + kLbExtra);
  // filter: one CTA row per query (nothing reads the sizes here)
  launch_filter_many(g, a.fds, a.bm_out, g.thr ? nullptr : a.sizes, a.nq, a.n_words, s);
  // level 1: every query's candidate list for its first matched vertex
  k_b_list<<<(unsigned)std::max<int64_t>(std::min<int64_t>(list_tiles, G), 1), 256, 0, s>>>(
      g, a.qs, a.nq, a.list_off, a.state, std::min(a.cap_rows, a.cap_elems), a.F[0], a.rseg[0],
      a.counts, a.lb_list, a.lb_pivot, a.spin_limit, a.scan_stall_tile, a.overflow);
  int launches = 3;
  for (int32_t i = 1; i < a.kmax; ++i) {
    const int cur = (i - 1) & 1, nxt = i & 1;
    k_b_pivot_scan<<<G, 256, 0, s>>>(g, a.qs, i, a.state, a.F[cur], a.rseg[cur], a.pstart,
                                     a.pslot, a.woff, a.tile_row, tile_items, a.cap_rows,
                                     a.cap_elems, a.cap_items, a.lb_pivot, a.lb_level,
                                     a.spin_limit, a.scan_stall_tile, a.overflow);
    auto level = [&](auto kernel) {
      kernel<<<G, B, level_smem(B), s>>>(g, a.qs, i, a.state, a.F[cur], a.rseg[cur], a.pstart,
                                         a.pslot, a.woff, a.tile_row, a.cap_rows, a.cap_elems,
                                         a.cap_final, a.counts, a.F[nxt], a.rseg[nxt],
                                         a.final_rows, a.lb_level, a.lb_pivot, a.spin_limit,
                                         a.stall_tile, a.overflow);
    };
    B <= 256 ? level(k_b_level<256>) : level(k_b_level<1024>);
    launches += 2;
  }
  return launches;
}

}  // namespace gsm
