// Internal interface of the batched form (batch.cu) for the host driver.
#pragma once

#include <cstddef>
#include <cstdint>

#include "kernels.cuh"

namespace gsm {

// Verification level i of one query (extending rows of width i by pi_i).
struct BatchLevel {
  const uint32_t *bitmap;   // C(pi_i); null: every entry of a cut label segment is in it
  int32_t lab;              // dense label of pi_i (the row segment traversed)
  int32_t rlo, rhi;         // bounds of the new vertex, as in LevelDesc
  int8_t cut, ngt, nb, ninj;
  int8_t gt[kMaxK];
  int8_t bpos[kMaxK];       // row positions of pi_i's mapped query neighbours
  int8_t inj[kMaxK];        // same-label, non-adjacent positions
};

struct BatchQuery {
  int32_t k;
  // counted queries: rows of width kc are whole but for the leaves (LeafDesc);
  // listed queries: kc = k, no leaves
  int32_t kc;
  int32_t enumerate;            // 1: the last level writes result rows
  int32_t word0;                // first word of root_bitmap that can be non-zero
  const uint32_t *root_bitmap;  // C(pi_0)
  int8_t out_col[kMaxK];        // result column of row position j (= pi_j)
  LeafDesc leaf;
  BatchLevel lv[kMaxK];         // lv[1 .. kc-1]
};

// Device-side sizes of one level (rows at level i and their leading dimension,
// candidates checked while extending it, tiles, survivors that continue; FB =
// first element of the step's result rows in the result arena, FS = result
// rows the step writes).
struct BatchStep {
  int64_t R, ld, W, tiles, S, FB, FS;
};

constexpr int32_t kBatchOverflow = 1, kBatchTimeout = 2;  // values of BatchArgs::overflow
constexpr int64_t kBatchListTile = 1024;   // root-bitmap words a list tile covers
constexpr int64_t kBatchPivotTile = 256;   // rows a pivot tile covers
constexpr int64_t kBatchMinTile = 128 * kItemsPerThread;  // candidates of the smallest level tile

struct BatchArgs {
  int32_t nq, kmax, n_words;
  int32_t block, grid;
  int64_t cap_rows, cap_elems, cap_items;
  const FilterDesc *fds;          // [nq]
  uint32_t *const *bm_out;        // [nq] bitmap output of each query
  const BatchQuery *qs;           // [nq]
  const int64_t *list_off;        // [nq + 1] root-bitmap words of the queries before
  // what the host reads back, in one piece: the steps, the overflow flag and
  // the counts (per query the sums of the low and high 32-bit halves)
  BatchStep *state;               // [kMaxK + 1]
  int32_t *overflow;
  unsigned long long *counts;     // [2 * nq]
  unsigned long long *sizes;      // [nq * kMaxK] |C(u)| (graphs without threshold bitmaps)
  int32_t *F[2], *rseg[2];        // frontiers: cap_elems / cap_rows each
  int32_t *pstart;                // [cap_rows]
  uint8_t *pslot;                 // [cap_rows]
  int64_t *woff;                  // [cap_rows + 1]
  int32_t *tile_row;              // [cap_items / kBatchMinTile + 2]
  // look-back words, each array followed by kLbExtra of them
  unsigned long long *lb_list;    // [nq * n_words / kBatchListTile + 1 + kLbExtra]
  unsigned long long *lb_pivot;   // [cap_rows / kBatchPivotTile + 1 + kLbExtra]
  unsigned long long *lb_level;   // [cap_items / kBatchMinTile + 1 + kLbExtra]
  int32_t spin_limit;
  // fault injection (-1: none): tiles that never publish their look-back words,
  // of the levels, and of the list and the pivot scans
  int32_t stall_tile, scan_stall_tile;
  // enumerate batches: result rows of the queries that list them (null: a
  // counting batch).  The rows of step i (queries with k = i + 1) are
  // row-major, k ints each, in query-id column order, from element
  // state[i].FB on; within a step the queries follow batch order, each query's
  // rows in lexicographic order of its matching order.
  int64_t cap_final;              // arena elements
  int32_t *final_rows;            // [cap_final]
};

// The candidate filter of nq queries in one launch: query j's FilterDesc is
// fds[j], its k bitmaps go to bm_out[j], |C(u)| to sizes[j * kMaxK + u]
// (zeroed here).  fds and bm_out are device arrays.
void launch_filter_many(const GraphDev &g, const FilterDesc *fds, uint32_t *const *bm_out,
                        unsigned long long *sizes, int32_t nq, int32_t n_words,
                        cudaStream_t s);

// Raises the dynamic shared memory limit of the batch kernels on the current
// device (once per device; before the first capture).
void batch_setup();

// Issues the whole batch on stream s (no host synchronisation, fixed launch
// shapes, so the sequence can be captured as a CUDA graph).  Returns the
// number of kernels launched.
int batch_enqueue(const GraphDev &g, const BatchArgs &a, cudaStream_t s);

}  // namespace gsm
