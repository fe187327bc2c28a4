// Candidate filter body shared by the single-query and batched kernels
// (Sec. 3.2 filtering: label, degree and per-label neighbour counts).
#pragma once

#include "kernels.cuh"

namespace gsm {

// Requirement test of query vertex set `vneed` against per-slot neighbour
// counts cnt[] (slot s counts neighbours labelled d.slot_label[s]).
template <typename Desc>
__device__ __forceinline__ uint32_t nlc_pass(const Desc &d, uint32_t vneed,
                                             const int32_t (&cnt)[kMaxK]) {
  uint32_t pass = 0;
  for (int u = 0; u < d.k; ++u) {
    if (!((vneed >> u) & 1u)) continue;
    bool ok = true;
    for (int r = 0; r < d.nreq[u]; ++r) {
      const int slot = d.req_slot[u][r];
      int32_t c = 0;
#pragma unroll
      for (int s = 0; s < kMaxK; ++s) c = (s == slot) ? cnt[s] : c;
      ok = ok && c >= d.req_cnt[u][r];
    }
    if (ok) pass |= 1u << u;
  }
  return pass;
}

// Words of a bitmap that one thread of the filter handles together: four (one
// 16-byte load or store) when the bitmaps' words are a multiple of four, so
// that every bitmap starts on a 16-byte boundary, else one.
template <int kV>
struct FilterWords {
  uint32_t w[kV];
  __device__ __forceinline__ void load(const uint32_t *p) {
    if constexpr (kV == 4) {
      const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
      w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
    } else {
      w[0] = __ldg(p);
    }
  }
  __device__ __forceinline__ void store(uint32_t *p) const {
    if constexpr (kV == 4)
      *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    else
      *p = w[0];
  }
};

// Words at .. at + kV - 1 of C(u) from the graph's threshold and label bitmaps:
// the filter's tests for 32 vertices are ands of words.  A requirement above
// kThrLevels neighbours takes the top bitmap and then looks the counts of the
// vertices left up one by one.  (Enough neighbours of every label are enough
// neighbours, so the degree needs no test of its own beside them; with one
// label the bitmaps hold degrees.)
template <int kV, typename Desc>
__device__ __forceinline__ FilterWords<kV> filter_word(const GraphDev &g, const Desc &d, int u,
                                                       int32_t at) {
  FilterWords<kV> word;
  word.load(g.lab_bits + (int64_t)d.qlab[u] * d.n_words + at);
  const bool one = g.num_labels == 1;
  const int nr = one ? (d.qdeg[u] > 0 ? 1 : 0) : d.nreq[u];
  uint32_t deep = 0;  // requirements above the bitmaps' levels
  for (int r = 0; r < nr; ++r) {
    const int32_t l = one ? 0 : d.slot_label[d.req_slot[u][r]];
    const int32_t c = one ? d.qdeg[u] : d.req_cnt[u][r];
    FilterWords<kV> t;
    t.load(g.thr + ((int64_t)l * kThrLevels + min(c, kThrLevels) - 1) * d.n_words + at);
#pragma unroll
    for (int j = 0; j < kV; ++j) word.w[j] &= t.w[j];
    if (c > kThrLevels) deep |= 1u << r;
  }
#pragma unroll
  for (int j = 0; j < kV; ++j) {
    const int32_t v0 = (at + j) * 32;
    const int32_t lo = d.lo[u] - v0, hi = d.hi[u] - v0;  // the restriction inside the word
    if (lo > 0) word.w[j] &= lo < 32 ? ~0u << lo : 0u;
    if (hi < 32) word.w[j] &= hi > 0 ? ~0u >> (32 - hi) : 0u;
    if (!deep || !word.w[j]) continue;
    for (uint32_t m = word.w[j]; m; m &= m - 1) {
      const int bit = __ffs(m) - 1;
      const int64_t v = v0 + bit;
      bool ok = true;
      for (uint32_t x = deep; x && ok; x &= x - 1) {
        const int r = __ffs(x) - 1;
        if (one)
          ok = __ldg(g.rp + v + 1) - __ldg(g.rp + v) >= d.qdeg[u];
        else
          ok = (int32_t)__ldg(g.nlc + v * g.nlc_stride + d.slot_label[d.req_slot[u][r]]) >=
               d.req_cnt[u][r];
      }
      if (!ok) word.w[j] &= ~(1u << bit);
    }
  }
  return word;
}

// Words of C(u) for u = u0, u0 + du, ... of one query: thread t of the grid's
// x dimension takes kV words (filter_grid), so a warp's loads and stores are
// contiguous.  sizes (may be null) gains |C(u)|.  Bound by L2 and the bitmaps
// written: 256 queries on R-MAT 18 (13.6 M words) take 37 us with four
// words a thread, 71 with one, where a test per vertex, query and query vertex
// took 1,435 us (under ncu).
template <int kV, typename Desc>
__device__ __forceinline__ void filter_words(const GraphDev &g, const Desc &d,
                                             uint32_t *__restrict__ bitmaps,
                                             unsigned long long *__restrict__ sizes, int u0,
                                             int du) {
  const int32_t at = (blockIdx.x * blockDim.x + threadIdx.x) * kV;
  for (int u = u0; u < d.k; u += du) {
    int32_t c = 0;
    if (at < d.n_words) {
      const FilterWords<kV> word = filter_word<kV>(g, d, u, at);
      word.store(bitmaps + (int64_t)u * d.n_words + at);
#pragma unroll
      for (int j = 0; j < kV; ++j) c += __popc(word.w[j]);
    }
    if (sizes) {
      c = __reduce_add_sync(0xffffffffu, c);
      if ((threadIdx.x & 31) == 0 && c) atomicAdd(sizes + u, (unsigned long long)c);
    }
  }
}
// CTAs of 256 threads in x for bitmaps of n_words words.
inline unsigned filter_grid(int32_t n_words) {
  const int32_t per = n_words % 4 ? 256 : 1024;
  return (unsigned)((n_words + per - 1) / per);
}

// One warp handles 32 consecutive data vertices per iteration (warps
// warp_id, warp_id + n_warps, ...).  Each lane first applies the label /
// degree / range test for its own vertex.  With the graph's neighbour label
// count table the requirements are read from it; otherwise they are counted
// from the rows, as follows.  A vertex that also needs per-label
// neighbour counts is first counted by its own lane over its first
// kLaneScan neighbours (most rows of a power-law graph end there); only a
// vertex whose requirements are still unmet and whose row goes on is then
// scanned by the whole warp (coalesced reads of the CSR row, labels gathered
// through L2).  The k bitmap words of the group are formed by ballots.  Lane u
// adds |C(u)| into sizes[u].
constexpr int kLaneScan = 32;
template <typename Desc>
__device__ __forceinline__ void filter_warps(const GraphDev &g, const Desc &d,
                                             uint32_t *__restrict__ bitmaps,
                                             unsigned long long *__restrict__ sizes,
                                             int64_t warp_id, int64_t n_warps) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  unsigned long long my_size = 0;  // lane u accumulates |C(u)|
  for (int64_t grp = warp_id; grp < d.n_words; grp += n_warps) {
    const int64_t v64 = grp * 32 + lane;
    const bool valid = v64 < g.n;
    const int32_t v = (int32_t)v64;
    int32_t lv = -1, deg = -1;
    if (valid) {
      lv = g.lab[v];
      deg = g.rp[v + 1] - g.rp[v];
    }
    uint32_t pre = 0, need = 0;
    if (valid)
      for (int u = 0; u < d.k; ++u) {
        if (lv == d.qlab[u] && deg >= d.qdeg[u] && v >= d.lo[u] && v < d.hi[u]) {
          pre |= 1u << u;
          if (d.nreq[u] > 0) need |= 1u << u;
        }
      }
    uint32_t result = pre & ~need;
    bool rest = false;
    if (need) {
      const int32_t b = g.rp[v], e = g.rp[v + 1];
      const int32_t e1 = min(e, b + kLaneScan);
      int32_t cnt[kMaxK];
#pragma unroll
      for (int s = 0; s < kMaxK; ++s) cnt[s] = 0;
#pragma unroll 4
      for (int32_t idx = b; idx < e1; ++idx) {
        const int32_t lw = __ldg(g.lab + __ldg(g.col + idx));
#pragma unroll
        for (int s = 0; s < kMaxK; ++s)
          if (s < d.nslots && lw == d.slot_label[s]) ++cnt[s];
      }
      const uint32_t pass = nlc_pass(d, need, cnt);
      result |= pass;
      rest = pass != need && e > e1;
      need = rest ? need : 0;
    }
    uint32_t todo = __ballot_sync(kFull, rest);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int32_t vv = (int32_t)(grp * 32 + src);
      const uint32_t vneed = __shfl_sync(kFull, need, src);
      const int32_t b = g.rp[vv], e = g.rp[vv + 1];
      int32_t cnt[kMaxK], tot[kMaxK];
#pragma unroll
      for (int s = 0; s < kMaxK; ++s) cnt[s] = tot[s] = 0;
      uint32_t pass = 0;
      // Scan the row 256 neighbours at a time and stop as soon as every
      // requirement holds (counts only grow), so hubs end after one chunk.
      for (int32_t base = b; base < e; base += 256) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int32_t idx = base + j * 32 + lane;
          if (idx < e) {
            const int32_t lw = __ldg(g.lab + __ldg(g.col + idx));
#pragma unroll
            for (int s = 0; s < kMaxK; ++s)
              if (s < d.nslots && lw == d.slot_label[s]) ++cnt[s];
          }
        }
#pragma unroll
        for (int s = 0; s < kMaxK; ++s)
          if (s < d.nslots) tot[s] = __reduce_add_sync(kFull, cnt[s]);
        pass = nlc_pass(d, vneed, tot);
        if (pass == vneed) break;  // warp-uniform: tot is the same in every lane
      }
      if (lane == src) result |= pass;
    }
    for (int u = 0; u < d.k; ++u) {  // d.k is warp-uniform
      const uint32_t word = __ballot_sync(kFull, (result >> u) & 1u);
      if (lane == u) {
        bitmaps[(int64_t)u * d.n_words + grp] = word;
        my_size += __popc(word);
      }
    }
  }
  if (lane < d.k && my_size) atomicAdd(sizes + lane, my_size);
}

}  // namespace gsm
