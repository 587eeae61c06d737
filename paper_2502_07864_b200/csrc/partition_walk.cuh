// The producer warp's walk over its partition's sequences and pages, shared by the split-KV kernels on the tensor path.
#pragma once
#include "common.cuh"

namespace transmla {
namespace sm100 {

struct PartitionWalk {
  const int32_t* page_table;
  const int32_t* seqlens;
  const int32_t* cum;
  int32_t* counters;      // page counters of this block of query rows, one per sequence (run-time claims)
  float* partial_lse;
  int part;               // the CTA's partition
  int row0, rows;         // first query row and row count of the block
  int SH, max_pages, dynamic;
};

// Calls queries(b, slot, L) at the start of every segment (the part of sequence b that this CTA works on; its partial
// goes to `slot`) and page(b, page number within the sequence, first of the segment, last of the segment) for each of
// its pages.  All lanes of the warp call it together, with the partition's row of the plan.
template <class Queries, class Page>
__device__ __forceinline__ void walk_partition(const PartitionWalk& w, int4 pl, int lane, Queries&& queries, Page&& page) {
  constexpr uint32_t kAll = 0xffffffffu;
  auto empty_partial = [&](int slot) {
    for (int i = lane; i < w.rows && w.row0 + i < w.SH; i += 32)
      w.partial_lse[static_cast<size_t>(slot) * w.SH + w.row0 + i] = -INFINITY;
  };
  // Page-table entries [lo, hi) of sequence b are asked into L1 ahead of their use (one 128-byte line per lane
  // and round), so that the look-up in front of every page load does not cost a trip to L2.
  auto prefetch_table = [&](int b, int lo, int hi) {
    const int32_t* row = w.page_table + static_cast<size_t>(b) * w.max_pages;
    for (int i = (lo & ~31) + lane * 32; i < hi; i += 32 * 32)
      asm volatile("prefetch.global.L1 [%0];" ::"l"(row + max(i, lo)));
  };
  // The last sequence in which this partition owns pages: there it claims until the counter runs dry.  In the
  // sequences before it (a partition that straddles two or more) it takes no more pages than the plan gave it,
  // so that every sequence gets the share of CTA time that the plan meant it to have.
  int last_home = pl.w;
  if (w.dynamic) {
    const int cw = w.cum[pl.w], cw1 = w.cum[pl.w + 1];
    if (min(pl.y, cw1) <= max(pl.x, cw + kSegCost)) --last_home;
  }
  for (int b = pl.z; b <= pl.w; ++b) {
    const int cb = w.cum[b], cb1 = w.cum[b + 1];  // one round trip for the three of them
    const int L = clamped_len(w.seqlens[b], w.max_pages, nullptr);  // the plan block has already reported a bad length
    const int c0s = cb + kSegCost;  // slot of page 0 of sequence b
    const int pg_lo = max(pl.x, c0s) - c0s, pg_hi = min(pl.y, cb1) - c0s;
    if (pg_hi <= pg_lo) continue;
    const int slot = w.part + b;
    if (!w.dynamic) {  // exactly the plan's range
      prefetch_table(b, pg_lo, pg_hi);
      queries(b, slot, L);
      for (int pj = pg_lo; pj < pg_hi; ++pj) page(b, pj, pj == pg_lo, pj == pg_hi - 1);
      continue;
    }
    // Pages of sequence b from its counter until it runs dry.  Three are claimed in one go (one atomic
    // instruction, lanes 0..2) so that the stages fill at once.  After that the next two page numbers are
    // always in hand and the claim behind them is in flight while a page waits for its stage, which keeps the
    // counter's round trip off the critical path and tells at issue time whether a page is the segment's
    // last one: it is exactly when the claim behind it is past the end (claims only grow).
    const int n_b = cb1 - c0s;
    int32_t* counter = w.counters + b;
    int left = b < last_home ? pg_hi - pg_lo : 0x7fffffff;  // claims this partition may still make here
    const int take = min(3, left);
    left -= take;
    int head = 0x7fffffff;
    if (lane < take) head = atomicAdd(counter, 1);
    prefetch_table(b, 0, n_b);  // in flight together with the claim
    int c0 = __shfl_sync(kAll, head, 0), c1 = __shfl_sync(kAll, head, 1), c2 = __shfl_sync(kAll, head, 2);
    { int t; if (c0 > c1) { t = c0; c0 = c1; c1 = t; } if (c1 > c2) { t = c1; c1 = c2; c2 = t; } if (c0 > c1) { t = c0; c0 = c1; c1 = t; } }
    if (c0 >= n_b) {  // the others have taken everything: the combine still expects a partial from this slot
      empty_partial(slot);
      continue;
    }
    queries(b, slot, L);
    bool first = true;
    while (c0 < n_b) {
      int pend = 0x7fffffff;
      const bool ahead = c2 < n_b && left > 0;
      if (ahead) { --left; if (lane == 0) pend = atomicAdd(counter, 1); }
      page(b, c0, first, c1 >= n_b);
      first = false;
      c0 = c1;
      c1 = c2;
      c2 = ahead ? __shfl_sync(kAll, pend, 0) : 0x7fffffff;
    }
  }
}

}  // namespace sm100
}  // namespace transmla
