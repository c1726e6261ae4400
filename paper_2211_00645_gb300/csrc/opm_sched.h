// Work units of the fast projection and their static schedule onto the
// persistent CTAs.
#pragma once

#include <algorithm>
#include <cstdint>

#ifndef __CUDACC__
#define __align__(n) alignas(n)  // host-only builds of this header
#endif

namespace opm {

// Rows [ks, ke) of j-tile jt at x-tile xt of item `item` (0 for a single
// stack).  `list` and `seq` are scheduling scratch.  (The batch's general
// units: `pad` columns from column jt.)
struct __align__(16) WorkUnit {
  int item, xt, jt, ks, ke;
  int list, seq, pad;
};
static_assert(sizeof(WorkUnit) == 32, "WorkUnit is 32 bytes");

// Largest and smallest rows per work unit of the single-stack fast
// projection, the average units per CTA list the plan's choice between them
// aims for, and columns x per unit (one TMA box row of the fast kernels).
constexpr int kChunkRows = 256;
constexpr int kMinChunkRows = 16;
constexpr double kUnitsPerList = 1.1;
constexpr int kUnitX = 128;

// Upper bound on the number of CTA lists (4 CTAs per SM on up to 256 SMs).
constexpr int kMaxLists = 1024;

// Cost of a unit in ring stages (two camera rows each), plus a fixed
// per-unit term for the job's set-up and its z-MIP fold.
inline int unit_cost(const WorkUnit& u) { return (u.ke - u.ks + 1) / 2 + 3; }

// Moves units[i] to place units[i].seq, a permutation of 0 .. n - 1, in place.
inline void permute_units(WorkUnit* units, int n) {
  for (int i = 0; i < n; ++i)
    while (units[i].seq != i) std::swap(units[i], units[units[i].seq]);
}

// Longest-processing-time-first schedule: units are taken by decreasing
// cost (ties in the given order) and each goes to the list with the least
// load so far (ties to the lowest list).  On return `units` is ordered list
// by list, each list in the order its units were assigned, and
// offsets[l] .. offsets[l + 1] delimit list l (offsets has nlists + 1
// entries).  In place and without allocation; nlists <= kMaxLists.  The two
// orderings are counting sorts (a batch of 2816 general units is set in 137 us on
// the host, 208 with two comparison sorts); costs beyond kCosts, of units of more
// than 4000 rows, share a bucket and are sorted there.
inline void schedule_lpt(WorkUnit* units, int n, int nlists, int* offsets) {
  constexpr int kCosts = 2048;
  int first[kCosts > kMaxLists ? kCosts : kMaxLists];
  const auto bucket = [](const WorkUnit& u) { return std::max(0, kCosts - 1 - unit_cost(u)); };  // the dearest first
  std::fill(first, first + kCosts, 0);
  for (int i = 0; i < n; ++i) first[bucket(units[i])] += 1;
  const int beyond = first[0];
  for (int b = 0, at = 0; b < kCosts; ++b) {
    const int here = first[b];
    first[b] = at;
    at += here;
  }
  for (int i = 0; i < n; ++i) units[i].seq = first[bucket(units[i])]++;
  permute_units(units, n);
  if (beyond > 1)
    std::sort(units, units + beyond, [](const WorkUnit& a, const WorkUnit& b) {
      const int ca = unit_cost(a), cb = unit_cost(b);
      return ca != cb ? ca > cb : a.seq < b.seq;
    });
  // binary min-heap of (load, list)
  int64_t hload[kMaxLists];
  int hlist[kMaxLists];
  for (int l = 0; l < nlists; ++l) {
    hload[l] = 0;
    hlist[l] = l;
  }
  for (int i = 0; i < n; ++i) {
    const int64_t load = hload[0] + unit_cost(units[i]);
    const int list = hlist[0];
    units[i].list = list;
    // sift the grown root down
    int r = 0;
    for (int m; (m = 2 * r + 1) < nlists; r = m) {
      if (m + 1 < nlists && (hload[m + 1] != hload[m] ? hload[m + 1] < hload[m] : hlist[m + 1] < hlist[m])) m += 1;
      if (hload[m] != load ? hload[m] > load : hlist[m] > list) break;
      hload[r] = hload[m];
      hlist[r] = hlist[m];
    }
    hload[r] = load;
    hlist[r] = list;
  }
  for (int l = 0; l < nlists; ++l) first[l] = 0;
  for (int i = 0; i < n; ++i) first[units[i].list] += 1;
  offsets[0] = 0;
  for (int l = 0; l < nlists; ++l) {
    offsets[l + 1] = offsets[l] + first[l];
    first[l] = offsets[l];
  }
  for (int i = 0; i < n; ++i) units[i].seq = first[units[i].list]++;
  permute_units(units, n);
}

}  // namespace opm
