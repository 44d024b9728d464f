// Static tile schedule of a grouped GEMM launch.
//
// A grouped launch walks one work list (the tiles of all its problems) with a fixed set of
// persistent units (CTAs, or CTA pairs).  Dealing the list out round-robin gives every unit the
// same NUMBER of tiles, which is only balanced when the tiles cost the same.  The launches of the
// gated factorized layer mix tiles of different length: in H' = X Q^T and dH' = dY P the FFN
// matrices contract over 3072 features (48 k-blocks) next to attention matrices that contract
// over 768 (12 k-blocks).  The host therefore assigns tiles to units with the longest-processing-time rule (sort by cost,
// always hand the next tile to the least loaded unit) and passes the per-unit lists to the kernel
// as a table in its parameter block; every role of a unit (TMA producer, MMA issuer, epilogue
// warps, and both CTAs of a pair) walks the same list, so no run-time hand-over is needed.
// Launches with more work items than the table holds keep the round-robin order (with that many
// tiles per unit the imbalance is small anyway).
#pragma once
#include <stdint.h>

#ifndef __CUDACC_RTC__
#include <algorithm>
#include <vector>
#endif

namespace flop {
namespace tc {

constexpr int kMaxSched = 2048;   // work items a table can hold
constexpr int kSchedProblemShift = 11;   // grouped launches: entry = (problem index << 11) | work-list index
constexpr int kMaxUnits = 148;    // persistent CTAs (one-CTA kernel) or pairs (two-CTA kernel)

struct Schedule {
  int n_units;                       // 0: no table, round-robin over the work list
  uint16_t begin[kMaxUnits + 1];     // unit u walks item[begin[u] .. begin[u+1])
  uint16_t item[kMaxSched];          // work-list indices
};

// Work items of equal cost: first, first + stride, ... (count of them), of one problem.
struct ItemGroup { double cost; int rank, problem, first, count, stride; };

// Longest-processing-time assignment of the items of `groups` to `units` units: groups of a lower rank first, within a rank the
// costlier first (ties keep list order, so that neighbouring tiles share operand tiles in L2), every item to the least
// loaded unit.  Returns the largest unit load and fills the table; `shift` > 0 adds the problem index to the entries.
// rank is 0 except in launches whose tile count only the device knows: there it is the index of a tile along the extent that
// may end early.  Any prefix of the ranks is then balanced, whereas one list over all tiles leaves units with several live
// tiles next to units with none once the later tiles turn out empty (open components only, BERT shapes, a quarter of the
// gates open: the backward launches 39.5 -> 32.1 and 44.9 -> 39.8 us).
// Groups rather than items are sorted, the heap holds plain pairs and nothing is allocated per unit: a table is built for
// every launch, and at 500 items the item-wise form took longer than the launch it was for.
inline double deal_groups(std::vector<ItemGroup>& groups, int n, int units, int shift, Schedule* out) {
  out->n_units = 0;
  if (n <= 0 || n > kMaxSched || units <= 0 || units > kMaxUnits) return -1.0;
  std::stable_sort(groups.begin(), groups.end(), [](const ItemGroup& a, const ItemGroup& b) { return a.rank != b.rank ? a.rank < b.rank : a.cost > b.cost; });
  struct Slot { double load; int unit; };
  Slot heap[kMaxUnits];              // least loaded first, ties to the lower unit index
  for (int u = 0; u < units; ++u) heap[u] = Slot{0.0, u};
  uint8_t owner[kMaxSched];
  uint16_t entry[kMaxSched];
  int held[kMaxUnits + 1] = {};
  int pos = 0;
  for (const ItemGroup& g : groups)
    for (int i = 0; i < g.count; ++i, ++pos) {
      const int u = heap[0].unit;
      owner[pos] = (uint8_t)u;
      entry[pos] = (uint16_t)((shift ? g.problem << shift : 0) | (g.first + i * g.stride));
      ++held[u];
      const Slot s{heap[0].load + g.cost, u};
      int at = 0;
      for (;;) {                     // sift the unit down from the top
        int c = 2 * at + 1;
        if (c >= units) break;
        if (c + 1 < units && (heap[c + 1].load < heap[c].load || (heap[c + 1].load == heap[c].load && heap[c + 1].unit < heap[c].unit))) ++c;
        if (s.load < heap[c].load || (s.load == heap[c].load && s.unit < heap[c].unit)) break;
        heap[at] = heap[c];
        at = c;
      }
      heap[at] = s;
    }
  double makespan = 0.0;
  for (int u = 0; u < units; ++u) makespan = std::max(makespan, heap[u].load);
  int next[kMaxUnits], sum = 0;
  for (int u = 0; u < units; ++u) { out->begin[u] = (uint16_t)sum; next[u] = sum; sum += held[u]; }
  for (int u = units; u <= kMaxUnits; ++u) out->begin[u] = (uint16_t)sum;
  for (int i = 0; i < pos; ++i) out->item[next[owner[i]]++] = entry[i];
  out->n_units = units;
  return makespan;
}

// Largest load of the round-robin deal (item i to unit i % units); true when it is within 3 % of the lower bound
// max(mean load, longest item), so that a table has nothing to gain, and when a table could not name the units at all (more
// than kMaxUnits).  `groups` in work-list order.
inline bool round_robin_is_good(const std::vector<ItemGroup>& groups, int units, double* rr_makespan) {
  if (rr_makespan) *rr_makespan = 0.0;
  if (units <= 0 || units > kMaxUnits) return true;
  double load[kMaxUnits] = {};
  double total = 0.0, longest = 0.0, rr = 0.0;
  for (const ItemGroup& g : groups) {
    for (int i = 0; i < g.count; ++i) load[(g.first + i * g.stride) % units] += g.cost;
    total += g.cost * g.count;
    longest = std::max(longest, g.cost);
  }
  for (int u = 0; u < units; ++u) rr = std::max(rr, load[u]);
  if (rr_makespan) *rr_makespan = rr;
  return rr <= 1.03 * std::max(total / units, longest);
}

// The same for a plain list of costs (item i costs cost[i]); returns the largest unit load, or -1 without a table.
inline double build_schedule(const std::vector<double>& cost, int units, Schedule* out, double* rr_makespan) {
  const int n = (int)cost.size();
  out->n_units = 0;
  if (rr_makespan) *rr_makespan = 0.0;
  if (units <= 0 || units > kMaxUnits) return -1.0;
  std::vector<ItemGroup> groups;
  groups.reserve((size_t)n);
  for (int i = 0; i < n; ++i) groups.push_back(ItemGroup{cost[(size_t)i], 0, 0, i, 1, 1});
  if (round_robin_is_good(groups, units, rr_makespan) && rr_makespan) return -1.0;
  return deal_groups(groups, n, units, 0, out);
}

// Queue of a chained launch (gemm_tc2_chain.cuh): the work list holds the tiles of two stages, a tile of the
// second stage waits for first-stage tiles, and the persistent units draw tiles from the head of one queue.
// All first-stage tiles must therefore come before all second-stage tiles (a drawn tile then only waits for
// tiles that some unit already works on, so no wait can be circular).  Inside a stage the queue follows `key`
// (ties keep list order): the caller puts first what other tiles wait for, long tiles before short ones, and
// orders consumers like their producers.  out->item holds the queue (n_units = 1 marks the table as valid).
// Returns false when the table cannot hold the launch (the kernel then walks the work list in its own order,
// which the caller keeps stage-ordered).
inline bool build_chain_queue(const std::vector<int>& stage, const std::vector<int64_t>& key, Schedule* out) {
  const int n = (int)stage.size();
  out->n_units = 0;
  if (n == 0 || n > kMaxSched || (int)key.size() != n) return false;
  std::vector<int> order((size_t)n);
  for (int i = 0; i < n; ++i) order[(size_t)i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    const int sa = stage[(size_t)a] != 0, sb = stage[(size_t)b] != 0;
    if (sa != sb) return sa < sb;
    return key[(size_t)a] < key[(size_t)b];
  });
  for (int i = 0; i < n; ++i) out->item[i] = (uint16_t)order[(size_t)i];
  out->begin[0] = 0;
  for (int u = 1; u <= kMaxUnits; ++u) out->begin[u] = (uint16_t)n;
  out->n_units = 1;
  return true;
}

}  // namespace tc
}  // namespace flop
