// How much memory a search asks for at once. Plain functions, so that the host
// tests run the same code.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace sindi {

constexpr int kPlainLanes = 24;            // plain schedule: query chains in flight at once, launched one by one
constexpr int kGraphLanes = 56;            // and in a recorded graph, at most (graph_lanes)
constexpr uint32_t kSplitMinWindows = 8;   // plain schedule: a query of this many windows or more scans
                                           // its first windows in a launch of their own
constexpr size_t kGraphLaneBytes = (size_t)512 << 20;  // workspaces of a graph of more than kPlainLanes chains, at most

// Chains in flight of the plain schedule's recorded graph. A chain is a few microseconds of scan on many SMs and then
// latency on few, so a long call gains from more of them than the host can feed launch by launch; measured, ms a
// call of 1,000 queries (300 in the last row):
//   chains                       24    40    56    64
//   1M documents, 62 windows   2.89  2.76  2.74  2.75
//   300k, 37 windows           2.07  1.47  1.36  1.37
//   200k, 13 windows           1.96  1.34  1.11  1.10
//   400k, 25 windows           0.70  0.56  0.56  0.55
// A chain holds several queries, and an index of a few windows keeps 24 (100 exact queries over three windows: 24
// chains 109 us, 32 120, 40 122). Every chain keeps a workspace of lane_bytes while the graph lives: 0.5 MB each at
// 1M documents and 500 candidates, 141 MB at 8.8M and 8,192, where a query's windows fill the device by themselves;
// kGraphLaneBytes bounds what the chains beyond kPlainLanes may bring the total to.
inline int graph_lanes(uint32_t sigma, int64_t n_queries, size_t lane_bytes) {
    int64_t lanes = kPlainLanes;
    if (sigma >= kSplitMinWindows) {
        const int64_t fit = (int64_t)(kGraphLaneBytes / std::max<size_t>(lane_bytes, 1));
        lanes = std::max<int64_t>(lanes, std::min<int64_t>({(int64_t)kGraphLanes, n_queries / 5, fit}));
    }
    return (int)std::min<int64_t>(lanes, n_queries);
}

// The largest of n, ceil(n / 2), ceil(n / 4), ... 1 for which get(size) succeeds; 0 if none does.
template <typename Get>
int64_t largest_that_fits(int64_t n, Get&& get) {
    for (; n >= 1; n = (n + 1) / 2) {
        if (get(n)) return n;
        if (n == 1) break;
    }
    return 0;
}

}  // namespace sindi
