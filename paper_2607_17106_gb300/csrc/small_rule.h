// small_rule.h -- which searches run whole in one thread-block cluster.
#ifndef BFSGB_SMALL_RULE_H
#define BFSGB_SMALL_RULE_H

#include <cstdint>

#include "../../include/bfs.h"

namespace bfsgb {

// What the rule looks at of a graph: vertices, those with an edge, entries, maximum degree.
struct SmallGraph {
    int64_t n, n1, m;
    int32_t deg_max;
};

// In the cluster a level's barrier and counter read take 0.7 us, grid-wide 2.0,
// and the launch is cheaper; but 16 SMs do a level's work, not 152.  That pays
// where no level has much of it: up to three vertices with an edge for each of
// the cluster's 16,384 threads, and dense levels that pull, so that most rows
// end at their first entries.  us a search, 16 in a call (RMAT-10 and -14: 4),
// grid-wide / cluster:
//   RMAT, edge factor 16 (a hub: a row that reaches 1 / 256 of the vertices or
//     more): 2^10 vertices 36.0 / 30.2, 2^14 53.2 / 44.2, 2^15 45.3 / 38.4, 2^16
//     (46,700 with an edge) 47.2 / 43.5;
//   ER (none), vertices x degree: 24,000 x 12 49.6 / 43.3, 32,700 x 24 44.6 / 39.5,
//     49,000 x 12 50.9 / 46.6, 40,000 x 24 44.7 / 42.2, 24,000 x 40 43.6 / 43.2, 49,000 x
//     40 40.6 / 42.4: more rows are scanned to their ends, so fewer entries;
//   a star, whose one level claims every vertex: 32,700 leaves 19.9 / 19.7, 49,000
//     19.3 / 21.1.
// Dense levels that push take 2 to 3 times as long there (4 searches of RMAT-16:
// BFS_POLICY_PUSH 945 / 1961, all levels push-queue 332 / 815, alpha 0.01 901 /
// 1778; ER 49,000 x 40 pulled at every level 538 / 994), so other policies and
// thresholds far from the defaults only where the whole graph is a few entries a
// thread (RMAT-12, every form: 0.8 to 0.97 of the grid-wide time).  Nor on graphs
// without a hub where a lane leaves a row to its warp early (pull_serial 1, ER
// 49,000 x 8: 379 / 439).
// The hardware barrier takes no limit: a call with a limit below the default
// gets the grid-wide kernel, as does one that asks for a launch shape, for the
// aggregated claims (ER 49,000 x 40 208 / 283) or for no cluster.
constexpr int64_t SMALL_THREADS = 16 * 1024;
constexpr int64_t SMALL_GRAPH_N = 3 * SMALL_THREADS, SMALL_GRAPH_M = 1 << 21, SMALL_FLAT_M = 3 << 18;
constexpr int64_t SMALL_ANY_M = 8 * SMALL_THREADS;
constexpr int32_t SMALL_HUB = 256;

inline bool small_graph_pays(const SmallGraph& g, const bfs_options& o, const bfs_options& dflt) {
    if (o.mode != BFS_MODE_PERSISTENT || o.frontier_sort != BFS_SORT_NONE || o.push_filter != BFS_PUSH_FUSED) return false;
    if (o.small_levels != BFS_SMALL_AUTO || o.block_threads != dflt.block_threads || o.blocks_per_sm != 0) return false;
    if (o.barrier_timeout_ns < dflt.barrier_timeout_ns) return false;
    if (g.deg_max <= 16) return false;  // the small levels' kernels
    if (g.n1 > SMALL_GRAPH_N || g.m > SMALL_GRAPH_M || g.n > 4 * SMALL_GRAPH_N) return false;
    if (g.n1 <= SMALL_THREADS && g.m <= SMALL_ANY_M) return true;
    if (o.policy != BFS_POLICY_HEURISTIC && o.policy != BFS_POLICY_MLP) return false;
    if (o.alpha < 4.0f || o.alpha > 24.0f || o.beta < 16.0f || o.gamma > 64.0f || o.claim_aggregate) return false;
    if (g.deg_max > 2 * SMALL_THREADS && g.m < 4 * g.n1) return false;  // a star
    return (int64_t)g.deg_max * SMALL_HUB >= g.n1 || (g.m <= SMALL_FLAT_M && o.pull_serial >= 8);
}

}  // namespace bfsgb

#endif
