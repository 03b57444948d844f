// Sweeps of a small lattice, a group of them in one launch (cluster.cu).
#pragma once

#include "hs_impl.h"

namespace hs {

// The largest lattices that run in one cluster: beyond them its 16 SMs take
// longer over a pass than a barrier over the whole device costs (us per sweep
// FP32: 24^3 4.3 in the cluster, 32^3 5.1 there, 40^3 5.0 on the grid; FP64 16^3
// 6.0 and 20^3 7.9 in the cluster, 24^3 7.2 on the grid).
constexpr int64_t kClusterSites = 24000;   // FP32, FP16
constexpr int64_t kClusterSites64 = 5000;  // FP64
// The largest that run as one cooperative launch: beyond them the launches
// are a small part of a pass (times in cluster.cu).
constexpr int64_t kGridSites = 3000000;    // FP32, FP16
constexpr int64_t kGridSites64 = 1000000;  // FP64

// The largest that keep their spins in a cluster's shared memory.
constexpr int64_t kSlabSites = 50000;   // FP32, FP16 (16^3 2.8 against 4.2, 32^3 4.2 against 5.1, 36^3 4.4 against 5.0)
constexpr int64_t kSlabSites64 = 5000;  // FP64 (16^3 5.2 us per sweep against 6.0 with its spins in L2, 20^3 9.6 against 7.2 on the grid)

// CTAs (0: the launch chain instead) of how many threads, sites per work item,
// and how they run: one cluster with the spins in its shared memory or in L2,
// or a cooperative launch; bytes of the slab, passes whose sums a CTA holds.
enum GroupKind { kGroupCluster = 0, kGroupSlabs = 1, kGroupGrid = 2 };
struct GroupPlan {
    int ctas, threads, vec;
    GroupKind kind;
    size_t smem;
    int depth;
};
GroupPlan group_plan(int precision, const Layout &L, int zaxis, int n_blocks, int n_sm);

// n_sweeps sweeps from a.sweep on, sweep s to ring slot s; a.n_blocks = p.ctas,
// arrivals: those already counted in a.acc->passed.
cudaError_t launch_group(int precision, const Layout &L, const GroupPlan &p, const PassArgs &a, int n_sweeps,
                         unsigned long long arrivals, cudaStream_t s);

}  // namespace hs
