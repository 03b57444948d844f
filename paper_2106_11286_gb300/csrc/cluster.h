// Sweeps of a small lattice, a group of them in one launch (cluster.cu).
#pragma once

#include "hs_impl.h"

namespace hs {

// The largest lattices that run in one cluster, by the work items of a pass:
// beyond them its 16 SMs take longer than a barrier over the whole device
// costs.  us per sweep in a cluster with the spins in its shared memory (slabs),
// with them in L2, and on the grid:
//   V = 4, FP32: 768 items 2.8, 4.3, 4.8; 4096 4.2, 5.1, 5.0; 6144 5.6, 6.0, 5.0
//   V = 2, FP32: 3584 items 3.2, 3.9, 4.3; 9216 7.9, 9.6, 4.4
//   V = 1, FP32: 1792 items 3.0, 3.8, 4.5; 2816 3.9, 3.9, 4.3; 3840 4.9, 4.4, 4.5
//   FP64: 2048 items (16^3) 5.2, 6.0, 7; 4000 9.6, 7.9, 7.2
constexpr int64_t kSlabItems = 4800;     // FP32, FP16
constexpr int64_t kSlabItems1 = 3300;    // of one site each
constexpr int64_t kClusterItems = 3600;
constexpr int64_t kClusterItems64 = 2500;  // FP64, either way
// The largest that run as one cooperative launch: beyond them the launches
// are a small part of a pass (times in cluster.cu).
constexpr int64_t kGridSites = 3000000;    // FP32, FP16
constexpr int64_t kGridSites64 = 1000000;  // FP64

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
// room: how many such cooperative launches the device must hold at once (group_room).
GroupPlan group_plan(int precision, const Layout &L, int zaxis, int n_blocks, int n_sm, int room);

// n_sweeps sweeps from a.sweep on, sweep s to ring slot s; a.n_blocks = p.ctas,
// arrivals: those already counted in a.acc->passed.
cudaError_t launch_group(int precision, const Layout &L, const GroupPlan &p, const PassArgs &a, int n_sweeps,
                         unsigned long long arrivals, cudaStream_t s);

}  // namespace hs
