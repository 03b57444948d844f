// Sweeps of a small lattice inside one thread-block cluster (cluster.cu).
#pragma once

#include "hs_impl.h"

namespace hs {

// The largest lattices that run in one cluster: beyond them the 16 SMs of a
// cluster take longer over a pass than the whole device takes to launch it.
constexpr int64_t kClusterSites = 65536;    // FP32, FP16
constexpr int64_t kClusterSites64 = 16384;  // FP64

// CTAs (0: the launch chain instead) of how many threads, and sites per work item.
struct ClusterPlan {
    int ctas, threads, vec;
};
ClusterPlan cluster_plan(int precision, const Layout &L, int zaxis);

// n_sweeps sweeps from a.sweep on, sweep s to ring slot s; a.n_blocks = p.ctas.
cudaError_t launch_cluster(int precision, const Layout &L, const ClusterPlan &p, const PassArgs &a, int n_sweeps,
                           cudaStream_t s);

}  // namespace hs
