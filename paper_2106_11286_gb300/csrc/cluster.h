// Sweeps of a small lattice, a group of them in one launch (cluster.cu).
#pragma once

#include "hs_impl.h"

namespace hs {

// The largest lattices that run in one cluster, by the work items of a pass:
// beyond them its 16 SMs take longer than a barrier over the whole device
// costs.  us per sweep in a cluster with the spins in its shared memory (slabs),
// with them in L2, and on the grid:
//   V = 4, FP32: 3072 items 4.2, 4.5, 5.0; 4096 4.2, 5.1, 5.0; 4608 5.5, 5.3, 5.0; 5120 6.4, 5.5, 4.9
//   V = 4, FP16: 3072 items 4.2, 4.5, 4.8; 4096 4.2, 5.4, 5.0; 4608 5.6, 5.5, 4.7; 5120 6.9, 5.6, 4.7
//   V = 2, FP32 / FP16: 3200 items -, 3.9 / 4.1, 4.3 / 4.7; 4704 -, 4.6, 4.4 / 4.6
//   V = 1, FP32: 2304 items 3.7, 3.8, 4.5; 2816 4.0, 3.9, 4.4; 3840 4.9, 4.4, 4.5
//   V = 1, FP16: 2304 items 3.8, 4.0, 4.6; 2816 4.1, 4.1, 4.6; 3840 5.0, 4.6, 4.7
//   FP64: 2048 items (16^3) 5.2, 6.0, 7.8; 2304 5.8, -, 7.8; 4000 9.7, 7.9, 7.9
constexpr int64_t kSlabItems = 4300;     // FP32, FP16
constexpr int64_t kSlabItems1 = 3300;    // of one site each
constexpr int64_t kClusterItems = 3600;
constexpr int64_t kClusterItems64 = 2500;  // FP64, either way
// The largest that run as one cooperative launch, on the default stream: beyond
// them the launches are a small part of a pass and the narrower items of FP32
// and FP16 lose more by the grid's 128 registers.  us per sweep, group and chain:
//   FP32, V = 4: 2.37 million sites 17.2, 18.7; 2.99 20.6, 21.7; 4.10 27.5, 27.6
//         V = 2: 0.76 9.9, 11.9; 1.40 14.9, 16.3; 1.67 17.4, 18.0
//         V = 1: 132,300 items 7.7, 8.2; 176,400 9.6, 9.5; 255,840 11.5, 11.2; 396,900 15.7, 13.6
//   FP16, V = 4: 2.37 million sites 18.4, 19.0; 2.49 18.4, 19.1; 2.66 22.5, 20.4
//         V = 2: 190,440 items 10.5, 11.1; 245,000 13.5, 12.0; 417,136 19.0, 16.4
//         V = 1: 132,300 items 8.0, 8.4; 176,400 9.9, 9.7; 255,840 11.8, 11.5; 396,900 16.6, 14.1
//   FP64: 0.80 million sites of one an item 44.8, 45.9; 0.88 of two 46.3, 48.6; 1.00 55.2, 53.9; 1.12 57.3, 59.9
constexpr int64_t kGridSites = 3000000;    // FP32, V = 2 or 4
constexpr int64_t kGridSites16 = 2500000;  // FP16, V = 4
constexpr int64_t kGridItems2 = 230000;    // FP16, V = 2: work items
constexpr int64_t kGridItems1 = 150000;    // FP32, FP16, V = 1: work items
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
