// Sweeps of a small neighbour-table lattice, a group of them in one launch (table_group.cu).
#pragma once

#include "hs_impl.h"

namespace hs {

// The largest table lattices that sweep this way, where the device holds their
// CTAs at once: in FP32 and FP16 those of classes up to 117,000 sites (6 and 8
// neighbours) or 78,000 (12), which take a thread each (FP32 bcc of 221,184
// sites 5.6 us per sweep, chain 9.1; fcc of 296,352 10.0 and 23.0; beyond, the
// chain's sums would be grouped otherwise).  FP64, group and chain: fcc of
// 318,028 sites 69.6, 69.5; bcc of 601,526 54.1, 59.3; fcc of 595,508 78.4, 88.4.
constexpr int64_t kTableGroupSites = 600000;

// Renumbered sites of colour class c: begin[c] .. begin[c + 1] - 1.
struct TableClasses {
    int64_t begin[65];
};

// CTAs of the launch and their threads (the launch chain's n_blocks of kBlock,
// or spread_ctas), ctas 0 where it does not apply: the tensor term, widths
// other than 6, 8 and 12, larger lattices, or fewer than room such grids
// resident at once (group_room).
struct TableGroupPlan {
    int ctas, threads;
};
TableGroupPlan table_group_plan(int precision, const Layout &L, int n_blocks, int n_sm, int room);
cudaError_t launch_table_group(int precision, const Layout &L, const PassArgs &a, const TableGroupPlan &p,
                               int n_sweeps, unsigned long long arrivals, cudaStream_t s);

}  // namespace hs
