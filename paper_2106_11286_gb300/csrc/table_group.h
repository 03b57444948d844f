// Sweeps of a small neighbour-table lattice, a group of them in one launch (table_group.cu).
#pragma once

#include "hs_impl.h"

namespace hs {

// The largest table lattices that sweep this way.
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
