// Sweeps of a small periodic sc lattice inside one thread-block cluster.
//
// A colour pass of a small lattice is a few microseconds of launch, drain and
// load latency around some hundred nanoseconds of work: as a chain of
// launches (kernels.cu) a 16^3 FP64 sweep took 15.6 us.  One cluster of up to
// 16 CTAs, resident for a whole group of sweeps, separates its passes by the
// hardware's cluster barrier instead.  The spins stay in global memory (in L2
// at these sizes), stored before the barrier's release and loaded after its
// acquire by plain accesses, which so see them (loads past L1, ld.global.cg,
// measured slower: 128^3 FP32 17.4 against 15.9 us per sweep).
//
// What bounds a pass is its serial chain: the barrier with its stores' way to
// L2 (about 1000 cycles), the loads (800), the trial (1000 in FP64), the
// decision, and the FP64 sums across the CTA (2600 as four shuffle trees).
// So the next pass's trials, which need no spin, are drawn while the stores
// travel, and the sums of several passes are kept in shared memory and reduced
// together, independent chains side by side.  us per sweep, this launch and
// the launch chain: 16^3 FP64 6.0 and 15.6, 16^3 FP32 4.2 and 6.7, 24^3 FP32 4.3
// and 6.8.
//
// Lattices of up to some million sites (cluster.h) run the same loop on the whole device as
// one cooperative launch, with a barrier over the grid: it takes about as long
// as the cluster's plus one atomic and one poll, still less than ending a
// launch and starting the next: 64^3 FP32 5.4 and 8.6 us per sweep, 96^3 10.0
// and 11.9, 128^3 15.9 and 18.3; FP64 32^3 7.2 and 16.7, 64^3 20.5 and 26.2, 96^3
// 46.2 and 48.4.
#include <cuda_runtime.h>

#include <algorithm>

#include "cluster.h"
#include "fit_cache.h"
#include "group.cuh"

namespace hs {
namespace {

template <int P, int V, bool MEAS, int AX, bool TEN>
__global__ void __launch_bounds__(kClusterThreads, 1) sc_cluster_kernel(const PassArgs args, void *planes, int n_sweeps,
                                                                        int alternate, int depth) {
    pdl_enter();
    sweep_group<P, V, MEAS, AX, TEN, false>(args, planes, n_sweeps, alternate, depth, 0ull, (int)blockIdx.x,
                                              (int)gridDim.x);
}

// (Always ascending: a warp's items and their sum are the same in either direction.)
template <int P, int V, bool MEAS, int AX>
__global__ void __launch_bounds__(kClusterThreads, 1) sc_slab_kernel(const PassArgs args, void *planes, int n_sweeps,
                                                                     int depth) {
    pdl_enter();
    sweep_slabs<P, V, MEAS, AX>(args, planes, n_sweeps, depth, (int)blockIdx.x, (int)gridDim.x);
}

template <int P, int V, bool MEAS, int AX, bool TEN>
__global__ void __launch_bounds__(kBlock, 2) sc_grid_kernel(const PassArgs args, void *planes, int n_sweeps,
                                                            int alternate, int depth, unsigned long long arrivals) {
    if (abandoned(&args.acc->passed)) return;
    sweep_group<P, V, MEAS, AX, TEN, true>(args, planes, n_sweeps, alternate, depth, arrivals, (int)blockIdx.x,
                                             (int)gridDim.x);
}

// The variants of one precision and width: the tensor term, or FP32's S.e = S_z.
template <int P, int V, bool MEAS>
const void *grid_ptr(bool ten, bool ax) {
    if (ten) return (const void *)sc_grid_kernel<P, V, MEAS, 0, true>;
    if constexpr (P == HS_FP32)
        if (ax) return (const void *)sc_grid_kernel<P, V, MEAS, 1, false>;
    return (const void *)sc_grid_kernel<P, V, MEAS, 0, false>;
}

template <int P, int V, bool MEAS>
const void *cluster_ptr(GroupKind kind, bool ten, bool ax) {
    const bool slabs = kind == kGroupSlabs;
    if (ten) return slabs ? nullptr : (const void *)sc_cluster_kernel<P, V, MEAS, 0, true>;
    if constexpr (P == HS_FP32)
        if (ax)
            return slabs ? (const void *)sc_slab_kernel<P, V, MEAS, 1> : (const void *)sc_cluster_kernel<P, V, MEAS, 1, false>;
    return slabs ? (const void *)sc_slab_kernel<P, V, MEAS, 0> : (const void *)sc_cluster_kernel<P, V, MEAS, 0, false>;
}

template <int P, int V, bool MEAS>
const void *group_ptr(GroupKind kind, bool ten, bool ax) {
    if (kind == kGroupGrid) return grid_ptr<P, V, MEAS>(ten, ax);
    if constexpr (P != HS_FP64 || V == 1)  // FP64 clusters take one site a thread
        return cluster_ptr<P, V, MEAS>(kind, ten, ax);
    return nullptr;
}

template <int P>
const void *group_vec(int vec, bool meas, GroupKind kind, bool ten, bool ax) {
    switch (vec) {
    case 1: return meas ? group_ptr<P, 1, true>(kind, ten, ax) : group_ptr<P, 1, false>(kind, ten, ax);
    case 2: return meas ? group_ptr<P, 2, true>(kind, ten, ax) : group_ptr<P, 2, false>(kind, ten, ax);
    case 4:
        if constexpr (P != HS_FP64) return meas ? group_ptr<P, 4, true>(kind, ten, ax) : group_ptr<P, 4, false>(kind, ten, ax);
        break;
    default: break;
    }
    return nullptr;
}

const void *group_kernel(int precision, const GroupPlan &p, bool meas, bool ten, bool ax) {
    switch (precision) {
    case HS_FP64: return group_vec<HS_FP64>(p.vec, meas, p.kind, ten, ax);
    case HS_FP32: return group_vec<HS_FP32>(p.vec, meas, p.kind, ten, ax);
    case HS_FP16: return group_vec<HS_FP16>(p.vec, meas, p.kind, ten, ax);
    default: return nullptr;
    }
}

void group_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int precision, const GroupPlan &p,
                  cudaStream_t s) {
    cfg.gridDim = dim3((unsigned)p.ctas);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = p.smem + p.depth * pass_bytes(precision, p.threads);
    cfg.stream = s;
    cfg.attrs = attr;
    if (p.kind == kGroupGrid) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.numAttrs = 1;
        return;
    }
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
}

// How many of p's clusters, or of its CTAs per SM, the device holds at once.
int ask_held(int precision, const GroupPlan &p, const void *k) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    group_config(cfg, attr, precision, p, nullptr);
    int n = 0;
    cudaError_t e;
    if (p.kind == kGroupGrid) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, p.threads, cfg.dynamicSmemBytes);
    } else {
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
    }
    if (e == cudaSuccess) return n;
    cudaGetLastError();
    return 0;
}

// Both variants (with and without the fused measurement) fit the device as p asks.
bool plan_fits(int precision, const GroupPlan &p, bool ten, bool ax, int n_sm, int room) {
    for (int meas = 0; meas < 2; ++meas) {
        const void *k = group_kernel(precision, p, meas != 0, ten, ax);
        if (!k) return false;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(p.kind == kGroupSlabs ? kSlabBytes : kHeldBytes)) != cudaSuccess ||
            (p.kind != kGroupGrid && p.ctas > 8 &&
             cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
            cudaGetLastError();
            return false;
        }
        const int n = cached_fit(k, p.kind == kGroupGrid ? 0 : p.ctas, p.threads + (int)(p.smem / 1024) * 1024,
                                 [&] { return ask_held(precision, p, k); });
        if (p.kind == kGroupGrid ? n * n_sm < p.ctas * room : n < 1) return false;
    }
    return true;
}
}  // namespace

namespace {
// The cluster whose CTAs keep a slab each in shared memory, or ctas 0: at
// least 8 planes, and for FP32 / FP16 equal slabs of whole warps of items.
GroupPlan slab_plan(int precision, const Layout &L, bool ax, int n_sm) {
    const int vec = precision == HS_FP64 ? 1 : L.vec;  // FP64: one site a thread, the shortest chain
    for (int c = std::min(16, L.Lz); c >= 8; --c) {
        const int most = slab_planes(L.Lz, c);
        const int64_t items = (int64_t)most * L.Ly * (L.Lh / vec);
        if (precision != HS_FP64 && (L.Lz % c != 0 || items % 32 != 0)) continue;
        GroupPlan p{c, (int)std::min<int64_t>(kClusterThreads, (items + 31) / 32 * 32), vec, kGroupSlabs, 0, 0};
        p.smem = slab_bytes(storage_size(precision), L.Lz, L.Ly, L.Lh, c);
        if (p.smem + pass_bytes(precision, p.threads) > kSlabBytes) continue;
        p.depth = (int)std::min<size_t>(held_passes(precision, p.threads),
                                        (kSlabBytes - p.smem) / pass_bytes(precision, p.threads));
        if (plan_fits(precision, p, false, ax, n_sm, 1)) return p;
    }
    return GroupPlan{0, 0, L.vec, kGroupCluster, 0, 0};
}
}  // namespace

namespace {
// Sites up to which a lattice of this precision and width sweeps in groups (cluster.h has the times on both sides).
int64_t group_sites(int precision, int vec) {
    if (precision == HS_FP64) return kGridSites64;
    if (vec == 1) return 2 * kGridItems1;
    if (precision == HS_FP32) return kGridSites;
    return vec == 2 ? 4 * kGridItems2 : kGridSites16;
}
}  // namespace

GroupPlan group_plan(int precision, const Layout &L, int zaxis, int n_blocks, int n_sm, int room) {
    const GroupPlan none{0, 0, L.vec, kGroupCluster, 0, 0};
    const bool wide = precision == HS_FP64;
    if (!L.structured || L.slab || L.vec > 4 || L.n_sites > group_sites(precision, L.vec)) return none;
    const bool ten = L.tensor != 0, ax = zaxis != 0;
    const int64_t items = L.n_sites / 2 / (wide ? 1 : L.vec);
    if (!ten && items <= (wide ? kClusterItems64 : (L.vec == 1 ? kSlabItems1 : kSlabItems))) {
        const GroupPlan p = slab_plan(precision, L, ax, n_sm);
        if (p.ctas > 0) return p;
    }
    if (items <= (wide ? kClusterItems64 : kClusterItems)) {
        GroupPlan p = none;
        if (wide) p.vec = 1;
        const int warps = (int)((L.n_sites / 2 / p.vec + 31) / 32);
        // the largest cluster that the device schedules and the warps fill
        for (p.ctas = 16; p.ctas >= 1; p.ctas /= 2) {
            if (p.ctas > warps && p.ctas > 1) continue;
            p.threads = std::min(kClusterThreads, 32 * ((warps + p.ctas - 1) / p.ctas));
            p.depth = held_passes(precision, p.threads);
            if (plan_fits(precision, p, ten, ax, n_sm, 1)) return p;
        }
        return none;
    }
    GroupPlan p{n_blocks, kBlock, L.vec, kGroupGrid, 0, 0};  // FP32 / FP16: the launch chain's grid, so the same sums
    if (wide && L.n_sites / 2 <= (int64_t)n_sm * 2 * kBlock) {  // one site a thread while they last
        p.vec = 1;
        p.ctas = (int)((L.n_sites / 2 + kBlock - 1) / kBlock);
    }
    spread_ctas(L.n_sites / 2 / p.vec, n_sm, p.ctas, p.threads);
    p.depth = held_passes(precision, p.threads);
    return plan_fits(precision, p, ten, ax, n_sm, room) ? p : none;
}

cudaError_t launch_group(int precision, const Layout &L, const GroupPlan &p, const PassArgs &a, int n_sweeps,
                         unsigned long long arrivals, cudaStream_t s) {
    const void *k = group_kernel(precision, p, a.accumulate != 0, L.tensor != 0, a.zaxis != 0);
    if (!k || n_sweeps < 1) return cudaErrorInvalidValue;
    PassArgs args = a;
    args.div_nxv = FastDiv((uint32_t)(L.Lh / p.vec));
    void *planes = L.planes;
    int alternate = L.order == 2 ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    group_config(cfg, attr, precision, p, s);
    int depth = p.depth;
    void *slabs[] = {&args, &planes, &n_sweeps, &depth};
    void *params[] = {&args, &planes, &n_sweeps, &alternate, &depth, &arrivals};  // a cluster's kernel takes the first five
    return cudaLaunchKernelExC(&cfg, k, p.kind == kGroupSlabs ? slabs : params);
}

}  // namespace hs
