// Sweeps of a small neighbour-table lattice, a group of them in one
// cooperative launch.
//
// As for the small sc lattices (cluster.cu) a colour pass is mostly launch,
// drain and the latency of dependent loads: the table row, then the
// neighbours' spins.  Here the CTAs stay for the whole group, passes separated
// by the bounded grid barrier; a site's row and its trial, which no pass
// changes or needs a spin for, are fetched and drawn ahead of the barrier's
// wait, and the sums of several passes are reduced together.  The threads take
// the sites of the launch chain's, so the sums are grouped alike.  us per sweep,
// chain and group: fcc FP64 of 73,656 sites 35.6 and 20.6, FP32 16.5 and 8.0;
// bcc FP32 of 128,000 9.1 and 4.8; a nanoparticle of 223,989 FP32 9.7 and 5.9.
#include <cuda_runtime.h>

#include <algorithm>

#include "group.cuh"
#include "table.cuh"
#include "fit_cache.h"
#include "table_group.h"

namespace hs {
namespace {

template <int P, bool MEAS, int W>
__global__ void __launch_bounds__(kBlock, P == HS_FP64 || W > 8 ? 2 : 3) table_group_kernel(const PassArgs args,
                                                                                   const TableClasses cls, int n_sweeps,
                                                                                   int depth,
                                                                                   unsigned long long arrivals) {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using S4 = Vec<S, 4>;
    extern __shared__ __align__(16) unsigned char table_smem[];
    if (abandoned(&args.acc->passed)) return;
    PassArgs a = args;
    PassSums held;
    held.warps = (int)blockDim.x / 32;
    held.units = P == HS_FP64 ? (int)blockDim.x : held.warps;
    held.depth = depth;
    held.cta = (int)blockIdx.x;
    held.ctas = (int)gridDim.x;
    held.v = reinterpret_cast<double *>(table_smem);
    held.n = reinterpret_cast<unsigned *>(held.v + (size_t)depth * 4 * held.units);
    PassBarrier<true> bar{&a.acc->passed, arrivals, &a.acc->error};
    S4 *spins = reinterpret_cast<S4 *>(a.spins4);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    const int passes = n_sweeps * a.n_colours;
    int used = 0;
    bool pending = false;
    TableAcc<P> acc;
    int c = 0;
    a.sweep = args.sweep;
    int64_t first = 0;  // of the thread's sites this pass
    for (int pass = 0; pass < passes;) {
        a.colour = c;
        a.colour_begin = cls.begin[c];
        const int64_t i = a.colour_begin + first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        const bool mine = i < cls.begin[c + 1];
        int32_t jj[W];
        TableTrial<P> t;
        if (mine) {
#pragma unroll
            for (int k = 0; k < W; ++k) jj[k] = __ldg(a.nbr + (int64_t)k * a.n_pad + i);
            draw_table_trial<P>(a, i, t);
        }
        if (pending && !bar.wait()) return;
        pending = false;
        if (mine) {
            TableField<P, MEAS, false> f;
            S4 s = spins[i];
#pragma unroll
            for (int k = 0; k < W; ++k) f.add(a, jj[k], spins[jj[k]]);
            if (table_update<P, MEAS, false>(a, i, spins, f, t, s, J, K, ex, ey, ez, beta, acc)) spins[i] = s;
        }
        first += stride;
        if (first < cls.begin[c + 1] - cls.begin[c]) continue;  // the same for every thread
        const bool end = pass == passes - 1;
        if (!end) bar.arrive();
        pending = !end;
        const unsigned n = __reduce_add_sync(0xffffffffu, acc.n);
        double sum[4] = {0.0, 0.0, 0.0, 0.0};
        if constexpr (P == HS_FP64) {
            sum[0] = acc.e, sum[1] = acc.x, sum[2] = acc.y, sum[3] = acc.z;
        } else if (MEAS) {
            sum[0] = warp_sum(acc.e), sum[1] = warp_sum(acc.x), sum[2] = warp_sum(acc.y), sum[3] = warp_sum(acc.z);
        }
        if (P == HS_FP64 || lane == 0) {
            const int u = P == HS_FP64 ? (int)threadIdx.x : warp;
#pragma unroll
            for (int q = 0; q < 4; ++q) held.v[(used * 4 + q) * held.units + u] = sum[q];
        }
        if (lane == 0) held.n[used * held.warps + warp] = n;
        if (++used == depth || end) {
            reduce_held<P>(a, held, used, pass);
            used = 0;
        }
        acc = TableAcc<P>();
        first = 0;
        ++pass;
        if (++c == a.n_colours) {
            c = 0;
            a.sweep += 1u;
        }
    }
}

template <int P, bool MEAS>
const void *table_group_width(int width) {
    switch (width) {
    case 6: return (const void *)table_group_kernel<P, MEAS, 6>;
    case 8: return (const void *)table_group_kernel<P, MEAS, 8>;
    case 12: return (const void *)table_group_kernel<P, MEAS, 12>;
    default: return nullptr;
    }
}

const void *table_group(int precision, int width, bool meas) {
    switch (precision) {
    case HS_FP64: return meas ? table_group_width<HS_FP64, true>(width) : table_group_width<HS_FP64, false>(width);
    case HS_FP32: return meas ? table_group_width<HS_FP32, true>(width) : table_group_width<HS_FP32, false>(width);
    case HS_FP16: return meas ? table_group_width<HS_FP16, true>(width) : table_group_width<HS_FP16, false>(width);
    default: return nullptr;
    }
}

size_t table_held_bytes(int precision, int threads) {
    return held_passes(precision, threads) * pass_bytes(precision, threads);
}

}  // namespace

TableGroupPlan table_group_plan(int precision, const Layout &L, int n_blocks, int n_sm, int room) {
    TableGroupPlan p{0, kBlock};
    if (L.structured || L.tensor || L.n_present < 1 || L.n_present > kTableGroupSites) return p;
    int64_t items = 0;
    for (int c = 0; c < L.n_colours; ++c) items = std::max<int64_t>(items, L.colour_begin[c + 1] - L.colour_begin[c]);
    int ctas = n_blocks;  // the launch chain's, so its sums
    spread_ctas(items, n_sm, ctas, p.threads);
    for (int meas = 0; meas < 2; ++meas) {
        const void *k = table_group(precision, L.width, meas != 0);
        auto ask = [&] {
            int n = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, p.threads, table_held_bytes(precision, p.threads)) !=
                cudaSuccess) {
                cudaGetLastError();
                return 0;
            }
            return n;
        };
        if (!k) return p;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHeldBytes) != cudaSuccess) {
            cudaGetLastError();
            return p;
        }
        if (cached_fit(k, 0, p.threads, ask) * n_sm < ctas * room) return p;
    }
    p.ctas = ctas;
    return p;
}

cudaError_t launch_table_group(int precision, const Layout &L, const PassArgs &a, const TableGroupPlan &p,
                               int n_sweeps, unsigned long long arrivals, cudaStream_t s) {
    const void *k = table_group(precision, L.width, a.accumulate != 0);
    if (!k || n_sweeps < 1) return cudaErrorInvalidValue;
    TableClasses cls;
    for (int c = 0; c <= L.n_colours; ++c) cls.begin[c] = L.colour_begin[c];
    PassArgs args = a;
    int depth = held_passes(precision, p.threads);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)p.ctas);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = table_held_bytes(precision, p.threads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *params[] = {&args, &cls, &n_sweeps, &depth, &arrivals};
    return cudaLaunchKernelExC(&cfg, k, params);
}

}  // namespace hs
