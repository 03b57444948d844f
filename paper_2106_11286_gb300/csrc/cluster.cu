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
// and 6.8, 32^3 FP32 5.1 and 6.9.
//
// Lattices of up to kGridSites sites run the same loop on the whole device as
// one cooperative launch, with a barrier over the grid: it takes about as long
// as the cluster's plus one atomic and one poll, still less than ending a
// launch and starting the next: 64^3 FP32 5.6 and 8.6 us per sweep, 96^3 10.0
// and 11.9, 128^3 15.9 and 18.3, 160^3 27.4 and 27.6; FP64 32^3 8.9 and 16.7,
// 64^3 20.7 and 26.2, 96^3 46.2 and 48.4, 128^3 94.0 and 92.3.
#include <cuda_runtime.h>

#include <algorithm>

#include "cluster.h"
#include "device.cuh"

namespace hs {
namespace {

constexpr int kClusterThreads = 512;  // 128 registers a thread

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// What a pass leaves in shared memory until its sums are reduced: E, Sx, Sy, Sz
// by unit (FP64: a thread; FP32 / FP16: a warp, whose lanes have been added in
// FP32 item by item, as the launch chain does for lattices of this size with
// their one item per thread, so the moments come out the same), and the
// accepted moves by warp.
struct PassSums {
    double *v;        // [depth][4][units]
    unsigned *n;      // [depth][warps]
    int depth, units, warps;
};

// Reduce the first `used` passes held, the last of them pass index `last`
// (2 sweep + colour) of the group: FP32 / FP16, with a few units a pass, one
// lane per pass and quantity; FP64 one warp per pass, its four sums'
// independent chains side by side.
template <int P>
__device__ void reduce_held(const PassArgs &a, const PassSums &h, int used, int last) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *const out = a.partials + ((size_t)(last - used + 1) * gridDim.x + blockIdx.x) * kPartials;
    const size_t next = (size_t)gridDim.x * kPartials;  // from one pass's sums to the next's
    __syncthreads();
    if constexpr (P == HS_FP64) {
        for (int i = warp; i < used; i += h.warps) {
            double t[4] = {0.0, 0.0, 0.0, 0.0};
            for (int u = lane; u < h.units; u += 32)
#pragma unroll
                for (int q = 0; q < 4; ++q) t[q] += h.v[(i * 4 + q) * h.units + u];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < 4; ++q) t[q] += __shfl_xor_sync(0xffffffffu, t[q], o);
            unsigned n = lane < h.warps ? h.n[i * h.warps + lane] : 0u;
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) out[i * next + q] = t[q];
                out[i * next + 4] = (double)n;
            }
        }
    } else {
        for (int r = threadIdx.x; r < used * kPartials; r += (int)blockDim.x) {
            const int i = r / kPartials, q = r - i * kPartials;
            double t = 0.0;
            if (q < 4) {
                for (int u = 0; u < h.units; ++u) t += h.v[(i * 4 + q) * h.units + u];
            } else {
                unsigned n = 0;
                for (int u = 0; u < h.warps; ++u) n += h.n[i * h.warps + u];
                t = (double)n;
            }
            out[i * next + q] = t;
        }
    }
    __syncthreads();  // the slots are written again by warps that need not wait for this one at the pass's barrier
}

constexpr long long kBarrierCycles = 2000000000LL;  // about one second

// The barrier between two passes.  Cluster: the hardware's.  Grid: a count of
// arrivals in device memory that only grows (zeroed by hs_sweep); thread 0
// arrives for its CTA with a release, and polls with acquires for at most
// about a second, after which it latches the error word and every CTA leaves.
template <bool GRID>
struct PassBarrier {
    unsigned long long *count;
    unsigned long long target;
    int *error;
    __device__ __forceinline__ void arrive() {
        if constexpr (GRID) {
            __syncthreads();
            if (threadIdx.x == 0)
                asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(count) : "memory");
            target += gridDim.x;
        } else {
            cluster_arrive();
        }
    }
    __device__ __forceinline__ bool wait() {
        if constexpr (GRID) {
            __shared__ int s_ok;
            if (threadIdx.x == 0) {
                int ok = 1;
                unsigned long long v;
                const long long t0 = clock64();
                for (uint32_t it = 0;; ++it) {
                    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(count) : "memory");
                    if (v >= target) break;
                    if (it > (1u << 30) || clock64() - t0 > kBarrierCycles) {
                        ok = 0;
                        atomicExch(error, 1);
                        break;
                    }
                }
                s_ok = ok;
            }
            __syncthreads();
            return s_ok != 0;
        } else {
            cluster_wait();
            return true;
        }
    }
};

// Work item t of a pass belongs to thread t mod (threads of the grid, which in
// a cluster launch is the cluster).
template <int P, int V, bool MEAS, int AX, bool TEN, bool GRID>
__device__ __forceinline__ void sweep_group(const PassArgs &args, void *planes, int n_sweeps, int alternate, int depth,
                                            unsigned long long arrivals) {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using VT = Vec<S, V>;
    extern __shared__ __align__(16) unsigned char cluster_smem[];
    PassArgs a = args;
    PassSums held;
    held.warps = (int)blockDim.x / 32;
    held.units = P == HS_FP64 ? (int)blockDim.x : held.warps;
    held.depth = depth;
    held.v = reinterpret_cast<double *>(cluster_smem);
    held.n = reinterpret_cast<unsigned *>(held.v + (size_t)depth * 4 * held.units);
    PassBarrier<GRID> bar{&a.acc->passed, arrivals, &a.acc->error};
    const uint32_t nxv = a.Lh / V;
    const uint32_t n_items = (uint32_t)a.Lz * a.Ly * nxv;
    const size_t plane = (size_t)a.Lz * a.Ly * a.Lh;
    const uint32_t stride = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t t_first = blockIdx.x * blockDim.x + threadIdx.x;
    const int rounds = (int)((n_items + stride - 1) / stride);  // items of a thread, the same for all
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    double sum[4] = {0.0, 0.0, 0.0, 0.0};
    unsigned n = 0;
    SiteAcc<P> acc;
    // a cluster's FP32 / FP16 sums are added across the warp item by item (PassSums)
    constexpr bool kByItem = P != HS_FP64 && !GRID;
    auto add_warp = [&]() {
        if (MEAS) {
            sum[0] += (double)warp_sum(acc.E(J, K));
            sum[1] += (double)warp_sum(acc.X());
            sum[2] += (double)warp_sum(acc.Y());
            sum[3] += (double)warp_sum(acc.Z());
        }
        n += acc.n;
        acc = SiteAcc<P>();
    };
    int used = 0;
    // hold the sums of pass `pass` (2 sweep + colour)
    auto hold = [&](int pass) {
        if constexpr (P == HS_FP64) {
            n = acc.n;
            sum[0] = acc.E(J, K);
            sum[1] = acc.X();
            sum[2] = acc.Y();
            sum[3] = acc.Z();
            acc = SiteAcc<P>();
        } else if constexpr (!kByItem) {
            add_warp();
        }
        n = __reduce_add_sync(0xffffffffu, n);
        if (P == HS_FP64 || lane == 0) {
            const int u = P == HS_FP64 ? (int)threadIdx.x : warp;
#pragma unroll
            for (int q = 0; q < 4; ++q) held.v[(used * 4 + q) * held.units + u] = sum[q];
        }
        if (lane == 0) held.n[used * held.warps + warp] = n;
        sum[0] = sum[1] = sum[2] = sum[3] = 0.0;
        n = 0;
        if (++used == depth || pass == 2 * n_sweeps - 1) {
            reduce_held<P>(a, held, used, pass);
            used = 0;
        }
    };
    int pass = 0, round = 0;
    bool pending = false;  // the previous pass's barrier is still to be passed
    while (true) {
        // an item's place and trials, which need no spin, ahead of the barrier
        const int c = pass & 1;
        const uint32_t t = t_first + (uint32_t)round * stride;
        const bool mine = t < n_items;
        a.sweep = args.sweep + (uint32_t)(pass >> 1);
        a.colour = c;
        const uint32_t item = mine ? (alternate && c == 1 ? n_items - 1u - t : t) : 0u;
        const uint32_t row = a.div_nxv.div(item);
        const uint32_t z = a.div_ly.div(row);
        const ItemOffsets f = item_offsets<V>(a, row - z * a.Ly, z, item - row * nxv);
        Trials<P, V> pre;
        if (mine) draw_trials<P, V>(a, c, f.site0, f.rank0, pre);
        if (pending) {
            if constexpr (!GRID) {  // its stores are on their way while the trials are drawn: the release finds them done
                bar.arrive();
                hold(pass - 1);
            }
            if (!bar.wait()) return;
            pending = false;
        }
        if (mine) {
            S *const base = static_cast<S *>(planes);
            S *own_w[3];
            const S *own[3], *oth[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                own[q] = own_w[q] = base + (size_t)(3 * c + q) * plane;
                oth[q] = base + (size_t)(3 * (1 - c) + q) * plane;
            }
            const S *const(&own_c)[3] = reinterpret_cast<const S *const(&)[3]>(own);
            const S *const(&oth_c)[3] = reinterpret_cast<const S *const(&)[3]>(oth);
            StencilItem<P, V> it;
            load_item_from<P, V>(f, own_c, oth_c, it);
            typename ItemField<P, V>::T h;
            fields_of<P, V, MEAS, TEN>(it.o, it.nym, it.nyp, it.nzm, it.nzp, it.ed, it.p, c, h);
            if (update_item_h<P, V, MEAS, TEN, AX, false, true>(it.s, h, it.site0, it.rank0, c, a, J, K, ex, ey, ez, beta,
                                                               acc, oth_c, it.b0, &pre)) {
#pragma unroll
                for (int q = 0; q < 3; ++q) *reinterpret_cast<VT *>(own_w[q] + it.b0) = it.s[q];
            }
        }
        if constexpr (kByItem) add_warp();
        if (++round < rounds) continue;
        round = 0;
        const bool end = pass == 2 * n_sweeps - 1;
        if constexpr (GRID) {
            if (!end) bar.arrive();
            hold(pass);
        }
        if (end) break;
        ++pass;
        pending = true;
    }
    if constexpr (!GRID) hold(pass);
}

template <int P, int V, bool MEAS, int AX, bool TEN>
__global__ void __launch_bounds__(kClusterThreads, 1) sc_cluster_kernel(const PassArgs args, void *planes, int n_sweeps,
                                                                        int alternate, int depth) {
    pdl_enter();
    sweep_group<P, V, MEAS, AX, TEN, false>(args, planes, n_sweeps, alternate, depth, 0ull);
}

template <int P, int V, bool MEAS, int AX, bool TEN>
__global__ void __launch_bounds__(kBlock, 2) sc_grid_kernel(const PassArgs args, void *planes, int n_sweeps,
                                                            int alternate, int depth, unsigned long long arrivals) {
    sweep_group<P, V, MEAS, AX, TEN, true>(args, planes, n_sweeps, alternate, depth, arrivals);
}

// The variants of one precision and width: the tensor term, or FP32's S.e = S_z.
template <int P, int V, bool MEAS>
const void *group_ptr(bool grid, bool ten, bool ax) {
    if (ten)
        return grid ? (const void *)sc_grid_kernel<P, V, MEAS, 0, true> : (const void *)sc_cluster_kernel<P, V, MEAS, 0, true>;
    if constexpr (P == HS_FP32)
        if (ax)
            return grid ? (const void *)sc_grid_kernel<P, V, MEAS, 1, false>
                        : (const void *)sc_cluster_kernel<P, V, MEAS, 1, false>;
    return grid ? (const void *)sc_grid_kernel<P, V, MEAS, 0, false> : (const void *)sc_cluster_kernel<P, V, MEAS, 0, false>;
}

template <int P>
const void *group_vec(int vec, bool meas, bool grid, bool ten, bool ax) {
    switch (vec) {
    case 1: return meas ? group_ptr<P, 1, true>(grid, ten, ax) : group_ptr<P, 1, false>(grid, ten, ax);
    case 2: return meas ? group_ptr<P, 2, true>(grid, ten, ax) : group_ptr<P, 2, false>(grid, ten, ax);
    case 4:
        if constexpr (P != HS_FP64) return meas ? group_ptr<P, 4, true>(grid, ten, ax) : group_ptr<P, 4, false>(grid, ten, ax);
        break;
    default: break;
    }
    return nullptr;
}

const void *group_kernel(int precision, const GroupPlan &p, bool meas, bool ten, bool ax) {
    switch (precision) {
    case HS_FP64: return group_vec<HS_FP64>(p.vec, meas, p.grid, ten, ax);
    case HS_FP32: return group_vec<HS_FP32>(p.vec, meas, p.grid, ten, ax);
    case HS_FP16: return group_vec<HS_FP16>(p.vec, meas, p.grid, ten, ax);
    default: return nullptr;
    }
}

// Passes whose sums a CTA holds (16, or what fits in 96 KB), and the bytes they take.
size_t pass_bytes(int precision, int threads) {
    const int units = precision == HS_FP64 ? threads : threads / 32;
    return 4 * units * sizeof(double) + threads / 32 * sizeof(unsigned);
}
constexpr size_t kHeldBytes = 96 * 1024;
int held_passes(int precision, int threads) {
    const int fit = (int)(kHeldBytes / pass_bytes(precision, threads));
    return fit < 16 ? fit : 16;
}

void group_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int precision, const GroupPlan &p,
                  cudaStream_t s) {
    cfg.gridDim = dim3((unsigned)p.ctas);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = held_passes(precision, p.threads) * pass_bytes(precision, p.threads);
    cfg.stream = s;
    cfg.attrs = attr;
    if (p.grid) {
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

// Both variants (with and without the fused measurement) fit the device as p asks.
bool plan_fits(int precision, const GroupPlan &p, bool ten, bool ax, int n_sm) {
    for (int meas = 0; meas < 2; ++meas) {
        const void *k = group_kernel(precision, p, meas != 0, ten, ax);
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[2];
        group_config(cfg, attr, precision, p, nullptr);
        int n = 0;
        bool ok = k && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHeldBytes) == cudaSuccess;
        if (ok && p.grid) {
            ok = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, p.threads, cfg.dynamicSmemBytes) == cudaSuccess &&
                 n * n_sm >= p.ctas;
        } else if (ok) {
            cfg.numAttrs = 1;
            ok = (p.ctas <= 8 ||
                  cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
                 cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n >= 1;
        }
        if (!ok) {
            cudaGetLastError();
            return false;
        }
    }
    return true;
}

}  // namespace

GroupPlan group_plan(int precision, const Layout &L, int zaxis, int n_blocks, int n_sm) {
    const GroupPlan none{0, 0, L.vec, false};
    if (!L.structured || L.slab || L.vec > 4 || L.n_sites > (precision == HS_FP64 ? kGridSites64 : kGridSites)) return none;
    const bool ten = L.tensor != 0, ax = zaxis != 0;
    if (L.n_sites <= (precision == HS_FP64 ? kClusterSites64 : kClusterSites)) {
        GroupPlan p = none;
        if (precision == HS_FP64) p.vec = 1;  // one site a thread: the shortest chain
        const int warps = (int)((L.n_sites / 2 / p.vec + 31) / 32);
        // the largest cluster that the device schedules and the warps fill
        for (p.ctas = 16; p.ctas >= 1; p.ctas /= 2) {
            if (p.ctas > warps && p.ctas > 1) continue;
            p.threads = std::min(kClusterThreads, 32 * ((warps + p.ctas - 1) / p.ctas));
            if (plan_fits(precision, p, ten, ax, n_sm)) return p;
        }
        return none;
    }
    GroupPlan p{n_blocks, kBlock, L.vec, true};  // FP32 / FP16: the launch chain's grid, so the same sums
    if (precision == HS_FP64 && L.n_sites / 2 <= (int64_t)n_sm * 2 * kBlock) {  // one site a thread while they last
        p.vec = 1;
        p.ctas = (int)((L.n_sites / 2 + kBlock - 1) / kBlock);
    }
    return plan_fits(precision, p, ten, ax, n_sm) ? p : none;
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
    int depth = held_passes(precision, p.threads);
    void *params[] = {&args, &planes, &n_sweeps, &alternate, &depth, &arrivals};  // a cluster's kernel takes the first five
    return cudaLaunchKernelExC(&cfg, k, params);
}

}  // namespace hs
