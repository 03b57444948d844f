// Sweeps of a small periodic sc lattice inside one thread-block cluster.
//
// A colour pass of a small lattice is a few microseconds of launch, drain and
// load latency around some hundred nanoseconds of work: as a chain of
// launches (kernels.cu) a 16^3 FP64 sweep took 16.6 us.  One cluster of up to
// 16 CTAs, resident for a whole group of sweeps, separates its passes by the
// hardware's cluster barrier instead.  The spins stay in global memory (in L2
// at these sizes): stores are released and acquired by the barrier, and loads
// go to L2 (ld.global.cg), since another SM wrote what they read.  The CTA's
// sums of a pass are reduced between arriving at the barrier and waiting for
// it, and go to the same ring of per-sweep slots as the launch chain's, so the
// ring fold that follows is the same.
#include <cuda_runtime.h>

#include "cluster.h"
#include "device.cuh"

namespace hs {
namespace {

constexpr int kClusterThreads = 512;  // 128 registers a thread

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Work item t of a pass belongs to thread t mod (threads of the cluster).  An
// FP32 / FP16 item's sums are added across its warp before they are widened,
// as the launch chain does for lattices of this size (one item per thread
// there), so the moments come out the same.
template <int P, int V, bool MEAS, int AX>
__global__ void __launch_bounds__(kClusterThreads, 1) sc_cluster_kernel(const PassArgs args, void *planes, int n_sweeps,
                                                                        int alternate) {
    pdl_enter();
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using VT = Vec<S, V>;
    __shared__ double s_w[kClusterThreads / 32][kPartials];
    PassArgs a = args;
    const uint32_t n_items = (uint32_t)a.Lz * a.Ly * (a.Lh / V);
    const size_t plane = (size_t)a.Lz * a.Ly * a.Lh;
    const uint32_t stride = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    for (int s = 0; s < n_sweeps; ++s) {
        a.sweep = args.sweep + (uint32_t)s;
        for (int c = 0; c < 2; ++c) {
            a.colour = c;
            a.rev = (alternate && c == 1) ? n_items - 1u : 0u;
            S *own_w[3];
            const S *own[3], *oth[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                own_w[q] = static_cast<S *>(planes) + (size_t)(3 * c + q) * plane;
                own[q] = own_w[q];
                oth[q] = static_cast<const S *>(planes) + (size_t)(3 * (1 - c) + q) * plane;
            }
            const S *const(&own_c)[3] = reinterpret_cast<const S *const(&)[3]>(own);
            const S *const(&oth_c)[3] = reinterpret_cast<const S *const(&)[3]>(oth);
            double sum[4] = {0.0, 0.0, 0.0, 0.0};
            unsigned n = 0;
            SiteAcc<P> acc;
            // whole warps walk the items together
            for (uint32_t t0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < n_items; t0 += stride) {
                if constexpr (P != HS_FP64) acc = SiteAcc<P>();
                if (t0 + lane < n_items) {
                    StencilItem<P, V> it;
                    load_item<P, V, true>(a, t0 + lane, own_c, oth_c, it);
                    if (update_item<P, V, MEAS, false, AX, true>(it.s, it.o, it.nym, it.nyp, it.nzm, it.nzp, it.ed, it.p,
                                                                 it.site0, it.rank0, c, a, J, K, ex, ey, ez, beta, acc,
                                                                 oth_c, it.b0)) {
#pragma unroll
                        for (int q = 0; q < 3; ++q) *reinterpret_cast<VT *>(own_w[q] + it.b0) = it.s[q];
                    }
                }
                if constexpr (P != HS_FP64) {
                    n += acc.n;
                    if (MEAS) {
                        sum[0] += (double)warp_sum(acc.E(J, K));
                        sum[1] += (double)warp_sum(acc.X());
                        sum[2] += (double)warp_sum(acc.Y());
                        sum[3] += (double)warp_sum(acc.Z());
                    }
                }
            }
            cluster_arrive();
            if constexpr (P == HS_FP64) {
                n = acc.n;
                if (MEAS) {
                    sum[0] = warp_sum(acc.E(J, K));
                    sum[1] = warp_sum(acc.X());
                    sum[2] = warp_sum(acc.Y());
                    sum[3] = warp_sum(acc.Z());
                }
            }
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) s_w[warp][q] = sum[q];
                s_w[warp][4] = (double)n;
            }
            __syncthreads();
            if (threadIdx.x < kPartials) {
                double v = 0.0;
                for (int w = 0; w < (int)blockDim.x / 32; ++w) v += s_w[w][threadIdx.x];
                a.partials[(((size_t)s * 2 + c) * gridDim.x + blockIdx.x) * kPartials + threadIdx.x] = v;
            }
            cluster_wait();  // also: the slots of s_w are read before the next pass writes them
        }
    }
}

template <int P, int V>
const void *cluster_ptr(bool meas, bool ax) {
    if constexpr (P == HS_FP32)
        if (ax)
            return meas ? (const void *)sc_cluster_kernel<P, V, true, 1> : (const void *)sc_cluster_kernel<P, V, false, 1>;
    return meas ? (const void *)sc_cluster_kernel<P, V, true, 0> : (const void *)sc_cluster_kernel<P, V, false, 0>;
}

const void *cluster_kernel(int precision, int vec, bool meas, bool ax) {
    switch (precision) {
    case HS_FP64: return vec == 2 ? cluster_ptr<HS_FP64, 2>(meas, ax) : cluster_ptr<HS_FP64, 1>(meas, ax);
    case HS_FP32: return vec == 4 ? cluster_ptr<HS_FP32, 4>(meas, ax)
                                  : (vec == 2 ? cluster_ptr<HS_FP32, 2>(meas, ax) : cluster_ptr<HS_FP32, 1>(meas, ax));
    case HS_FP16: return vec == 4 ? cluster_ptr<HS_FP16, 4>(meas, ax)
                                  : (vec == 2 ? cluster_ptr<HS_FP16, 2>(meas, ax) : cluster_ptr<HS_FP16, 1>(meas, ax));
    default: return nullptr;
    }
}

void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int ctas, int threads, cudaStream_t s) {
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
}

}  // namespace

ClusterPlan cluster_plan(int precision, const Layout &L, int zaxis) {
    ClusterPlan p{0, 0, L.vec};
    if (!L.structured || L.slab || L.tensor || L.vec > 4) return p;
    if (L.n_sites > (precision == HS_FP64 ? kClusterSites64 : kClusterSites)) return p;
    if (precision == HS_FP64) p.vec = 1;  // one site a thread: the shortest chain
    const int warps = (int)((L.n_sites / 2 / p.vec + 31) / 32);
    // the largest cluster that the device schedules and the warps fill
    for (int c = 16; c >= 1; c /= 2) {
        if (c > warps && c > 1) continue;
        const int threads = 32 * ((warps + c - 1) / c);
        const int t = threads < kClusterThreads ? threads : kClusterThreads;
        bool fits = true;
        for (int meas = 0; meas < 2 && fits; ++meas) {
            const void *k = cluster_kernel(precision, p.vec, meas != 0, zaxis != 0);
            int n = 0;
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute attr[2];
            cluster_config(cfg, attr, c, t, nullptr);
            cfg.numAttrs = 1;
            fits = k && (c <= 8 || cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
                   cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n >= 1;
        }
        if (!fits) {
            cudaGetLastError();
            continue;
        }
        p.ctas = c;
        p.threads = t;
        return p;
    }
    return p;
}

cudaError_t launch_cluster(int precision, const Layout &L, const ClusterPlan &p, const PassArgs &a, int n_sweeps,
                           cudaStream_t s) {
    const void *k = cluster_kernel(precision, p.vec, a.accumulate != 0, a.zaxis != 0);
    if (!k || n_sweeps < 1) return cudaErrorInvalidValue;
    PassArgs args = a;
    args.div_nxv = FastDiv((uint32_t)(L.Lh / p.vec));
    void *planes = L.planes;
    int alternate = L.order == 2 ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    cluster_config(cfg, attr, p.ctas, p.threads, s);
    void *params[] = {&args, &planes, &n_sweeps, &alternate};
    return cudaLaunchKernelExC(&cfg, k, params);
}

}  // namespace hs
