// Device side of the launches that run a group of sweeps of one lattice
// (cluster.cu: single lattices; batch.cu: FP64 batches of small members).
#pragma once

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
    int cta, ctas;    // this CTA of the lattice's
};

// Reduce the first `used` passes held, the last of them pass index `last`
// (2 sweep + colour) of the group: FP32 / FP16, with a few units a pass, one
// lane per pass and quantity; FP64 one warp per pass, its four sums'
// independent chains side by side.
template <int P>
__device__ void reduce_held(const PassArgs &a, const PassSums &h, int used, int last) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *const out = a.partials + ((size_t)(last - used + 1) * h.ctas + h.cta) * kPartials;
    const size_t next = (size_t)h.ctas * kPartials;  // from one pass's sums to the next's
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
// about a second, after which it latches the error word and marks the count
// abandoned.  The mark ends the waits of the other CTAs, and the launches that
// the same call has queued behind this one, whose targets the count can no
// longer reach, leave as they start (abandoned) with their folds (kernels.cu).
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
                    if (v & kAbandoned) {
                        ok = 0;
                        break;
                    }
                    if (v >= target) break;
                    if (it > (1u << 30) || clock64() - t0 > kBarrierCycles) {
                        ok = 0;
                        atomicExch(error, 1);
                        atomicOr(count, kAbandoned);
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

// A wait of this hs_sweep call ran out: in an earlier launch, or in another CTA
// of this one before this CTA started.  The same answer for the whole CTA.
__device__ __forceinline__ bool abandoned(const unsigned long long *count) {
    return __syncthreads_or(threadIdx.x == 0 && (*(volatile const unsigned long long *)count & kAbandoned) != 0) != 0;
}

// n_sweeps sweeps of one lattice by its ctas CTAs (the whole grid, or one
// cluster), of which this is number cta.  Work item t of a pass belongs to
// thread t mod (their threads).
template <int P, int V, bool MEAS, int AX, bool TEN, bool GRID>
__device__ __forceinline__ void sweep_group(const PassArgs &args, void *planes, int n_sweeps, int alternate, int depth,
                                            unsigned long long arrivals, int cta, int ctas) {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using VT = Vec<S, V>;
    extern __shared__ __align__(16) unsigned char cluster_smem[];
    PassArgs a = args;
    PassSums held;
    held.warps = (int)blockDim.x / 32;
    held.units = P == HS_FP64 ? (int)blockDim.x : held.warps;
    held.depth = depth;
    held.cta = cta;
    held.ctas = ctas;
    held.v = reinterpret_cast<double *>(cluster_smem);
    held.n = reinterpret_cast<unsigned *>(held.v + (size_t)depth * 4 * held.units);
    PassBarrier<GRID> bar{&a.acc->passed, arrivals, &a.acc->error};
    const uint32_t nxv = a.Lh / V;
    const uint32_t n_items = (uint32_t)a.Lz * a.Ly * nxv;
    const size_t plane = (size_t)a.Lz * a.Ly * a.Lh;
    const uint32_t stride = (uint32_t)ctas * blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t t_first = (uint32_t)cta * blockDim.x + threadIdx.x;
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

// Store a vector into the same shared-memory place of CTA `rank` of the cluster.
template <typename VT>
__device__ __forceinline__ void store_remote(uint32_t local, uint32_t rank, const VT &v) {
    uint32_t addr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local), "r"(rank));
    if constexpr (sizeof(VT) == 16) {
        uint4 w;
        memcpy(&w, &v, 16);
        asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w.x), "r"(w.y), "r"(w.z),
                     "r"(w.w)
                     : "memory");
    } else if constexpr (sizeof(VT) == 8) {
        uint2 w;
        memcpy(&w, &v, 8);
        asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(w.x), "r"(w.y) : "memory");
    } else if constexpr (sizeof(VT) == 4) {
        uint32_t w;
        memcpy(&w, &v, 4);
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(w) : "memory");
    } else {
        unsigned short w;
        memcpy(&w, &v, 2);
        asm volatile("st.shared::cluster.b16 [%0], %1;" ::"r"(addr), "h"(w) : "memory");
    }
}

// Planes of the fullest slab when Lz planes are dealt to ctas CTAs: CTA k owns
// planes Lz k / ctas .. Lz (k + 1) / ctas - 1.
__host__ __device__ inline int slab_planes(int Lz, int ctas) { return (Lz + ctas - 1) / ctas; }

// n_sweeps sweeps of one lattice by a cluster whose CTAs keep a z-slab each in
// shared memory, with a halo plane below and above: a pass loads from the
// CTA's own memory (30 cycles, against the 800 of L2) and stores an accepted
// spin of a boundary plane into the neighbour's halo as well, which the
// barrier's release waits for without a way to L2 (sweep_group took 2.8 us a
// pass of 16^3 FP64, of which its loads and its release were 1.0).
// FP32 / FP16: every slab must start at a multiple of 32 items, so that the
// warps' items are the launch chain's (see PassSums).
// The sums of sweep_group, held and reduced alike.
template <int P, int V, bool MEAS, int AX>
__device__ __forceinline__ void sweep_slabs(const PassArgs &args, void *planes, int n_sweeps, int depth, int cta,
                                            int ctas) {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using VT = Vec<S, V>;
    extern __shared__ __align__(16) unsigned char cluster_smem[];
    PassArgs a = args;
    const int Lz = args.Lz;
    const int z0 = Lz * cta / ctas, nz = Lz * (cta + 1) / ctas - z0, most = slab_planes(Lz, ctas);
    const int below = cta == 0 ? ctas - 1 : cta - 1, above = cta == ctas - 1 ? 0 : cta + 1;
    const int nz_below = Lz * (below + 1) / ctas - Lz * below / ctas;
    const uint32_t row_plane = (uint32_t)a.Ly * a.Lh;           // elements of one z plane of one component
    const uint32_t comp = (uint32_t)(most + 2) * row_plane;     // of one component's slab with its halos
    const size_t plane = (size_t)Lz * row_plane;                // of one component in device memory
    S *const st = reinterpret_cast<S *>(cluster_smem);
    PassSums held;
    held.warps = (int)blockDim.x / 32;
    held.units = P == HS_FP64 ? (int)blockDim.x : held.warps;
    held.depth = depth;
    held.cta = cta;
    held.ctas = ctas;
    held.v = reinterpret_cast<double *>(cluster_smem + ((size_t)6 * comp * sizeof(S) + 15) / 16 * 16);
    held.n = reinterpret_cast<unsigned *>(held.v + (size_t)depth * 4 * held.units);
    S *const dev = static_cast<S *>(planes);
    // the slab and its halos, array plane z holding lattice plane z0 + z - 1
    for (uint32_t k = threadIdx.x; k < (uint32_t)(nz + 2) * row_plane; k += blockDim.x) {
        const int z = z0 + (int)(k / row_plane) - 1;
        const size_t from = (size_t)(z < 0 ? Lz - 1 : (z >= Lz ? 0 : z)) * row_plane + k % row_plane;
#pragma unroll
        for (int q = 0; q < 6; ++q) st[q * comp + k] = dev[q * plane + from];
    }
    a.Lz = most + 2;
    a.zpar = (z0 - 1) & 1;
    a.site_off = (uint32_t)((int64_t)(z0 - 1) * a.Ly * a.Lx);
    a.rank_off = (uint32_t)((int64_t)(z0 - 1) * row_plane);
    const uint32_t nxv = a.Lh / V;
    const uint32_t own_items = (uint32_t)nz * a.Ly * nxv;
    const int rounds = (int)(((uint32_t)most * a.Ly * nxv + blockDim.x - 1) / blockDim.x);  // the same for all CTAs
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t st_addr = (uint32_t)__cvta_generic_to_shared(st);
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    double sum[4] = {0.0, 0.0, 0.0, 0.0};
    unsigned n = 0;
    SiteAcc<P> acc;
    int used = 0;
    auto hold = [&](int pass) {
        if constexpr (P == HS_FP64) {
            n = acc.n;
            sum[0] = acc.E(J, K);
            sum[1] = acc.X();
            sum[2] = acc.Y();
            sum[3] = acc.Z();
            acc = SiteAcc<P>();
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
    cluster_arrive();  // every slab is loaded before a neighbour writes its halos
    cluster_wait();
    int pass = 0, round = 0;
    bool pending = false;
    while (true) {
        const int c = pass & 1;
        const uint32_t t = threadIdx.x + (uint32_t)round * blockDim.x;
        const bool mine = t < own_items;
        a.sweep = args.sweep + (uint32_t)(pass >> 1);
        a.colour = c;
        const uint32_t row = a.div_nxv.div(mine ? t : 0u);
        const uint32_t zl = a.div_ly.div(row) + 1u;
        const ItemOffsets f = item_offsets<V>(a, row - (zl - 1u) * a.Ly, zl, (mine ? t : 0u) - row * nxv);
        Trials<P, V> pre;
        if (mine) draw_trials<P, V>(a, c, f.site0, f.rank0, pre);
        if (pending) {
            cluster_arrive();
            hold(pass - 1);
            cluster_wait();
            pending = false;
        }
        if (mine) {
            const S *own[3], *oth[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                own[q] = st + (3 * c + q) * comp;
                oth[q] = st + (3 * (1 - c) + q) * comp;
            }
            const S *const(&own_c)[3] = reinterpret_cast<const S *const(&)[3]>(own);
            const S *const(&oth_c)[3] = reinterpret_cast<const S *const(&)[3]>(oth);
            StencilItem<P, V> it;
            load_item_from<P, V>(f, own_c, oth_c, it);
            typename ItemField<P, V>::T h;
            fields_of<P, V, MEAS, false>(it.o, it.nym, it.nyp, it.nzm, it.nzp, it.ed, it.p, c, h);
            if (update_item_h<P, V, MEAS, false, AX, false, true>(it.s, h, it.site0, it.rank0, c, a, J, K, ex, ey, ez,
                                                                  beta, acc, oth_c, it.b0, &pre)) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const uint32_t at = (uint32_t)(3 * c + q) * comp + it.b0;
                    *reinterpret_cast<VT *>(st + at) = it.s[q];
                    // array plane 1 is the halo above the slab below, plane nz the halo below the slab above
                    if (zl == 1u)
                        store_remote(st_addr + (at + (uint32_t)nz_below * row_plane) * (uint32_t)sizeof(S), below,
                                     it.s[q]);
                    if (zl == (uint32_t)nz)
                        store_remote(st_addr + (at - (uint32_t)nz * row_plane) * (uint32_t)sizeof(S), above, it.s[q]);
                }
            }
        }
        if constexpr (P != HS_FP64) {
            if (MEAS) {
                sum[0] += (double)warp_sum(acc.E(J, K));
                sum[1] += (double)warp_sum(acc.X());
                sum[2] += (double)warp_sum(acc.Y());
                sum[3] += (double)warp_sum(acc.Z());
            }
            n += acc.n;
            acc = SiteAcc<P>();
        }
        if (++round < rounds) continue;
        round = 0;
        if (pass == 2 * n_sweeps - 1) break;
        ++pass;
        pending = true;
    }
    hold(pass);
    cluster_arrive();  // no CTA ends while a neighbour may still write into its shared memory
    cluster_wait();
    for (uint32_t k = threadIdx.x; k < (uint32_t)nz * row_plane; k += blockDim.x)
#pragma unroll
        for (int q = 0; q < 6; ++q) dev[q * plane + (size_t)z0 * row_plane + k] = st[q * comp + row_plane + k];
}

// Passes whose sums a CTA holds (16, or what fits in 96 KB), and the bytes of one pass.
inline size_t pass_bytes(int precision, int threads) {
    const int units = precision == HS_FP64 ? threads : threads / 32;
    return 4 * units * sizeof(double) + threads / 32 * sizeof(unsigned);
}
constexpr size_t kHeldBytes = 96 * 1024;
// shared memory of a CTA that keeps its slab there (sweep_slabs), before its held sums
inline size_t slab_bytes(size_t elem, int Lz, int Ly, int Lh, int ctas) {
    return ((size_t)6 * (slab_planes(Lz, ctas) + 2) * Ly * Lh * elem + 15) / 16 * 16;
}
constexpr size_t kSlabBytes = 200 * 1024;  // slab and held sums together, of the 227 KB a CTA may have
inline int held_passes(int precision, int threads) {
    const int fit = (int)(kHeldBytes / pass_bytes(precision, threads));
    return fit < 16 ? fit : 16;
}

}  // namespace
}  // namespace hs
