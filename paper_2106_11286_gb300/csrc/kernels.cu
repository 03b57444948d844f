// Colour-pass Metropolis kernels for sm_103a (arXiv 2106.11286: Eq. 1, the
// Metropolis steps (i)-(iii), Eq. 2), plus initialisation, layout
// conversion and measurement.
//
// Every kernel here is HBM- or ALU-bound elementwise work over one colour
// class: no dense contraction exists, so no tensor-core path is used.  The
// stencil pass reads its own colour and the other colour with 128-bit
// coalesced loads (own values, plus the other colour's rows at y+-1, z+-1 and
// the same row for the x neighbours, all at the same xh); the neighbour rows
// are shared by adjacent rows of the grid through L1/L2.  Random numbers come
// from an in-register Philox4x32-10 keyed by (seed, replica, sweep, colour,
// site): nothing of the generator lives in memory.
//
// Reductions: per-thread partials -> warp shuffle -> CTA (FP64) -> one slot
// per CTA and pass, in a ring of slot sets, one per sweep of a group of up to
// 64.  Within hs_sweep the passes only write slots; after each full group
// (and after the loop) a ring fold sums every sweep's slots in a fixed order
// (bit-reproducible), one CTA per sweep, and the last of them applies the
// totals to the FP64 accumulator in sweep order, so no pass carries a serial reduction
// (a last-arriving CTA reducing inside the finishing pass cost 8 % at 256^3,
// a fold in the next sweep's first pass 5 %).  Single passes and standalone
// measurements keep the last-arriving-CTA form.
#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "device.cuh"
#include "table.cuh"

namespace hs {
namespace {

// Register stencil: every operand is loaded from global memory (L1/L2 serve
// the neighbour rows shared by adjacent work items).  Launch bounds of two
// resident CTAs per SM (128 registers) measured fastest on GB300.  Prefetch
// modes (PF):
//   0  none;
//   1  the loads of the thread's next work item are issued before the
//      current one is computed (two items in flight in registers, unrolled by
//      hand so no operand is copied);
//   2  split prefetch: as soon as the current item's local fields are summed
//      (its neighbour vectors are dead then), the next item's own row,
//      same-row and z-1 / z+1 rows -- the operands most often in DRAM -- are
//      loaded, so they travel during the current item's Metropolis
//      arithmetic; the y-1 / y+1 rows (the rows of neighbouring work items
//      of the same CTA, usually in L1 or L2) are loaded when an item is
//      taken up.
//   TEN adds the on-site anisotropy tensor term (built with PF = 0 only).
//   AX = 1: the FP32 variant chosen at launch when e = (0, 0, 1) exactly:
//   S.e = S_z, three packed instructions fewer per site pair, with no branch
//   in the item loop (a run-time branch there measured slower).
//   DIR = false: a variant with ascending passes only, whose item indices
//   never refer to PassArgs::rev (built for FP32 V = 4 and FP16 V = 8 with
//   PF = 0, the launches of lattices beyond 2^31 sites, where it measured
//   faster: 137 against 103-112 attempts/ns at 2048^3 FP32, while the
//   direction-capable code is faster at 256^3 to 1024^3).
template <int P, int V, bool MEAS, int PF, bool TEN = false, bool DIR = true, int AX = 0>
__global__ void __launch_bounds__(kBlock, 2) sc_pass_kernel(const PassArgs a) {
    pdl_enter();
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using VT = Vec<S, V>;
    const uint32_t n_items = (uint32_t)a.nz * a.Ly * (a.Lh / V);  // own planes only; < 2^31
    const int c = a.colour;
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    S *own_w[3] = {(S *)a.own[0], (S *)a.own[1], (S *)a.own[2]};
    const S *const own[3] = {(const S *)a.own[0], (const S *)a.own[1], (const S *)a.own[2]};
    const S *const oth[3] = {(const S *)a.oth[0], (const S *)a.oth[1], (const S *)a.oth[2]};
    SiteAcc<P> acc;
    const uint32_t stride = gridDim.x * blockDim.x;
    // slabs offset the ranks by whole planes, which hold a multiple of V sites: pairs stay pairs
    constexpr bool kEarly = P == HS_FP16 && V <= 4 && PF == 0 && DIR;
    auto compute = [&](StencilItem<P, V> &it) {
        bool any;
        if constexpr (P == HS_FP64)
            any = update_item<P, V, MEAS, TEN, AX>(it.s, it.o, it.nym, it.nyp, it.nzm, it.nzp, it.ed, it.p, it.site0,
                                                   it.rank0, c, a, J, K, ex, ey, ez, beta, acc, oth, it.b0);
        else
            any = update_item<P, V, MEAS, TEN, AX, false, kEarly>(it.s, it.o, it.nym, it.nyp, it.nzm, it.nzp, it.ed, it.p,
                                                                  it.site0, it.rank0, c, a, J, K, ex, ey, ez, beta, acc);
        if (any) {
#pragma unroll
            for (int q = 0; q < 3; ++q) *reinterpret_cast<VT *>(own_w[q] + it.b0) = it.s[q];
        }
    };
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (PF == 0) {
        for (; t < n_items; t += stride) {
            StencilItem<P, V> it;
            load_item<P, V, false, DIR>(a, t, own, oth, it);
            compute(it);
        }
    } else if (PF == 2) {
        if (t < n_items) {
            SplitItem<P, V> A;
            load_split_a<P, V, false, DIR>(a, t, own, oth, A);
            while (true) {
                VT nym[3], nyp[3];
                load_split_b<P, V>(A, oth, nym, nyp);
                typename ItemField<P, V>::T h;
                fields_of<P, V, MEAS, TEN>(A.o, nym, nyp, A.nzm, A.nzp, A.ed, A.f.p, c, h);
                VT sv[3] = {A.s[0], A.s[1], A.s[2]};
                const uint32_t b0 = A.f.b0, site0 = A.f.site0, rank0 = A.f.rank0;
                const uint32_t tn = t + stride;
                const bool more = tn < n_items;
                if (more) load_split_a<P, V, false, DIR>(a, tn, own, oth, A);  // the neighbour vectors are dead now
                if (update_item_h<P, V, MEAS, TEN, AX>(sv, h, site0, rank0, c, a, J, K, ex, ey, ez, beta, acc, oth,
                                                       b0)) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) *reinterpret_cast<VT *>(own_w[q] + b0) = sv[q];
                }
                if (!more) break;
                t = tn;
            }
        }
    } else if (t < n_items) {
        StencilItem<P, V> A, B;
        load_item<P, V, false, DIR>(a, t, own, oth, A);
        while (true) {
            if (t + stride < n_items) load_item<P, V, false, DIR>(a, t + stride, own, oth, B);
            compute(A);
            t += stride;
            if (t >= n_items) break;
            if (t + stride < n_items) load_item<P, V, false, DIR>(a, t + stride, own, oth, A);
            compute(B);
            t += stride;
            if (t >= n_items) break;
        }
    }
    write_partials<C, MEAS>(a, acc.E(J, K), acc.X(), acc.Y(), acc.Z(), acc.n);
}

// ----------------------------------------------------------------- pipelined stencil pass
// The register stencil with one landing slot per thread in shared memory: the
// operands of the thread's next work item travel global -> shared through
// cp.async while the current item, already in registers, is computed.  Each
// thread thus keeps one item of loads in flight during its arithmetic without
// holding a second item in registers (which would not fit in 128 registers).
// Only the issuing thread reads its slot, so cp.async.wait_all alone orders
// the copy before the reads (no CTA barrier).  The slot is refilled after the
// reads of the previous item: a thread's shared-memory reads and its later
// cp.async go through the load/store pipe in program order, and the copy's
// shared-memory write lands only when its global data returns.
//
// Slot layout (structure of arrays over the CTA's threads, so a warp's
// accesses to one operand are consecutive): 18 vectors (own s[3], other
// colour o[3], y-1, y+1, z-1, z+1 rows) at [j][thread], then 3 edge words at
// [q][thread].  An edge word is one element, or for 2-byte storage the
// aligned 4-byte pair holding it (cp.async copies 4, 8 or 16 bytes).
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

template <int B>
__device__ __forceinline__ void cp_async_ca(uint32_t dst, const void *src) {
    static_assert(B == 4 || B == 8 || B == 16, "cp.async copies 4, 8 or 16 bytes");
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(B) : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int P>
struct PipeEdge {
    using S = typename Tr<P>::S;
    using W = typename std::conditional<(sizeof(S) >= 4), S, uint32_t>::type;
};

template <int P, int V>
struct PipeSlot {
    using S = typename Tr<P>::S;
    using VT = Vec<S, V>;
    using W = typename PipeEdge<P>::W;
    static constexpr size_t kVecBytes = 18u * kBlock * sizeof(VT);
    static constexpr size_t kBytes = kVecBytes + 3u * kBlock * sizeof(W);
};

// Issue the copies of work item t's operands into this thread's slot.
template <int P, int V>
__device__ __forceinline__ ItemOffsets pipe_issue(const PassArgs &a, uint32_t t, const typename Tr<P>::S *const (&own)[3],
                                                  const typename Tr<P>::S *const (&oth)[3], uint32_t slot_v,
                                                  uint32_t slot_e) {
    using S = typename Tr<P>::S;
    using Sl = PipeSlot<P, V>;
    constexpr int VB = (int)sizeof(typename Sl::VT);
    constexpr int WB = (int)sizeof(typename Sl::W);
    const uint32_t nxv = a.Lh / V;
    const uint32_t row = a.div_nxv.div(t);
    const uint32_t xv = t - row * nxv;
    const uint32_t z = a.div_ly.div(row);
    const uint32_t y = row - z * a.Ly;
    const ItemOffsets f = item_offsets<V>(a, y, z, xv);
    // for 2-byte storage the edge word starts at the even element of the pair
    const uint32_t bed_w = (sizeof(S) >= 4) ? f.bed : (f.bed & ~1u);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        cp_async_ca<VB>(slot_v + (uint32_t)((0 + q) * kBlock * VB), own[q] + f.b0);
        cp_async_ca<VB>(slot_v + (uint32_t)((3 + q) * kBlock * VB), oth[q] + f.b0);
        cp_async_ca<VB>(slot_v + (uint32_t)((6 + q) * kBlock * VB), oth[q] + f.bym);
        cp_async_ca<VB>(slot_v + (uint32_t)((9 + q) * kBlock * VB), oth[q] + f.byp);
        cp_async_ca<VB>(slot_v + (uint32_t)((12 + q) * kBlock * VB), oth[q] + f.bzm);
        cp_async_ca<VB>(slot_v + (uint32_t)((15 + q) * kBlock * VB), oth[q] + f.bzp);
        cp_async_ca<WB>(slot_e + (uint32_t)(q * kBlock * WB), oth[q] + bed_w);
    }
    cp_async_commit();
    return f;
}

// Read this thread's slot (after cp.async.wait_all) into registers.
template <int P, int V>
__device__ __forceinline__ void pipe_read(const typename PipeSlot<P, V>::VT *sv, const typename PipeSlot<P, V>::W *se,
                                          const ItemOffsets &f, StencilItem<P, V> &it) {
    using S = typename Tr<P>::S;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        it.s[q] = sv[(0 + q) * kBlock];
        it.o[q] = sv[(3 + q) * kBlock];
        it.nym[q] = sv[(6 + q) * kBlock];
        it.nyp[q] = sv[(9 + q) * kBlock];
        it.nzm[q] = sv[(12 + q) * kBlock];
        it.nzp[q] = sv[(15 + q) * kBlock];
        if constexpr (sizeof(S) >= 4) {
            it.ed[q] = to_c(se[q * kBlock]);
        } else {
            const uint32_t w = se[q * kBlock];
            const unsigned short bits = (unsigned short)((f.bed & 1u) ? (w >> 16) : (w & 0xffffu));
            it.ed[q] = to_c(__ushort_as_half(bits));
        }
    }
    it.b0 = f.b0;
    it.p = f.p;
    it.site0 = f.site0;
    it.rank0 = f.rank0;
}

template <int P, int V, bool MEAS, int AX = 0>
__global__ void __launch_bounds__(kBlock, 2) sc_pipe_kernel(const PassArgs a) {
    pdl_enter();
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using Sl = PipeSlot<P, V>;
    using VT = typename Sl::VT;
    using W = typename Sl::W;
    extern __shared__ __align__(16) unsigned char pipe_smem[];
    const uint32_t n_items = (uint32_t)a.Lz * a.Ly * (a.Lh / V);
    const int c = a.colour;
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    S *own_w[3] = {(S *)a.own[0], (S *)a.own[1], (S *)a.own[2]};
    const S *const own[3] = {(const S *)a.own[0], (const S *)a.own[1], (const S *)a.own[2]};
    const S *const oth[3] = {(const S *)a.oth[0], (const S *)a.oth[1], (const S *)a.oth[2]};
    const VT *sv = reinterpret_cast<const VT *>(pipe_smem) + threadIdx.x;
    const W *se = reinterpret_cast<const W *>(pipe_smem + Sl::kVecBytes) + threadIdx.x;
    const uint32_t slot_v = smem_addr(sv);
    const uint32_t slot_e = smem_addr(se);
    SiteAcc<P> acc;
    const uint32_t stride = gridDim.x * blockDim.x;
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_items) {
        ItemOffsets f = pipe_issue<P, V>(a, t, own, oth, slot_v, slot_e);
        while (true) {
            cp_async_wait_all();
            StencilItem<P, V> it;
            pipe_read<P, V>(sv, se, f, it);
            const uint32_t tn = t + stride;
            const bool more = tn < n_items;
            if (more) f = pipe_issue<P, V>(a, tn, own, oth, slot_v, slot_e);
            if (update_item<P, V, MEAS, false, AX>(it.s, it.o, it.nym, it.nyp, it.nzm, it.nzp, it.ed, it.p, it.site0,
                                                   it.rank0, c, a, J, K, ex, ey, ez, beta, acc, oth, it.b0)) {
#pragma unroll
                for (int q = 0; q < 3; ++q) *reinterpret_cast<VT *>(own_w[q] + it.b0) = it.s[q];
            }
            if (!more) break;
            t = tn;
        }
    }
    write_partials<C, MEAS>(a, acc.E(J, K), acc.X(), acc.Y(), acc.Z(), acc.n);
}

// ----------------------------------------------------------------- z-marching stencil pass
// Register stencil in slab order: the plane-slabs (ty rows of one z plane)
// of every y slab, z fastest, are split into equal contiguous ranges, one per
// CTA, so a CTA walks along z.  On small lattices it spreads a pass over more
// SMs than the grid-stride stencil, whose CTAs each take 256 work items (the
// autotuner picks it for the 16^3 FP64 lattice, which is bound by the FP64
// pipe of the SMs it runs on).  The other colour's rows at z and z+1, loaded
// as the z+-1 neighbours of plane z, come back from L1 for plane z+1; only
// the own plane z+1 and the other colour's plane z+2 are new, and thread 0
// asks the bulk-copy engine to prefetch those into L2 one plane ahead.
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

template <int P, int V, bool MEAS>
__global__ void __launch_bounds__(kBlock, 2) sc_march_kernel(const PassArgs a) {
    pdl_enter();
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using VT = Vec<S, V>;
    const int c = a.colour;
    const uint32_t Lh = a.Lh, Ly = a.Ly, Lz = a.Lz;
    const uint32_t ty = (uint32_t)a.ty;
    const uint32_t nxv = Lh / V;
    const uint32_t items = ty * nxv;
    const uint32_t n_slabs = Ly / ty;
    const uint64_t total = (uint64_t)n_slabs * Lz;  // plane-slabs
    const uint32_t q0 = (uint32_t)(total * blockIdx.x / gridDim.x);
    const uint32_t q1 = (uint32_t)(total * (blockIdx.x + 1) / gridDim.x);
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    S *own_w[3] = {(S *)a.own[0], (S *)a.own[1], (S *)a.own[2]};
    const S *const own[3] = {(const S *)a.own[0], (const S *)a.own[1], (const S *)a.own[2]};
    const S *const oth[3] = {(const S *)a.oth[0], (const S *)a.oth[1], (const S *)a.oth[2]};
    const uint32_t slab_bytes = ty * Lh * (uint32_t)sizeof(S);
    const bool pf = (slab_bytes % 16u) == 0u;
    SiteAcc<P> acc;
    for (uint32_t q = q0; q < q1; ++q) {
        const uint32_t slab = q / Lz;  // once per plane-slab: plain division is fine
        const uint32_t z = q - slab * Lz;
        const uint32_t y0 = slab * ty;
        if (pf && threadIdx.x == 0 && q + 1 < q1) {
            const uint32_t z1 = (z + 1 == Lz) ? 0 : z + 1;
            const uint32_t z2 = (z1 + 1 == Lz) ? 0 : z1 + 1;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                prefetch_l2(own[k] + ((size_t)z1 * Ly + y0) * Lh, slab_bytes);
                prefetch_l2(oth[k] + ((size_t)z2 * Ly + y0) * Lh, slab_bytes);
            }
        }
        for (uint32_t it = threadIdx.x; it < items; it += kBlock) {
            const uint32_t yl = a.div_nxv.div(it);
            const uint32_t xv = it - yl * nxv;
            StencilItem<P, V> item;
            load_item_at<P, V>(a, y0 + yl, z, xv, own, oth, item);
            if (update_item<P, V, MEAS>(item.s, item.o, item.nym, item.nyp, item.nzm, item.nzp, item.ed, item.p,
                                        item.site0, item.rank0, c, a, J, K, ex, ey, ez, beta, acc, oth,
                                        item.b0)) {
#pragma unroll
                for (int k = 0; k < 3; ++k) *reinterpret_cast<VT *>(own_w[k] + item.b0) = item.s[k];
            }
        }
    }
    write_partials<C, MEAS>(a, acc.E(J, K), acc.X(), acc.Y(), acc.Z(), acc.n);
}

// ----------------------------------------------------------------- table pass
// One colour pass over renumbered sites [begin, end) with a neighbour table.
// Neighbours sum in stored order; padding points at a zero dummy spin.
// Each site waits on two dependent gathers (its table row, then the
// neighbours' spins), so resident warps set the throughput: FP32 / FP16 fit
// five CTAs per SM in 48 registers without spilling (measured 51.8 -> 56.0
// attempts/ns on the FP32 bcc nanoparticle, 45.2 -> 48.0 on bcc 128^3,
// 65.0 -> 68.3 FP16); FP64 would spill and keeps four.
// TEN adds the on-site anisotropy tensor term.  PFL2 asks L2 for the next
// site's table row and own spin (prefetch instructions, no registers held)
// while the current site waits for its gathers: the table is streamed from
// DRAM once, so its first-hop latency is otherwise exposed at every site
// (measured 56.0 -> 62.4 attempts/ns on the FP32 bcc nanoparticle; slower
// for FP16 and for the 12-neighbour fcc table, so the autotuner decides).
// W > 0: a table of exactly W neighbours, unrolled: the W row entries load
// together, then the W gathers, then the sums in stored order (the same
// sums), so each site waits two round trips instead of 2 W.  It needs 64
// registers (four CTAs per SM) at W = 8 in FP32: at 48 the compiler issues the
// gathers one after another again.  Measured on the FP32 bcc nanoparticle at
// W = 8: 65.9 -> 76.9 attempts/ns without PFL2 (74.9 with it); a version that
// also loaded the next site's row into registers measured lower.  The trial is
// drawn while the gathers travel: 144.7 -> 137.6 us per sweep there (76.3 ->
// 80.2 attempts/ns), 44.8 -> 42.6 on one of 3.1 M sites; for the loop (W = 0),
// whose gathers come one by one, after them (fcc FP32 37.9 against 44.0).
// FP64 runs one CTA per SM (139 registers), or two (TWO: 128, with a few
// spills) where a class has sites for them: fcc 864,000 sites 145.5 -> 117.3 us
// per sweep, bcc 1,024,000 118.2 -> 92.7; fcc of 73,656 35.6 -> 50.4.
template <int P, bool MEAS, bool TEN = false, bool PFL2 = false, int W = 0, bool TWO = false>
__global__ void __launch_bounds__(kBlock, P == HS_FP64 ? (TWO ? 2 : 1) : (P == HS_FP32 && W == 8 ? 4 : 5))
    table_pass_kernel(const PassArgs a) {
    pdl_enter();
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using S4 = Vec<S, 4>;
    S4 *spins = reinterpret_cast<S4 *>(a.spins4);
    C J, K, ex, ey, ez, beta;
    load_params(a, J, K, ex, ey, ez, beta);
    TableAcc<P> acc;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = a.begin + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.end; i += stride) {
        TableField<P, MEAS, TEN> f;
        TableTrial<P> t;
        if (PFL2 && i + stride < a.end) {
            for (int k = 0; k < a.width; ++k)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a.nbr + (int64_t)k * a.n_pad + i + stride));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(spins + i + stride));
        }
        if constexpr (W > 0) {
            int32_t jj[W];
            S4 nn[W];
#pragma unroll
            for (int k = 0; k < W; ++k) jj[k] = __ldg(a.nbr + (int64_t)k * a.n_pad + i);
#pragma unroll
            for (int k = 0; k < W; ++k) nn[k] = spins[jj[k]];
            draw_table_trial<P>(a, i, t);  // while the gathers are on their way
#pragma unroll
            for (int k = 0; k < W; ++k) f.add(a, jj[k], nn[k]);
        } else {
            for (int k = 0; k < a.width; ++k) {
                const int32_t j = __ldg(a.nbr + (int64_t)k * a.n_pad + i);
                f.add(a, j, spins[j]);
            }
        }
        S4 s = spins[i];
        if constexpr (W == 0) draw_table_trial<P>(a, i, t);
        if (table_update<P, MEAS, TEN>(a, i, spins, f, t, s, J, K, ex, ey, ez, beta, acc)) spins[i] = s;
    }
    write_partials<C, MEAS>(a, acc.e, acc.x, acc.y, acc.z, acc.n);
}

// ----------------------------------------------------------------- measure
// Standalone Eq. 1 / Eq. 2 of the current state to FP64 accuracy.
//
// FP32 / FP16 storage sums in unevaluated triples of floats: every addition
// keeps its rounding error (TwoSum, Knuth, The Art of Computer Programming
// vol. 2, 4.2.2), whose own sum keeps its errors in turn, and every product its
// remainder (one fma), so a thread's sums carry 72 bits where FP64's carry 53;
// a field of six neighbours is a pair, exact for components of 2^-20 and more
// (or 0), off by 2^-45 at most where one is smaller.  The FP64 pipe, which
// issues 2 instructions per cycle per SM against 128 for FP32, is left with
// the threads' totals.  A whole hs_measure, us: 256^3 FP32 140, FP16 155; 464^3
// 621 and 747.  With FP64 throughout, 45 FP64 instructions and 21 conversions a
// site, 2102 and 12224; in pairs of floats, too few bits, 116 and 498 (FP32).
// On the sc stencil every bond is counted once, at its colour-1 site, from the
// vector loads of the sweep's work items; colour 0 adds its own spins only.
template <typename T>
__device__ __forceinline__ T sub_exact(T a, T b) { return f_fma(splat<T>(-1.0f), b, a); }  // a - b, one rounding

// a += v; returns the rounding error
template <typename T>
__device__ __forceinline__ T two_sum(T &a, T v) {
    const T s = f_add(a, v);
    const T bb = sub_exact(s, a);
    const T e = f_add(sub_exact(a, sub_exact(s, bb)), sub_exact(v, bb));
    a = s;
    return e;
}

// A sum a + b + c: b holds what a's additions left over, c what b's did.
template <typename T>
struct Sum3 {
    T a = splat<T>(0.0f), b = splat<T>(0.0f), c = splat<T>(0.0f);
    __device__ __forceinline__ void add_rest(T v) { c = f_add(c, two_sum(b, v)); }
    __device__ __forceinline__ void add(T v) { add_rest(two_sum(a, v)); }
    __device__ __forceinline__ void add_square(T s) {
        const T p = f_mul(s, s);
        add(p);
        add_rest(f_fma(s, s, f_mul(splat<T>(-1.0f), p)));
    }
    // s (hh + hl)
    __device__ __forceinline__ void add_product(T s, T hh, T hl) {
        const T p = f_mul(s, hh), q = f_mul(s, hl);
        add(p);
        add_rest(f_fma(s, hh, f_mul(splat<T>(-1.0f), p)));
        add_rest(q);
        c = f_add(c, f_fma(s, hl, f_mul(splat<T>(-1.0f), q)));
    }
    __device__ __forceinline__ double value() const;
};
template <>
__device__ __forceinline__ double Sum3<float>::value() const { return (double)a + ((double)b + (double)c); }
template <>
__device__ __forceinline__ double Sum3<float2>::value() const {
    return ((double)a.x + (double)a.y) + (((double)b.x + (double)b.y) + ((double)c.x + (double)c.y));
}

// Sums of one thread: bonds, (S.e)^2 and the spin components.
template <typename T>
struct TripleSums {
    Sum3<T> b, k, m[3];
};

// FP32's products hold their remainders down to 2^-126: a thread's sum below this is taken again in FP64.
constexpr double kSmallSum = 0x1p-70;

__device__ __forceinline__ uint32_t bits_of(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t bits_of(float2 v) { return __float_as_uint(v.x) | __float_as_uint(v.y); }

template <typename T, typename S, int V>
__device__ __forceinline__ T lanes(const Vec<S, V> &v, int j) {
    if constexpr (std::is_same<T, float2>::value)
        return make_float2(to_c(v.v[2 * j]), to_c(v.v[2 * j + 1]));
    else
        return to_c(v.v[j]);
}

// quotient of a work-item or row index, beyond FastDiv's range by division
__device__ __forceinline__ uint32_t div_any(const FastDiv &d, uint32_t n) {
    return n < 0x80000000u ? d.div(n) : n / d.d;
}

// The on-site terms of one site in FP64 (an easy axis other than z, or the tensor): K (S.e)^2 + S^T A S.
__device__ __forceinline__ double onsite64(const PassArgs &a, double x, double y, double z) {
    const double se = x * a.e[0] + y * a.e[1] + z * a.e[2];
    const double k = a.K * se * se;
    return a.tensor ? k + quad64(x, y, z, a.A) : k;
}

// GEN: the on-site terms need FP64 (onsite64); else S.e = S_z or K = 0.
template <int P, int V, bool GEN>
__global__ void __launch_bounds__(kBlock) sc_measure_kernel(const PassArgs a, const void *planes, uint32_t n_items) {
    using S = typename Tr<P>::S;
    using VT = Vec<S, V>;
    const S *pl = (const S *)planes;
    const int64_t plane = (int64_t)a.Lz * a.Ly * a.Lh;
    const S *const c0[3] = {pl, pl + plane, pl + 2 * plane};
    const S *const c1[3] = {pl + 3 * plane, pl + 4 * plane, pl + 5 * plane};
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t t0 = blockIdx.x * blockDim.x + threadIdx.x;
    double accG = 0.0;
    // colour-1 work item t (a.colour = 1): its own spins and their neighbours'
    auto load = [&](uint32_t t, StencilItem<P, V> &it) {
        const uint32_t nxv = a.Lh / V;
        const uint32_t row = div_any(a.div_nxv, t);
        const uint32_t z = div_any(a.div_ly, row);
        load_item_at<P, V>(a, row - z * a.Ly, z, t - row * nxv, c1, c0, it);
    };
    if constexpr (P == HS_FP64) {
        double b = 0, k = 0, m[3] = {0, 0, 0};
        auto own = [&](const VT (&s)[3]) {
#pragma unroll
            for (int j = 0; j < V; ++j) {
#pragma unroll
                for (int q = 0; q < 3; ++q) m[q] += s[q].v[j];
                if (GEN)
                    accG += onsite64(a, s[0].v[j], s[1].v[j], s[2].v[j]);
                else
                    k = fma(s[2].v[j], s[2].v[j], k);
            }
        };
        for (uint64_t t = t0; t < n_items; t += stride) {
            VT s[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) s[q] = *reinterpret_cast<const VT *>(c0[q] + t * V);
            own(s);
        }
        for (uint64_t t = t0; t < n_items; t += stride) {
            StencilItem<P, V> it;
            load((uint32_t)t, it);
            Field64<V> h;
            item_fields64<V>(it.o, it.nym, it.nyp, it.nzm, it.nzp, it.ed, it.p, true, h);
#pragma unroll
            for (int j = 0; j < V; ++j)
#pragma unroll
                for (int q = 0; q < 3; ++q) b = fma(it.s[q].v[j], h.d[q][j], b);
            own(it.s);
        }
        write_partials<double, true>(a, -a.J * b - (GEN ? accG : (a.K == 0.0 ? 0.0 : a.K * k)), m[0], m[1], m[2], 0u);
    } else {
        using T = typename std::conditional<(V >= 2), float2, float>::type;
        constexpr int W = V >= 2 ? V / 2 : 1;  // lane groups of an item
        TripleSums<T> A;
        uint32_t zbits = 0;  // of every S_z: none but zeros leave k at 0 exactly
        auto own = [&](const VT (&s)[3]) {
#pragma unroll
            for (int j = 0; j < W; ++j) {
#pragma unroll
                for (int q = 0; q < 3; ++q) A.m[q].add(lanes<T>(s[q], j));
                if (!GEN) {
                    const T z = lanes<T>(s[2], j);
                    A.k.add_square(z);
                    zbits |= bits_of(z);
                }
            }
            if (GEN)
#pragma unroll
                for (int j = 0; j < V; ++j) accG += onsite64(a, to_c(s[0].v[j]), to_c(s[1].v[j]), to_c(s[2].v[j]));
        };
        for (uint64_t t = t0; t < n_items; t += stride) {
            VT s[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) s[q] = *reinterpret_cast<const VT *>(c0[q] + t * V);
            own(s);
        }
        for (uint64_t t = t0; t < n_items; t += stride) {
            StencilItem<P, V> it;
            load((uint32_t)t, it);
#pragma unroll
            for (int j = 0; j < W; ++j)
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    // the x neighbours: the same row's vector and its edge element on the side that p picks
                    T x;
                    if constexpr (V >= 2) {
                        const float prev = j == 0 ? it.ed[q] : to_c(it.o[q].v[j == 0 ? 0 : 2 * j - 1]);
                        const float next = j == W - 1 ? it.ed[q] : to_c(it.o[q].v[j == W - 1 ? 0 : 2 * j + 2]);
                        x = it.p ? make_float2(to_c(it.o[q].v[2 * j + 1]), next)
                                 : make_float2(prev, to_c(it.o[q].v[2 * j]));
                    } else {
                        x = it.ed[q];
                    }
                    T h = lanes<T>(it.o[q], j), hl;
                    hl = two_sum(h, x);
                    hl = f_add(hl, two_sum(h, lanes<T>(it.nym[q], j)));
                    hl = f_add(hl, two_sum(h, lanes<T>(it.nyp[q], j)));
                    hl = f_add(hl, two_sum(h, lanes<T>(it.nzm[q], j)));
                    hl = f_add(hl, two_sum(h, lanes<T>(it.nzp[q], j)));
                    A.b.add_product(lanes<T>(it.s[q], j), h, hl);
                }
            own(it.s);
        }
        double b = A.b.value(), k = A.k.value();
        double m[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) m[q] = A.m[q].value();
        // beyond FP32's range, or so small that it held no remainders (no unit vectors): the same sums in FP64
        const bool small = P == HS_FP32 && (fabs(b) < kSmallSum || (!GEN && k < kSmallSum && (zbits << 1) != 0u));
        if (small || !(isfinite(b) && isfinite(k) && isfinite(m[0]) && isfinite(m[1]) && isfinite(m[2]))) {
            b = k = m[0] = m[1] = m[2] = accG = 0.0;
            for (uint64_t t = t0; t < n_items; t += stride) {
                StencilItem<P, V> it;
                load((uint32_t)t, it);
                for (int j = 0; j < V; ++j)
                    for (int c = 0; c < 2; ++c) {
                        double s[3];
                        for (int q = 0; q < 3; ++q) {
                            s[q] = (double)to_c(c == 0 ? c0[q][t * V + j] : it.s[q].v[j]);
                            m[q] += s[q];
                            if (c == 0) continue;
                            const double x = it.p ? (double)(j == V - 1 ? it.ed[q] : to_c(it.o[q].v[j + 1]))
                                                  : (double)(j == 0 ? it.ed[q] : to_c(it.o[q].v[j - 1]));
                            b += s[q] * ((double)to_c(it.o[q].v[j]) + x + (double)to_c(it.nym[q].v[j]) +
                                         (double)to_c(it.nyp[q].v[j]) + (double)to_c(it.nzm[q].v[j]) +
                                         (double)to_c(it.nzp[q].v[j]));
                        }
                        if (GEN)
                            accG += onsite64(a, s[0], s[1], s[2]);
                        else
                            k += s[2] * s[2];
                    }
            }
        }
        write_partials<double, true>(a, -a.J * b - (GEN ? accG : (a.K == 0.0 ? 0.0 : a.K * k)), m[0], m[1], m[2], 0u);
    }
}

// Neighbour table: every site adds -J/2 S_i.h_i and its on-site terms, so each bond is counted once overall.
template <int P>
__global__ void __launch_bounds__(kBlock) table_measure_kernel(const PassArgs a, int64_t n_present) {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using S4 = Vec<S, 4>;
    const S4 *spins = reinterpret_cast<const S4 *>(a.spins4);
    const bool onsite = a.K != 0.0 || a.tensor;
    double b = 0, g = 0, m[3] = {0, 0, 0};
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    TripleSums<float> A;
    for (int64_t i = t0; i < n_present; i += stride) {
        C h[3] = {C(0), C(0), C(0)}, hl[3] = {C(0), C(0), C(0)};
        const S4 sv = spins[i];
        // four row entries, then their four gathers: two round trips per four neighbours (20 sweeps of a 3.1 M-site
        // nanoparticle with this measurement 1136 -> 1115 us)
        for (int k0 = 0; k0 < a.width; k0 += 4) {
            S4 n[4];
            int32_t j[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                j[k] = k0 + k < a.width ? __ldg(a.nbr + (int64_t)(k0 + k) * a.n_pad + i) : (int32_t)n_present;
#pragma unroll
            for (int k = 0; k < 4; ++k) n[k] = spins[j[k]];  // beyond the width: the zero dummy
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if constexpr (P == HS_FP64)
                        h[q] += n[k].v[q];
                    else
                        hl[q] = f_add(hl[q], two_sum(h[q], to_c(n[k].v[q])));
                }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const C s = to_c(sv.v[q]);
            if constexpr (P == HS_FP64) {
                b = fma(s, h[q], b);
                m[q] += s;
            } else {
                A.b.add_product(s, h[q], hl[q]);
                A.m[q].add(s);
            }
        }
        if (onsite) g += onsite64(a, to_c(sv.v[0]), to_c(sv.v[1]), to_c(sv.v[2]));
    }
    if constexpr (P != HS_FP64) {
        b = A.b.value();
#pragma unroll
        for (int q = 0; q < 3; ++q) m[q] = A.m[q].value();
        const bool small = P == HS_FP32 && fabs(b) < kSmallSum;
        if (small || !(isfinite(b) && isfinite(m[0]) && isfinite(m[1]) && isfinite(m[2]))) {  // as above
            b = m[0] = m[1] = m[2] = 0.0;
            for (int64_t i = t0; i < n_present; i += stride)
                for (int q = 0; q < 3; ++q) {
                    double h = 0.0;
                    for (int k = 0; k < a.width; ++k)
                        h += (double)to_c(spins[a.nbr[(int64_t)k * a.n_pad + i]].v[q]);
                    b += (double)to_c(spins[i].v[q]) * h;
                    m[q] += (double)to_c(spins[i].v[q]);
                }
        }
    }
    write_partials<double, true>(a, -0.5 * a.J * b - g, m[0], m[1], m[2], 0u);
}

// ----------------------------------------------------------------- fold
// Ring fold, after the last pass of a group of sweeps: CTA i sums ring slot i
// (sweep i of the group) and writes that sweep's record (its totals and
// observables); the last CTA to finish adds the records to the accumulator in
// sweep order, one lane per accumulated quantity.  Bound by that serial chain
// of FP64 additions, one per sweep and quantity: 64 of them in parallel lanes
// over records staged in shared memory, where one thread walking all of them
// through global memory took 26 us for 50 sweeps, in a launch of its own.
__device__ void fold_apply(const PassArgs &a, int n_slots) {
    __shared__ double s_rec[kRingMax][kSweepRecord];
    for (int k = threadIdx.x; k < n_slots * kSweepRecord; k += kBlock)
        s_rec[k / kSweepRecord][k % kSweepRecord] = __ldcg(a.sweep_tot + k);
    __syncthreads();
    const bool acc = a.accumulate == 1;
    DevAccum &A = *a.acc;
    const int t = threadIdx.x;
    // lane t < HS_N_MOMENTS: moment t += x y over the sweeps, x and y from the record (y = 1 but for E^2)
    constexpr int kE = kPartials, kMx = kPartials + 1;
    if (t < HS_N_MOMENTS) {
        if (acc) {
            const int idx[HS_N_MOMENTS] = {kE, kE, kMx + 3, kMx + 4, kMx + 5, kMx, kMx + 1, kMx + 2, kMx + 6};
            int at = 0;
#pragma unroll
            for (int q = 0; q < HS_N_MOMENTS; ++q) at = t == q ? idx[q] : at;
            double m = A.moments[t];
#pragma unroll 8
            for (int i = 0; i < n_slots; ++i) m = fma(s_rec[i][at], t == HS_SUM_E2 ? s_rec[i][at] : 1.0, m);
            A.moments[t] = m;
        }
    } else if (t == HS_N_MOMENTS) {
        if (acc) {
            double n = A.count;
            for (int i = 0; i < n_slots; ++i) n += 1.0;
            A.count = n;
        }
    } else if (t == 32) {
        double n = A.accepted;
#pragma unroll 8
        for (int i = 0; i < n_slots; ++i) n += s_rec[i][4];
        A.accepted = n;
    } else if (t >= 64 && t < 64 + kPartials) {
        A.sums[t - 64] = s_rec[n_slots - 1][t - 64];
    } else if (t >= 96 && t < 96 + 8) {
        if (acc) A.last[t - 96] = s_rec[n_slots - 1][kPartials + t - 96];
    }
}

__global__ void __launch_bounds__(kBlock) fold_kernel(const PassArgs a) {
    __shared__ int s_last;
    pdl_enter();
    // the group launch before it gave up (kAbandoned): its slots are incomplete, and nothing of them is added
    if (__ldcg(&a.acc->passed) & kAbandoned) return;
    double tot[kPartials];
    slot_totals<kBlock>(a, blockIdx.x, tot);
    if (threadIdx.x == 0) {
        double o[8];
        sweep_observables(tot, a.n_present, a.e, o);
        double *rec = a.sweep_tot + (size_t)blockIdx.x * kSweepRecord;
#pragma unroll
        for (int q = 0; q < kPartials; ++q) rec[q] = tot[q];
#pragma unroll
        for (int q = 0; q < 8; ++q) rec[kPartials + q] = o[q];
        __threadfence();
        s_last = atomicAdd(&a.acc->done, 1u) == gridDim.x - 1u;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    fold_apply(a, (int)gridDim.x);
    if (threadIdx.x == 0) a.acc->done = 0u;
}

// ----------------------------------------------------------------- init / layout
// Own sites of a periodic sc lattice or z-slab (nz planes from global plane
// z0, stored from array plane z_off of Lz_arr): index i runs over them in
// natural order; the global natural index is i + z0 Ly Lx.
template <int P>
__global__ void sc_init_kernel(void *planes, int Lx, int Ly, int nz, int Lz_arr, int z_off, int z0, int Lh, int mode,
                               double e0, double e1, double e2, uint32_t k0, uint32_t k1, uint32_t replica) {
    using S = typename Tr<P>::S;
    S *pl = (S *)planes;
    const int64_t plane = (int64_t)Lz_arr * Ly * Lh;
    const int64_t n = (int64_t)Lx * Ly * nz;
    const int64_t glob0 = (int64_t)z0 * Ly * Lx;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % Lx);
        const int64_t r = i / Lx;
        const int y = (int)(r % Ly), z = (int)(r / Ly);
        const int c = (x + y + z + z0) & 1;
        const int64_t idx = (r + (int64_t)z_off * Ly) * Lh + (x >> 1);
        double v[3] = {e0, e1, e2};
        if (mode == HS_INIT_RANDOM) {
            // counter (index lo, index hi, tag 1, replica): an initial spin has no sweep
            const uint64_t gi = (uint64_t)(i + glob0);
            const uint4 w = philox10(make_uint4((uint32_t)gi, (uint32_t)(gi >> 32), kTagInit << 24, replica), k0, k1);
            sphere_fp64(w, v[0], v[1], v[2]);
        }
        for (int q = 0; q < 3; ++q) pl[(int64_t)(3 * c + q) * plane + idx] = store_from_double<S>(v[q]);
    }
}

template <int P>
__global__ void table_init_kernel(void *spins4, const uint32_t *nat, int64_t n_present, int mode, double e0,
                                  double e1, double e2, uint32_t k0, uint32_t k1, uint32_t replica) {
    using S = typename Tr<P>::S;
    using S4 = Vec<S, 4>;
    S4 *sp = reinterpret_cast<S4 *>(spins4);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_present;
         i += (int64_t)gridDim.x * blockDim.x) {
        double v[3] = {e0, e1, e2};
        if (mode == HS_INIT_RANDOM) {
            const uint4 w = philox10(make_uint4(nat[i], 0u, kTagInit << 24, replica), k0, k1);
            sphere_fp64(w, v[0], v[1], v[2]);
        }
        S4 s;
        s.v[0] = store_from_double<S>(v[0]);
        s.v[1] = store_from_double<S>(v[1]);
        s.v[2] = store_from_double<S>(v[2]);
        s.v[3] = store_from_double<S>(0.0);
        sp[i] = s;
    }
}

template <int P>
__global__ void sc_scatter_kernel(void *planes, const double *xyz, int Lx, int Ly, int nz, int Lz_arr, int z_off,
                                  int z0, int Lh) {
    using S = typename Tr<P>::S;
    S *pl = (S *)planes;
    const int64_t plane = (int64_t)Lz_arr * Ly * Lh;
    const int64_t n = (int64_t)Lx * Ly * nz;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % Lx);
        const int64_t r = i / Lx;
        const int y = (int)(r % Ly), z = (int)(r / Ly);
        const int c = (x + y + z + z0) & 1;
        const int64_t idx = (r + (int64_t)z_off * Ly) * Lh + (x >> 1);
        for (int q = 0; q < 3; ++q) pl[(int64_t)(3 * c + q) * plane + idx] = store_from_double<S>(xyz[3 * i + q]);
    }
}

// A float's value as a double, from its bit fields in the integer pipe: the
// conversion instruction runs at the FP64 pipe's rate, 2 a cycle per SM.
__device__ __forceinline__ double widen(float f) {
    const uint32_t b = __float_as_uint(f), e = b & 0x7F800000u, m = b & 0x7FFFFFFFu;
    if (m != 0u && (e == 0u || e == 0x7F800000u)) return (double)f;  // subnormal, infinity, NaN
    const uint32_t hi = m == 0u ? b : ((b & 0x80000000u) | ((m >> 3) + (896u << 20)));
    return __hiloint2double((int)hi, (int)(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

// The whole state in natural order, FP64.  V sites of each colour at one row
// offset are 2 V consecutive sites; a CTA stages its kBlock such runs in
// shared memory and stores them as consecutive 16-byte pairs (8-byte ones
// where the caller's buffer is not 16-byte aligned), evict-first: the lattice
// stays in L2 for the next sweep.  Bound by HBM (read once, 24 bytes a site
// written: 3.6 GB at 464^3 FP32 in about 650 us); one thread per site with
// three strided stores and 64-bit divisions took 1102 us there.
template <int P, int V>
__global__ void __launch_bounds__(kBlock) sc_export_kernel(const void *planes, double *xyz, int Ly, int64_t plane,
                                                           int Lh, int z_off, int z0, FastDiv div_nxv, FastDiv div_ly,
                                                           uint32_t n_vec, int aligned) {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    using VT = Vec<S, V>;
    __shared__ __align__(16) C st[kBlock * 6 * V];
    const S *pl = (const S *)planes;
    for (uint64_t t0 = (uint64_t)blockIdx.x * kBlock; t0 < n_vec; t0 += (uint64_t)gridDim.x * kBlock) {
        const uint32_t cnt = (uint32_t)(n_vec - t0 < kBlock ? n_vec - t0 : kBlock);
        if (threadIdx.x < cnt) {
            const uint32_t t = (uint32_t)t0 + threadIdx.x;
            const uint32_t row = div_any(div_nxv, t);
            const uint32_t z = div_any(div_ly, row);
            const uint32_t y = row - z * (uint32_t)Ly;
            const int first = (int)((y + z + (uint32_t)z0) & 1u);  // the colour of even x in this row
            const int64_t idx = (int64_t)t * V + (int64_t)z_off * Ly * Lh;
            VT v[2][3];
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    v[c][q] = *reinterpret_cast<const VT *>(pl + (3 * (c ^ first) + q) * plane + idx);
            C *d = st + threadIdx.x * 6 * V;
            C out[6 * V];
#pragma unroll
            for (int j = 0; j < V; ++j)
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int q = 0; q < 3; ++q) out[6 * j + 3 * c + q] = to_c(v[c][q].v[j]);
#pragma unroll
            for (int k = 0; k < 3 * V; ++k)
                *reinterpret_cast<Vec<C, 2> *>(d + 2 * k) = Vec<C, 2>{{out[2 * k], out[2 * k + 1]}};
        }
        __syncthreads();
        double *o = xyz + t0 * 6 * V;
        for (uint32_t k = threadIdx.x; k < cnt * 3 * V; k += kBlock) {
            const Vec<C, 2> f = *reinterpret_cast<const Vec<C, 2> *>(st + 2 * k);
            const double2 w = make_double2(widen(f.v[0]), widen(f.v[1]));
            if (aligned) {
                __stcs(reinterpret_cast<double2 *>(o) + k, w);
            } else {
                __stcs(o + 2 * k, w.x);
                __stcs(o + 2 * k + 1, w.y);
            }
        }
        __syncthreads();
    }
}

// Spins of selected sites (global natural indices, own sites of the lattice
// or slab), in FP64, for lattices too large to copy whole.
template <int P>
__global__ void sc_gather_kernel(const void *planes, int Lx, int Ly, int Lz_arr, int z_off, int z0, int Lh, int64_t n,
                                 const int64_t *sites, double *out) {
    using S = typename Tr<P>::S;
    const S *pl = (const S *)planes;
    const int64_t plane = (int64_t)Lz_arr * Ly * Lh;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = sites[t];
        const int x = (int)(i % Lx);
        const int64_t r = i / Lx;
        const int y = (int)(r % Ly), z = (int)(r / Ly);
        const int c = (x + y + z) & 1;
        const int64_t idx = ((int64_t)(z - z0 + z_off) * Ly + y) * Lh + (x >> 1);
        for (int q = 0; q < 3; ++q) out[3 * t + q] = (double)to_c(pl[(int64_t)(3 * c + q) * plane + idx]);
    }
}

template <int P>
__global__ void table_convert_kernel(void *spins4, const uint32_t *nat, int64_t n_present, double *xyz,
                                     int to_layout) {
    using S = typename Tr<P>::S;
    using S4 = Vec<S, 4>;
    S4 *sp = reinterpret_cast<S4 *>(spins4);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_present;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t site = nat[i];
        if (to_layout) {
            S4 s;
            s.v[0] = store_from_double<S>(xyz[3 * site]);
            s.v[1] = store_from_double<S>(xyz[3 * site + 1]);
            s.v[2] = store_from_double<S>(xyz[3 * site + 2]);
            s.v[3] = store_from_double<S>(0.0);
            sp[i] = s;
        } else {
            const S4 s = sp[i];
            xyz[3 * site] = (double)to_c(s.v[0]);
            xyz[3 * site + 1] = (double)to_c(s.v[1]);
            xyz[3 * site + 2] = (double)to_c(s.v[2]);
        }
    }
}

inline int grid_for(int64_t n, int cap = 152 * 16) {
    int64_t g = (n + kBlock - 1) / kBlock;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

// Launch with programmatic stream serialisation (see pdl_enter).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_pdl_ptr(const void *kernel, int grid, int block, cudaStream_t s, const PassArgs &a) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    PassArgs args = a;
    void *params[] = {&args};
    return cudaLaunchKernelExC(&cfg, kernel, params);
}

// The neighbour-table kernel of a layout: unrolled rows for the crystals'
// widths (FP32: 6 and 8; its 12 would hold 60 registers of neighbours; FP16,
// whose spins are half as wide, 12 as well), a loop otherwise.  us per sweep,
// loop and unrolled: FP16 fcc 70^3 42.5 and 33.9, bcc 90^3 27.9 and 23.3, open
// sc 121^3 30.2 and 24.2; FP32 open sc 121^3 33.0 (with the L2 prefetch that it
// had; 27.7 without) and 24.6.
template <int P, int W, bool PFL2, bool TWO = false>
const void *table_variant(bool meas) {
    return meas ? (const void *)table_pass_kernel<P, true, false, PFL2, W, TWO>
                : (const void *)table_pass_kernel<P, false, false, PFL2, W, TWO>;
}
template <int P>
const void *table_kernel_ptr(const Layout &L, bool meas) {
    if (L.tensor)
        return meas ? (const void *)table_pass_kernel<P, true, true> : (const void *)table_pass_kernel<P, false, true>;
    if constexpr (P == HS_FP32)
        if (L.width == 8) return L.prefetch == 1 ? table_variant<P, 8, true>(meas) : table_variant<P, 8, false>(meas);
    if (L.prefetch == 1) return table_variant<P, 0, true>(meas);
    if constexpr (P != HS_FP64)
        if (L.width == 6) return table_variant<P, 6, false>(meas);
    if constexpr (P == HS_FP16) {
        if (L.width == 8) return table_variant<P, 8, false>(meas);
        if (L.width == 12) return table_variant<P, 12, false>(meas);
    }
    if constexpr (P == HS_FP64) {
        int64_t most = 0;  // sites of the largest class
        for (int c = 0; c < L.n_colours; ++c) most = std::max(most, L.colour_begin[c + 1] - L.colour_begin[c]);
        if (most > (int64_t)L.n_sm * kBlock) return table_variant<P, 0, false, true>(meas);
    }
    return table_variant<P, 0, false>(meas);
}

template <int P, int V, int PF>
cudaError_t launch_sc_pf(const PassArgs &a, int n_blocks, cudaStream_t s, bool meas) {
    return meas ? launch_pdl(sc_pass_kernel<P, V, true, PF>, n_blocks, kBlock, 0, s, a)
                : launch_pdl(sc_pass_kernel<P, V, false, PF>, n_blocks, kBlock, 0, s, a);
}

// the precisions and widths that have the ascending-only stencil variant
template <int P, int V>
constexpr bool has_plain_variant() {
    return (P == HS_FP32 && V == 4) || (P == HS_FP16 && V == 8);
}

template <int P, int V>
cudaError_t launch_sc_v(const PassArgs &a, int n_blocks, cudaStream_t s, bool meas, int pf, bool ten, bool plain) {
    // e = (0, 0, 1): the AX = 1 variant of the direction-capable stencil (lattices up to 2^31 sites).  The
    // ascending-only variant beyond keeps the general products: with AX = 1 it measured 120 against
    // 132-137 attempts/ns at 2048^3.
    if constexpr (P == HS_FP32 && V == 4)
        if (a.zaxis && pf == 0 && !ten && !plain)
            return meas ? launch_pdl(sc_pass_kernel<P, V, true, 0, false, true, 1>, n_blocks, kBlock, 0, s, a)
                        : launch_pdl(sc_pass_kernel<P, V, false, 0, false, true, 1>, n_blocks, kBlock, 0, s, a);
    if constexpr (has_plain_variant<P, V>())
        if (plain && pf == 0 && !ten)
            return meas ? launch_pdl(sc_pass_kernel<P, V, true, 0, false, false>, n_blocks, kBlock, 0, s, a)
                        : launch_pdl(sc_pass_kernel<P, V, false, 0, false, false>, n_blocks, kBlock, 0, s, a);
    if (ten)
        return meas ? launch_pdl(sc_pass_kernel<P, V, true, 0, true>, n_blocks, kBlock, 0, s, a)
                    : launch_pdl(sc_pass_kernel<P, V, false, 0, true>, n_blocks, kBlock, 0, s, a);
    if (pf == 1) return launch_sc_pf<P, V, 1>(a, n_blocks, s, meas);
    if (pf == 2) return launch_sc_pf<P, V, 2>(a, n_blocks, s, meas);
    return launch_sc_pf<P, V, 0>(a, n_blocks, s, meas);
}

// FP16 V = 8 (the pipelined kernel the FP16 workloads run) has the S.e = S_z
// variant for e = (0, 0, 1), chosen here rather than per work item.
template <int P, int V>
constexpr bool has_pipe_ax_variant() { return P == HS_FP16 && V == 8; }

template <int P, int V>
cudaError_t launch_pipe_v(const PassArgs &a, int n_blocks, cudaStream_t s, bool meas) {
    const size_t smem = PipeSlot<P, V>::kBytes;
    if constexpr (has_pipe_ax_variant<P, V>())
        if (a.zaxis)
            return meas ? launch_pdl(sc_pipe_kernel<P, V, true, 1>, n_blocks, kBlock, smem, s, a)
                        : launch_pdl(sc_pipe_kernel<P, V, false, 1>, n_blocks, kBlock, smem, s, a);
    return meas ? launch_pdl(sc_pipe_kernel<P, V, true>, n_blocks, kBlock, smem, s, a)
                : launch_pdl(sc_pipe_kernel<P, V, false>, n_blocks, kBlock, smem, s, a);
}

template <int P, int V>
cudaError_t launch_march_v(const PassArgs &a, int n_blocks, cudaStream_t s, bool meas) {
    return meas ? launch_pdl(sc_march_kernel<P, V, true>, n_blocks, kBlock, 0, s, a)
                : launch_pdl(sc_march_kernel<P, V, false>, n_blocks, kBlock, 0, s, a);
}

template <int P>
cudaError_t launch_pass_p(const Layout &L, const PassArgs &a, int n_blocks, cudaStream_t s) {
    const bool meas = a.accumulate != 0;
    if (L.kernel == kMarch) {
        switch (L.vec) {
        case 1: return launch_march_v<P, 1>(a, n_blocks, s, meas);
        case 2: return launch_march_v<P, 2>(a, n_blocks, s, meas);
        case 4: if constexpr (P != HS_FP64) return launch_march_v<P, 4>(a, n_blocks, s, meas); break;
        case 8: if constexpr (P == HS_FP16) return launch_march_v<P, 8>(a, n_blocks, s, meas); break;
        default: break;
        }
        return cudaErrorInvalidValue;
    }
    if (L.kernel == kPipe) {
        switch (L.vec) {
        case 1: if constexpr (P != HS_FP16) return launch_pipe_v<P, 1>(a, n_blocks, s, meas); break;
        case 2: return launch_pipe_v<P, 2>(a, n_blocks, s, meas);
        case 4: if constexpr (P != HS_FP64) return launch_pipe_v<P, 4>(a, n_blocks, s, meas); break;
        case 8: if constexpr (P == HS_FP16) return launch_pipe_v<P, 8>(a, n_blocks, s, meas); break;
        default: break;
        }
        return cudaErrorInvalidValue;
    }
    if (L.kernel == kStencil) {
        switch (L.vec) {
        case 1: return launch_sc_v<P, 1>(a, n_blocks, s, meas, L.prefetch, L.tensor != 0, L.plain);
        case 2: return launch_sc_v<P, 2>(a, n_blocks, s, meas, L.prefetch, L.tensor != 0, L.plain);
        case 4: if constexpr (P != HS_FP64) return launch_sc_v<P, 4>(a, n_blocks, s, meas, L.prefetch, L.tensor != 0, L.plain); break;
        case 8: if constexpr (P == HS_FP16) return launch_sc_v<P, 8>(a, n_blocks, s, meas, L.prefetch, L.tensor != 0, L.plain); break;
        default: break;
        }
        return cudaErrorInvalidValue;
    }
    return launch_pdl_ptr(table_kernel_ptr<P>(L, meas), n_blocks, kBlock, s, a);
}

}  // namespace

cudaError_t launch_fold(const PassArgs &a, int n_slots, cudaStream_t s) {
    if (n_slots < 1 || n_slots > kRingMax) return cudaErrorInvalidValue;
    return launch_pdl(fold_kernel, n_slots, kBlock, 0, s, a);
}

size_t storage_size(int precision) {
    return precision == HS_FP64 ? 8 : (precision == HS_FP32 ? 4 : 2);
}

static int64_t pass_items(const Layout &L) {
    if (L.structured) return (int64_t)L.nz * L.Ly * (L.Lh / L.vec);
    int64_t items = 0;
    for (int c = 0; c < L.n_colours; ++c)
        items = std::max<int64_t>(items, L.colour_begin[c + 1] - L.colour_begin[c]);
    return items;
}

template <int P, int V, int PF>
static const void *sc_ptr_pf(bool meas) {
    return meas ? (const void *)sc_pass_kernel<P, V, true, PF> : (const void *)sc_pass_kernel<P, V, false, PF>;
}

template <int P, int V>
static const void *sc_ptr(bool meas, int pf, bool ten, bool plain) {
    if constexpr (has_plain_variant<P, V>())
        if (plain && pf == 0 && !ten)
            return meas ? (const void *)sc_pass_kernel<P, V, true, 0, false, false>
                        : (const void *)sc_pass_kernel<P, V, false, 0, false, false>;
    if (ten)
        return meas ? (const void *)sc_pass_kernel<P, V, true, 0, true> : (const void *)sc_pass_kernel<P, V, false, 0, true>;
    if (pf == 1) return sc_ptr_pf<P, V, 1>(meas);
    if (pf == 2) return sc_ptr_pf<P, V, 2>(meas);
    return sc_ptr_pf<P, V, 0>(meas);
}

template <int P, int V>
static const void *march_ptr(bool meas) {
    return meas ? (const void *)sc_march_kernel<P, V, true> : (const void *)sc_march_kernel<P, V, false>;
}

template <int P, int V>
static const void *pipe_ptr(bool meas) {
    return meas ? (const void *)sc_pipe_kernel<P, V, true> : (const void *)sc_pipe_kernel<P, V, false>;
}

// the S.e = S_z twin of the pipelined kernel for this precision and width, or nullptr
static const void *pipe_ax_ptr(int precision, int vec, bool meas) {
    if (precision == HS_FP16 && vec == 8)
        return meas ? (const void *)sc_pipe_kernel<HS_FP16, 8, true, 1> : (const void *)sc_pipe_kernel<HS_FP16, 8, false, 1>;
    return nullptr;
}

template <int P>
static size_t pipe_bytes(int vec) {
    switch (vec) {
    case 1: if constexpr (P != HS_FP16) return PipeSlot<P, 1>::kBytes; break;
    case 2: return PipeSlot<P, 2>::kBytes;
    case 4: if constexpr (P != HS_FP64) return PipeSlot<P, 4>::kBytes; break;
    case 8: if constexpr (P == HS_FP16) return PipeSlot<P, 8>::kBytes; break;
    default: break;
    }
    return 0;
}

// 0 when the pipelined stencil has no variant for this precision and width
// (a slot vector must be 4, 8 or 16 bytes).
size_t pipe_smem_bytes(int precision, int vec) {
    switch (precision) {
    case HS_FP64: return pipe_bytes<HS_FP64>(vec);
    case HS_FP32: return pipe_bytes<HS_FP32>(vec);
    case HS_FP16: return pipe_bytes<HS_FP16>(vec);
    default: return 0;
    }
}

template <int P>
static const void *pass_kernel_ptr(const Layout &L, bool meas) {
    if (L.kernel == kMarch) {
        switch (L.vec) {
        case 1: return march_ptr<P, 1>(meas);
        case 2: return march_ptr<P, 2>(meas);
        case 4:
            if constexpr (P != HS_FP64) return march_ptr<P, 4>(meas);
            break;
        case 8:
            if constexpr (P == HS_FP16) return march_ptr<P, 8>(meas);
            break;
        default: break;
        }
        return nullptr;
    }
    if (L.kernel == kPipe) {
        switch (L.vec) {
        case 1:
            if constexpr (P != HS_FP16) return pipe_ptr<P, 1>(meas);
            break;
        case 2: return pipe_ptr<P, 2>(meas);
        case 4:
            if constexpr (P != HS_FP64) return pipe_ptr<P, 4>(meas);
            break;
        case 8:
            if constexpr (P == HS_FP16) return pipe_ptr<P, 8>(meas);
            break;
        default: break;
        }
        return nullptr;
    }
    if (L.kernel == kStencil) {
        switch (L.vec) {
        case 1: return sc_ptr<P, 1>(meas, L.prefetch, L.tensor != 0, L.plain);
        case 2: return sc_ptr<P, 2>(meas, L.prefetch, L.tensor != 0, L.plain);
        case 4:
            if constexpr (P != HS_FP64) return sc_ptr<P, 4>(meas, L.prefetch, L.tensor != 0, L.plain);
            break;
        case 8:
            if constexpr (P == HS_FP16) return sc_ptr<P, 8>(meas, L.prefetch, L.tensor != 0, L.plain);
            break;
        default: break;
        }
        return nullptr;
    }
    return table_kernel_ptr<P>(L, meas);
}

int pass_occupancy(int precision, const Layout &L, int accumulate) {
    const void *k = nullptr;
    switch (precision) {
    case HS_FP64: k = pass_kernel_ptr<HS_FP64>(L, accumulate != 0); break;
    case HS_FP32: k = pass_kernel_ptr<HS_FP32>(L, accumulate != 0); break;
    case HS_FP16: k = pass_kernel_ptr<HS_FP16>(L, accumulate != 0); break;
    default: break;
    }
    if (!k) return 1;
    size_t smem = 0;
    if (L.kernel == kPipe) {
        // opt in to the slots' dynamic shared memory and ask for a carveout
        // that holds two CTAs' slots, leaving the rest of the SM's 256 KB to
        // L1 (the neighbour rows shared by adjacent items)
        smem = pipe_smem_bytes(precision, L.vec);
        int dev = 0, per_sm = 0;
        if (smem == 0 || cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
            per_sm <= 0)
            return 0;
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return 0;
        const size_t per_cta = smem + fa.sharedSizeBytes + 1024;  // + the driver's reserved 1 KB
        const int pct = std::min(100, (int)((200 * per_cta + (size_t)per_sm - 1) / (size_t)per_sm));
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct) != cudaSuccess)
            return 0;
        // the launch may take the kernel's S.e = S_z twin (same slots and registers): the same opt-in
        if (const void *kx = pipe_ax_ptr(precision, L.vec, accumulate != 0))
            if (cudaFuncSetAttribute(kx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
                cudaFuncSetAttribute(kx, cudaFuncAttributePreferredSharedMemoryCarveout, pct) != cudaSuccess)
                return 0;
    }
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k, kBlock, smem) != cudaSuccess) return 1;
    if (L.kernel == kPipe) return blocks;
    return blocks > 0 ? blocks : 1;
}

// Persistent-style grid: resident CTAs per SM x SMs, never more CTAs than
// work items need.
int pass_blocks(int precision, const Layout &L, int n_sm, int blocks_per_sm) {
    (void)precision;
    return grid_for(pass_items(L), n_sm * std::max(blocks_per_sm, 1));
}

cudaError_t launch_pass(int precision, const Layout &L, const PassArgs &a, int n_blocks, cudaStream_t s) {
    switch (precision) {
    case HS_FP64: return launch_pass_p<HS_FP64>(L, a, n_blocks, s);
    case HS_FP32: return launch_pass_p<HS_FP32>(L, a, n_blocks, s);
    case HS_FP16: return launch_pass_p<HS_FP16>(L, a, n_blocks, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int P, int V>
static void measure_sc(const PassArgs &a, const Layout &L, int n_blocks, cudaStream_t s) {
    const uint32_t n_items = (uint32_t)((int64_t)L.nz * L.Ly * (L.Lh / V));
    if (a.tensor || (a.K != 0.0 && !a.zaxis))
        sc_measure_kernel<P, V, true><<<n_blocks, kBlock, 0, s>>>(a, L.planes, n_items);
    else
        sc_measure_kernel<P, V, false><<<n_blocks, kBlock, 0, s>>>(a, L.planes, n_items);
}

template <int P>
static bool measure_p(const Layout &L, const PassArgs &a, int n_blocks, cudaStream_t s) {
    if (!L.structured) {
        table_measure_kernel<P><<<n_blocks, kBlock, 0, s>>>(a, L.n_present);
        return true;
    }
    switch (L.vec) {
    case 1: measure_sc<P, 1>(a, L, n_blocks, s); return true;
    case 2: measure_sc<P, 2>(a, L, n_blocks, s); return true;
    case 4: if constexpr (P != HS_FP64) { measure_sc<P, 4>(a, L, n_blocks, s); return true; } break;
    case 8: if constexpr (P == HS_FP16) { measure_sc<P, 8>(a, L, n_blocks, s); return true; } break;
    default: break;
    }
    return false;
}

// CTAs of a measurement: enough threads to hide the loads of its short items (two sites of FP64 to eight of
// FP16), as many as the partials buffer holds at most.
int measure_blocks(const Layout &L, int n_sm, int max_blocks) {
    const int64_t items = L.structured ? pass_items(L) : L.n_present;
    return std::min(grid_for(items, n_sm * 6), max_blocks);
}

cudaError_t launch_measure(int precision, const Layout &L, const PassArgs &a, int n_blocks, cudaStream_t s) {
    bool known = false;
    switch (precision) {
    case HS_FP64: known = measure_p<HS_FP64>(L, a, n_blocks, s); break;
    case HS_FP32: known = measure_p<HS_FP32>(L, a, n_blocks, s); break;
    case HS_FP16: known = measure_p<HS_FP16>(L, a, n_blocks, s); break;
    default: break;
    }
    return known ? cudaGetLastError() : cudaErrorInvalidValue;
}

cudaError_t launch_init(int precision, const Layout &L, int mode, const double e[3], uint32_t key0, uint32_t key1,
                        uint32_t replica, cudaStream_t s) {
    if (L.structured) {
        const int g = grid_for(L.n_sites);
        switch (precision) {
        case HS_FP64:
            sc_init_kernel<HS_FP64><<<g, kBlock, 0, s>>>(L.planes, L.Lx, L.Ly, L.nz, L.Lz, L.slab ? 1 : 0, L.z0, L.Lh, mode, e[0], e[1], e[2],
                                                          key0, key1, replica);
            break;
        case HS_FP32:
            sc_init_kernel<HS_FP32><<<g, kBlock, 0, s>>>(L.planes, L.Lx, L.Ly, L.nz, L.Lz, L.slab ? 1 : 0, L.z0, L.Lh, mode, e[0], e[1], e[2],
                                                          key0, key1, replica);
            break;
        case HS_FP16:
            sc_init_kernel<HS_FP16><<<g, kBlock, 0, s>>>(L.planes, L.Lx, L.Ly, L.nz, L.Lz, L.slab ? 1 : 0, L.z0, L.Lh, mode, e[0], e[1], e[2],
                                                          key0, key1, replica);
            break;
        default: return cudaErrorInvalidValue;
        }
    } else {
        const int g = grid_for(L.n_present);
        switch (precision) {
        case HS_FP64:
            table_init_kernel<HS_FP64><<<g, kBlock, 0, s>>>(L.spins4, L.nat, L.n_present, mode, e[0], e[1], e[2],
                                                             key0, key1, replica);
            break;
        case HS_FP32:
            table_init_kernel<HS_FP32><<<g, kBlock, 0, s>>>(L.spins4, L.nat, L.n_present, mode, e[0], e[1], e[2],
                                                             key0, key1, replica);
            break;
        case HS_FP16:
            table_init_kernel<HS_FP16><<<g, kBlock, 0, s>>>(L.spins4, L.nat, L.n_present, mode, e[0], e[1], e[2],
                                                             key0, key1, replica);
            break;
        default: return cudaErrorInvalidValue;
        }
    }
    return cudaGetLastError();
}

template <int P>
static cudaError_t table_convert(const Layout &L, double *xyz, int to_layout, cudaStream_t s) {
    table_convert_kernel<P><<<grid_for(L.n_present), kBlock, 0, s>>>(L.spins4, L.nat, L.n_present, xyz, to_layout);
    return cudaGetLastError();
}

template <int P>
static cudaError_t scatter_p(const Layout &L, double *xyz, cudaStream_t s) {
    if (!L.structured) return table_convert<P>(L, xyz, 1, s);
    sc_scatter_kernel<P><<<grid_for(L.n_sites), kBlock, 0, s>>>(L.planes, xyz, L.Lx, L.Ly, L.nz, L.Lz, L.slab ? 1 : 0,
                                                                L.z0, L.Lh);
    return cudaGetLastError();
}

template <int P, int V>
static cudaError_t export_v(const Layout &L, double *xyz, cudaStream_t s) {
    const int64_t n_vec = (int64_t)L.nz * L.Ly * (L.Lh / V);
    sc_export_kernel<P, V><<<grid_for(n_vec, L.n_sm * 8), kBlock, 0, s>>>(
        L.planes, xyz, L.Ly, (int64_t)L.Lz * L.Ly * L.Lh, L.Lh, L.slab ? 1 : 0, L.z0, FastDiv((uint32_t)(L.Lh / V)),
        FastDiv((uint32_t)L.Ly), (uint32_t)n_vec, (uintptr_t)xyz % 16 == 0 ? 1 : 0);
    return cudaGetLastError();
}

// Vector width by what divides the row: four sites of FP32 / FP16, two of FP64 (16 bytes at most).
template <int P>
static cudaError_t gather_p(const Layout &L, double *xyz, cudaStream_t s) {
    if (!L.structured) return table_convert<P>(L, xyz, 0, s);
    if constexpr (P != HS_FP64)
        if (L.Lh % 4 == 0) return export_v<P, 4>(L, xyz, s);
    if (L.Lh % 2 == 0) return export_v<P, 2>(L, xyz, s);
    return export_v<P, 1>(L, xyz, s);
}

cudaError_t launch_gather_sites(int precision, const Layout &L, int64_t n, const int64_t *d_sites, double *d_out,
                                cudaStream_t s) {
    const int g = grid_for(n);
    const int z_off = L.slab ? 1 : 0;
    switch (precision) {
    case HS_FP64:
        sc_gather_kernel<HS_FP64><<<g, kBlock, 0, s>>>(L.planes, L.Lx, L.Ly, L.Lz, z_off, L.z0, L.Lh, n, d_sites, d_out);
        break;
    case HS_FP32:
        sc_gather_kernel<HS_FP32><<<g, kBlock, 0, s>>>(L.planes, L.Lx, L.Ly, L.Lz, z_off, L.z0, L.Lh, n, d_sites, d_out);
        break;
    case HS_FP16:
        sc_gather_kernel<HS_FP16><<<g, kBlock, 0, s>>>(L.planes, L.Lx, L.Ly, L.Lz, z_off, L.z0, L.Lh, n, d_sites, d_out);
        break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_scatter(int precision, const Layout &L, const double *d_xyz, cudaStream_t s) {
    double *xyz = const_cast<double *>(d_xyz);
    switch (precision) {
    case HS_FP64: return scatter_p<HS_FP64>(L, xyz, s);
    case HS_FP32: return scatter_p<HS_FP32>(L, xyz, s);
    case HS_FP16: return scatter_p<HS_FP16>(L, xyz, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_gather(int precision, const Layout &L, double *d_xyz, cudaStream_t s) {
    switch (precision) {
    case HS_FP64: return gather_p<HS_FP64>(L, d_xyz, s);
    case HS_FP32: return gather_p<HS_FP32>(L, d_xyz, s);
    case HS_FP16: return gather_p<HS_FP16>(L, d_xyz, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hs
