// Internal declarations of the GB300 Metropolis library (not part of the ABI).
//
// Device layouts (all in HBM, allocated by the lattice handle):
//  * stencil path (unmasked periodic sc, Lx/2 divisible by the vector width):
//    colour-major SoA.  Plane (colour c, component a) is an array
//    [Lz][Ly][Lx/2] of the storage type; site (x,y,z) of colour
//    c = (x+y+z)&1 sits at xh = x/2 in row (z,y).  Planes are ordered
//    c0x c0y c0z c1x c1y c1z so that one colour is 3 contiguous planes.
//  * table path (everything else): present sites renumbered colour by colour
//    (ascending natural index inside a class); spins as 4-vectors (x,y,z,0)
//    of the storage type, one per renumbered site plus one zero dummy at the
//    end; neighbour table [width][n_pad] of renumbered indices, padded with
//    the dummy; nat[i] = natural index of renumbered site i.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/hs.h"

namespace hs {

constexpr int kPartials = 5;  // E, Sx, Sy, Sz, accepted
constexpr int kRingMax = 64;  // sweeps whose slots a ring fold takes at most
constexpr int kSweepRecord = kPartials + 8;  // a ring fold's per-sweep record: totals, observables
constexpr int kBlock = 256;   // threads per CTA of the sweep kernels
// partial-sum sets per colour of a z-slab: first own plane, last own plane,
// the planes between them, the whole slab in one launch
constexpr int kSlabSets = 4;

// Division by a runtime constant d (1 <= d < 2^31) of numerators n < 2^31
// by multiply-high and shift: with l = ceil(log2 d) and m = ceil(2^(31+l)/d)
// (m < 2^32), floor(n m / 2^(31+l)) = floor(n / d) because the rounding
// excess n (m - 2^(31+l)/d) / 2^(31+l) stays below 2^-l <= 1/d.
#ifdef __CUDACC__
#define HS_HOST_DEVICE __host__ __device__
#else
#define HS_HOST_DEVICE
#endif

struct FastDiv {
    uint32_t d, m, l;
    HS_HOST_DEVICE FastDiv() : d(1), m(0), l(0) {}
    explicit FastDiv(uint32_t div) : d(div), l(0) {
        while ((1ull << l) < div) ++l;
        m = (l == 0) ? 0u : (uint32_t)(((1ull << (31 + l)) + div - 1) / div);
    }
#ifdef __CUDACC__
    __device__ __forceinline__ uint32_t div(uint32_t n) const { return l == 0 ? n : (__umulhi(n, m) >> (l - 1)); }
#endif
};

constexpr unsigned long long kAbandoned = 1ull << 63;  // in DevAccum::passed: a wait of this hs_sweep call ran out

// Device-resident accumulator block of one lattice.
struct DevAccum {
    double moments[HS_N_MOMENTS];
    double count;          // accumulated sweeps
    double accepted;       // accepted moves since the last hs_sweep began
    unsigned long long passed;  // CTA arrivals at the pass barrier of a cooperative sweep launch since then (kAbandoned)
    double last[8];        // E, Mx, My, Mz, |M|, M2, M4, |M.e| of the last finalised reduction
    unsigned int done;     // CTA arrival counter of the finishing pass
    int error;             // latched device error code (0 = none)
    double sums[5];        // E, sum S_x, sum S_y, sum S_z, accepted moves of the last finalised reduction
};

// Parameters of one colour pass.
struct PassArgs {
    // stencil layout
    void *own[3];
    const void *oth[3];
    int Lx, Ly, Lz, Lh;
    FastDiv div_nxv, div_ly;   // row = t / (Lh/V), z = row / Ly
    int nz, z_off;             // planes updated, array plane of the first (1 for a z-slab: plane 0 is a halo)
    int zpar;                  // parity of (global z - array z), for the colour of a row
    uint32_t site_off;         // global natural index - (array row Lx + x), mod 2^32
    uint32_t rank_off;         // colour rank of a site - (array row Lh + x / 2), mod 2^32
    int ty;                    // z-march stencil: rows per plane-slab
    uint32_t rev;              // register stencil: nonzero = work items in descending order, item t taken as
                               // rev - t (rev = items - 1)
    // table layout
    void *spins4;           // 4-vectors, renumbered order
    const int32_t *nbr;     // [width][n_pad]
    const uint32_t *nat;    // natural index per renumbered site
    int width;
    int64_t n_pad;
    int64_t begin, end;     // renumbered range of this colour
    int64_t colour_begin;   // first renumbered index of this colour (energy split)
    // common
    int colour;
    int n_colours;
    double J, K, e[3];
    double beta;
    float fJ, fK, fe[3], fbeta;  // the same in FP32 for the FP32 / FP16 kernels
    int tensor;             // 1: the on-site anisotropy tensor term is on
    double A[6];            // its symmetric tensor (xx, yy, zz, xy, xz, yz)
    float fA[6];
    const ulonglong2 *sc_tab;  // FP64 trial: sin, cos(pi j / 4096) in units of 2^-63, j = 0..1024
    int zaxis;              // 1: e = (0, 0, 1) exactly (the FP64 stencil takes S.e = S_z)
    uint32_t key0, key1, replica, sweep;
    float fdelta;           // FP64: bound on the error of the FP32 form of beta dH (decision_band); in what was
                            // padding: the FP32 stencil measured 4 % slower with the words before it shifted
    double *partials;       // [ring slots][n_colours][n_blocks][kPartials]; a slab has kSlabSets sets per colour
                            // (pass = kSlabSets colour + set, n_colours = 2 kSlabSets); a launch of fewer CTAs
                            // than n_blocks leaves the rest of its set zero
    double *sweep_tot;      // [ring slots][kSweepRecord]: per-sweep records of a ring fold
    int pass;               // colour index = partial slot
    int slot;               // ring slot: the sweep's index within its fold group (0 for single passes)
    int n_blocks;
    int finish;             // 1: last launch of the sequence, its last CTA to arrive reduces and finalises
    uint64_t skip_sets;     // finaliser: partial sets of the slot left out (bit p = set p; not written this sweep)
    int accumulate;         // 0: no fused measurement; 1: measure and add the moments to the accumulator;
                            // 2: measure only (the sums; a slab whose moments come from all slabs' sums)
    double n_present;
    DevAccum *acc;
};

// codes as in hs_kernel (include/hs.h)
enum KernelKind { kStencil = 1, kTable = 3, kMarch = 4, kPipe = 5 };

struct Layout {
    bool structured;
    bool slab;              // z-slab of a periodic sc lattice: Lz = nz + 2 array planes, halos at 0 and nz + 1
    int z0, nz, Lz_glob;    // first global plane, own planes, global Lz (slab); 0, Lz, Lz otherwise
    int kernel;             // KernelKind
    int vec;                // vector width of the stencil kernels
    int prefetch;           // register stencil: 0 none, 1 next work item in registers, 2 split prefetch
    int tensor;             // 1: the on-site anisotropy tensor term is on (register stencil without
                            //    prefetch, or the neighbour table)
    int ty;                 // z-march stencil: rows per plane-slab
    int order;              // register stencil: 1 ascending passes, 2 alternating (colour 1 descending)
    bool plain;             // register stencil: the ascending-only variant (lattices beyond 2^31 sites)
    int n_sm;               // SMs of the lattice's device
    int n_colours;
    int64_t n_sites, n_present;
    // stencil
    int Lx, Ly, Lz, Lh;
    void *planes;           // 6 planes of Lz*Ly*Lh elements
    // table
    void *spins4;
    int32_t *nbr;
    uint32_t *nat;
    int width;
    int64_t n_pad;
    int64_t colour_begin[65];  // renumbered colour ranges (n_colours + 1 entries)
};

// How far the FP32 form of beta dH may be from the FP64 one, for spins whose
// components are at most 1 + 2^-12 (of any length: unit vectors stay well
// inside) and w neighbours.  In units of 2^-24, per field component: w operands
// truncated to FP32 (2 each) and w - 1 additions of sums up to w (w each),
// w^2 + w at most; so S.h is off by at most 3 (w^2 + w) + 6 w (S truncated) +
// 9 w (the products' roundings), S'.h by less, and J (S.h - S'.h) by twice that
// + 6 w + 12 w: 6 w^2 + 54 w in all (540 for six neighbours, 3.2e-5; 1512 for
// fcc's twelve), a quarter more for what exceeds 1; a field taken from FP64 is
// closer.  The uniaxial term: S.e off by 12 each, times a sum of at most 3.5,
// with its roundings below 200 < 2e-5 / 2^-24 = 335.  Infinite (FP64 decides
// every site) where J, K or beta leave FP32's range.  No width is left out: a
// table of 14 neighbours whose sites FP64 all decided took its gathers twice,
// 103 us per sweep of 27,648 sites against 90 without the FP32 form, and 54 with
// it deciding (26 neighbours 211, 169 and 101; 1,024,000 sites of 14 259, 258
// and 127).
inline float decision_band(double beta, double J, double K, int width) {
    auto fits = [](double v) { return v == 0.0 || (v >= 1e-30 && v <= 1e30); };
    const double aJ = J < 0 ? -J : J, aK = K < 0 ? -K : K;
    if (!fits(beta) || !fits(aJ) || !fits(aK) || !fits(beta * aJ) || !fits(beta * aK)) return __builtin_inff();
    const double w = width, units = 1.25 * (6.0 * w * w + 54.0 * w);
    return (float)(beta * (aJ * units * 0x1p-24 + aK * 2e-5) * 1.001);
}

// Fewer items than the SMs have threads of one CTA each: CTAs of as few warps
// as spread them over every SM (a pass of few warps is bound by each SM's
// multiply and FP64 pipes and its load latency; the warps' items, and with them
// the FP32 sums, stay the same).  us per sweep with CTAs of 256 threads and so:
// FP64 32^3 8.9 and 7.2, fcc FP64 of 73,656 sites 26.3 and 20.6; 48^3 FP32 5.6
// and 5.0.
inline void spread_ctas(int64_t items, int n_sm, int &ctas, int &threads) {
    if (items >= (int64_t)n_sm * kBlock) return;
    threads = 32 * (int)((items + 32 * (int64_t)n_sm - 1) / (32 * (int64_t)n_sm));
    ctas = (int)((items + threads - 1) / threads);
}

size_t storage_size(int precision);

// Record the thread-local message returned by hs_last_error; returns code.
int set_last_error(int code, const std::string &msg);

// Kernel launchers (kernels.cu).  All return cudaError_t of the launch.
cudaError_t launch_pass(int precision, const Layout &L, const PassArgs &a, int n_blocks, cudaStream_t s);
cudaError_t launch_init(int precision, const Layout &L, int mode, const double e[3], uint32_t key0,
                        uint32_t key1, uint32_t replica, cudaStream_t s);
cudaError_t launch_gather_sites(int precision, const Layout &L, int64_t n, const int64_t *d_sites, double *d_out,
                                cudaStream_t s);
cudaError_t launch_scatter(int precision, const Layout &L, const double *d_xyz, cudaStream_t s);
cudaError_t launch_gather(int precision, const Layout &L, double *d_xyz, cudaStream_t s);
// Standalone measurement: a.colour = 1, a.n_blocks = n_blocks = measure_blocks(...).
cudaError_t launch_measure(int precision, const Layout &L, const PassArgs &a, int n_blocks, cudaStream_t s);
int measure_blocks(const Layout &L, int n_sm, int max_blocks);
// Fold ring slots 0 .. n_slots-1 (sweeps of a.n_colours passes each, in sweep
// order) into the accumulator: one CTA per slot sums it, the last of them
// applies the totals in order.  1 <= n_slots <= kRingMax.
cudaError_t launch_fold(const PassArgs &a, int n_slots, cudaStream_t s);
int pass_blocks(int precision, const Layout &L, int n_sm, int blocks_per_sm);
int pass_occupancy(int precision, const Layout &L, int accumulate);
size_t pipe_smem_bytes(int precision, int vec);  // dynamic shared memory of the pipelined stencil

}  // namespace hs
