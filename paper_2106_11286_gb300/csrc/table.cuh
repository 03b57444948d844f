// One site's update on the neighbour-table layout, shared by the colour-pass
// kernel (kernels.cu) and the launch of whole groups of sweeps (table_group.cu).
#pragma once

#include "device.cuh"

namespace hs {
namespace {

// A site's FP64 field, its neighbours read again through the table (for a decision that FP32 left open).
__device__ __noinline__ double3 table_field64(const Vec<double, 4> *spins, const int32_t *nbr, int64_t i, int64_t n_pad,
                                              int width) {
    double3 h = make_double3(0.0, 0.0, 0.0);
    for (int k = 0; k < width; ++k) {
        const Vec<double, 4> n = spins[__ldg(nbr + (int64_t)k * n_pad + i)];
        h.x += n.v[0];
        h.y += n.v[1];
        h.z += n.v[2];
    }
    return h;
}

// The local field of a site and, for the energy, the part of it from lower
// colour classes (j < a.colour_begin), its neighbours added in stored order.
// FP64 without the tensor term keeps the field in FP32 (g, the decision's) and
// the energy's part in FP64.
template <int P, bool MEAS, bool TEN>
struct TableField {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    static constexpr bool kNarrow = P == HS_FP64 && !TEN;
    C hx = C(0), hy = C(0), hz = C(0);
    C lx = C(0), ly = C(0), lz = C(0);
    float gx = 0.0f, gy = 0.0f, gz = 0.0f;
    int big = 0;
    __device__ __forceinline__ void add(const PassArgs &a, int32_t j, const Vec<S, 4> &n) {
        const C nx = to_c(n.v[0]), ny = to_c(n.v[1]), nz = to_c(n.v[2]);
        if constexpr (kNarrow) {
            gx = f_add(gx, narrow(nx, big));
            gy = f_add(gy, narrow(ny, big));
            gz = f_add(gz, narrow(nz, big));
        } else {
            hx += nx;
            hy += ny;
            hz += nz;
        }
        if (MEAS && j < a.colour_begin) {
            lx += nx;
            ly += ny;
            lz += nz;
        }
    }
};

// The trial and acceptance uniform of renumbered site i (they need no spin).
template <int P>
struct TableTrial {
    float x, y, z, u;
};
template <>
struct TableTrial<HS_FP64> {
    Trial64 t;
    uint32_t px, py;
};
template <int P>
__device__ __forceinline__ void draw_table_trial(const PassArgs &a, int64_t i, TableTrial<P> &t) {
    if constexpr (P == HS_FP64) {
        const uint32_t site = __ldg(a.nat + i);
        t.t = trial64(trial64_block(site, a.sweep, (uint32_t)a.colour, 0u, a.replica, a.key0, a.key1), a.sc_tab);
        const uint4 w = trial64_block(site, a.sweep, (uint32_t)a.colour, 1u, a.replica, a.key0, a.key1);
        t.px = w.x;
        t.py = w.y;
    } else {
        draw_trial_rank<P>((uint32_t)(i - a.colour_begin), a.sweep, (uint32_t)a.colour, a.replica, a.key0, a.key1, t.x,
                           t.y, t.z, t.u);
    }
}

// A thread's sums of a pass.
template <int P>
struct TableAcc {
    using C = typename Tr<P>::C;
    C e = C(0), x = C(0), y = C(0), z = C(0);
    unsigned n = 0;
};

// Metropolis step (iii) of site i: s becomes the trial if it is accepted (the
// caller stores it); the sums take the final spin.
template <int P, bool MEAS, bool TEN>
__device__ __forceinline__ bool table_update(const PassArgs &a, int64_t i, const Vec<typename Tr<P>::S, 4> *spins,
                                             TableField<P, MEAS, TEN> &f, const TableTrial<P> &t,
                                             Vec<typename Tr<P>::S, 4> &s, typename Tr<P>::C J, typename Tr<P>::C K,
                                             typename Tr<P>::C ex, typename Tr<P>::C ey, typename Tr<P>::C ez,
                                             typename Tr<P>::C beta, TableAcc<P> &acc) {
    using S = typename Tr<P>::S;
    using C = typename Tr<P>::C;
    C sx = to_c(s.v[0]), sy = to_c(s.v[1]), sz = to_c(s.v[2]);
    C tx, ty, tz;
    bool accepted;
    if constexpr (P == HS_FP64) {
        const float uf = (float)(t.px >> 8) * 0x1p-24f;
        tx = t.t.x;
        ty = t.t.y;
        tz = t.t.z;
        if constexpr (!TEN) {
            const float fx = narrow(sx, f.big), fy = narrow(sy, f.big), fz = narrow(sz, f.big);
            const Dots32<float> d = site_math32<float>(fx, fy, fz, t.t.fx, t.t.fy, t.t.fz, f.gx, f.gy, f.gz, a.fJ, a.fK,
                                                       a.fe[0], a.fe[1], a.fe[2]);
            int dec = decide64(-a.fbeta * d.dH, a.fdelta, uf);
            if (f.big > 0x3FF00100) dec = -1;  // 1 + 2^-12: no unit vectors
            if (dec < 0) {
                const double3 h = table_field64(spins, a.nbr, i, a.n_pad, a.width);
                dec = accept_wide<false>(sx, sy, sz, tx, ty, tz, h.x, h.y, h.z, J, K, ex, ey, ez, beta,
                                         (double)bits53(t.px, t.py) * 0x1p-53, uf);
            }
            accepted = dec > 0;
        } else {
            accepted = metropolis<C, TEN>(sx, sy, sz, tx, ty, tz, f.hx, f.hy, f.hz, J, K, ex, ey, ez, beta,
                                          (double)bits53(t.px, t.py) * 0x1p-53, uf, a.A)
                           .acc;
        }
    } else {
        tx = t.x;
        ty = t.y;
        tz = t.z;
        const Dots32<float> d = site_math32<float, TEN>(sx, sy, sz, tx, ty, tz, f.hx, f.hy, f.hz, J, K, ex, ey, ez, a.fA);
        accepted = accept32(d.dH, t.u, neg_beta_log2e(beta));
    }
    if (accepted) {
        sx = tx;
        sy = ty;
        sz = tz;
        s.v[0] = to_store<S, C>(tx);
        s.v[1] = to_store<S, C>(ty);
        s.v[2] = to_store<S, C>(tz);
        ++acc.n;
    }
    if (MEAS) {
        const C se = sx * ex + sy * ey + sz * ez;
        acc.e += -J * (sx * f.lx + sy * f.ly + sz * f.lz) - K * se * se;
        if constexpr (TEN) {
            if constexpr (P == HS_FP64)
                acc.e -= quad64(sx, sy, sz, a.A);
            else
                acc.e -= quad32<float>(sx, sy, sz, a.fA);
        }
        acc.x += sx;
        acc.y += sy;
        acc.z += sz;
    }
    return accepted;
}

}  // namespace
}  // namespace hs
