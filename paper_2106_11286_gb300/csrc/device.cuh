// Device building blocks shared by the colour-pass kernels (kernels.cu) and
// the batched persistent kernel (batch.cu): Philox4x32-10, the trial
// orientation, the Metropolis test of Eq. 1, the fused reductions and the
// stencil work item.  Internal to the library.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>
#include <string.h>

#include "hs_impl.h"

namespace hs {
namespace {


// ----------------------------------------------------------------- Philox
// Philox4x32-10 as published (Salmon et al., SC'11): ten rounds of two
// 32x32->64 multiplies with fixed odd multipliers, a cross-lane swap of the
// high halves xored with the round key, and a Weyl key schedule.
constexpr uint32_t kMulA = 0xD2511F53u;
constexpr uint32_t kMulB = 0xCD9E8D57u;
constexpr uint32_t kWeylA = 0x9E3779B9u;
constexpr uint32_t kWeylB = 0xBB67AE85u;

__device__ __forceinline__ uint4 philox10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t pa = (uint64_t)kMulA * c.x;  // one 32x32->64 multiply per lane pair
        const uint64_t pb = (uint64_t)kMulB * c.z;
        c = make_uint4((uint32_t)(pb >> 32) ^ c.y ^ k0, (uint32_t)pb, (uint32_t)(pa >> 32) ^ c.w ^ k1, (uint32_t)pa);
        k0 += kWeylA;
        k1 += kWeylB;
    }
    return c;
}

// Programmatic dependent launch: a pass kernel lets the next kernel in the
// stream be scheduled as its own CTAs retire, then waits until the previous
// kernel has completed and its writes are visible before touching memory.
// Without a programmatic dependency both instructions are no-ops.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr uint32_t kTagTrial = 0u;
constexpr uint32_t kTagInit = 1u;

// ----------------------------------------------------------------- precision
template <int P> struct Tr;
template <> struct Tr<HS_FP64> { using S = double; using C = double; };
template <> struct Tr<HS_FP32> { using S = float; using C = float; };
template <> struct Tr<HS_FP16> { using S = __half; using C = float; };

__device__ __forceinline__ double to_c(double v) { return v; }
__device__ __forceinline__ float to_c(float v) { return v; }
__device__ __forceinline__ float to_c(__half v) { return __half2float(v); }

template <typename S> __device__ __forceinline__ S store_from_double(double v);
template <> __device__ __forceinline__ double store_from_double<double>(double v) { return v; }
template <> __device__ __forceinline__ float store_from_double<float>(double v) { return __double2float_rn(v); }
template <> __device__ __forceinline__ __half store_from_double<__half>(double v) { return __double2half(v); }

template <typename T, int V>
struct alignas(sizeof(T) * V) Vec {
    T v[V];
};

// Uniform point on the sphere in FP64 from one Philox block (words 0,1 -> u_z,
// words 2,3 -> u_phi, 53 bits each): z = 2u_z - 1 and v = 2u_phi - 1 are
// formed exactly from the integers, r = sqrt((1-z)(1+z)) is correctly
// rounded, phi = pi v.
__device__ __forceinline__ void sphere_fp64(uint4 w, double &x, double &y, double &z) {
    const int64_t two52 = int64_t(1) << 52;
    const int64_t iz = (int64_t)((((uint64_t)(w.x >> 5)) << 26) | (uint64_t)(w.y >> 6));
    const int64_t iv = (int64_t)((((uint64_t)(w.z >> 5)) << 26) | (uint64_t)(w.w >> 6));
    z = (double)(iz - two52) * 0x1p-52;
    const double v = (double)(iv - two52) * 0x1p-52;
    const double r = sqrt((1.0 - z) * (1.0 + z));
    double sn, cs;
    sincospi(v, &sn, &cs);
    x = r * cs;
    y = r * sn;
}

// ---- FP64 trial orientation in the integer pipe.  The FP64 pipe issues 2
// instructions per cycle per SM, the integer units 32 (32x32->64 multiply) to
// 128 (add, logic), so the sphere point is formed in 64-bit fixed point, about
// 200 integer instructions, where FP64 took 26 that cost as much as 1600.
//
// floor(a b / 2^64), low partial product left out: at most 3 too small.
__device__ __forceinline__ uint64_t mulhi_64(uint64_t a, uint64_t b) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}

// v 2^-s as a double rounded to nearest (e0 = 1085 - s), with the given sign.
__device__ __forceinline__ double fixed_to_double(uint64_t v, int e0, bool neg) {
    const int n = __clzll((long long)(v | 1ull));
    const uint64_t w = v << n;  // leading bit at 63
    const uint64_t mant = (w >> 11) + ((w >> 10) & 1ull);
    const uint64_t bits = (mant + ((uint64_t)(uint32_t)(e0 - n) << 52)) | ((uint64_t)neg << 63);
    return v == 0 ? 0.0 : __longlong_as_double((long long)bits);
}

// The 53-bit uniform of two Philox words.
__device__ __forceinline__ uint64_t bits53(uint32_t a, uint32_t b) {
    return ((uint64_t)(a >> 5) << 26) | (uint64_t)(b >> 6);
}

// A trial spin and its components in FP32 (error below 2^-23).
struct Trial64 {
    double x, y, z;
    float fx, fy, fz;
};

// The sphere point of sphere_fp64 from one Philox block.  Small components carry
// their digits too: r and a small sine keep an exponent of their own.
//  * z = (iz - 2^52) 2^-52 exactly.
//  * r = sqrt((1 - |z|)(1 + |z|)): both factors are exact integers; 1 - |z| is
//    scaled up by an even power of two, so their product W lies in
//    [1/16, 1/2); sqrt(W) starts from the hardware reciprocal square root
//    (2^-22) and takes two Newton steps on the exact residual, W - Y^2 (2^-44,
//    then below 2^-60); the scale's root goes into the result's exponent.
//  * phi = pi v = pi t - pi, t = iv 2^-52: sin and cos of pi t by octant, so
//    that what may be small is a sine of an angle counted from its axis, table
//    and angle addition (Tang, "Table-lookup algorithms for elementary functions
//    and their error analysis", 1991): 1025 entries of sin, cos (pi j / 4096) in
//    units of 2^-63, then theta < pi/2 2^-11 by sin theta = theta - theta^3/6
//    (first omitted term 2^-58.6) and 1 - cos theta = theta^2/2 - theta^4/24
//    (omitted 2^-71).  In the first step (one site of 1024) the sine is theta's
//    own, from theta scaled up to 64 digits, with theta^5/120 (omitted term
//    2^-74 of theta).
// Against 128-bit arithmetic over 4 million words, most of them beside the poles
// and axes, components are within 0.52 units in their last place from 1/2 to 1,
// 1.2 above 2^-6, 3.2 above 2^-8 and 14 at any size; an FP64 form of this point
// (2048 centred entries, theta^3 and theta^4) was off by up to 6.7 above 1/16,
// 440 down to 2^-19, and by 2^-62 whatever the size below that.  With r and the
// sines in fixed point alone the small components lost digits (570 units at
// 2^-16, 5200 at 2^-19) for 3.5 % less time, 10 sweeps of 256^3 6.72 against 6.97
// ms, 100 of 16^3 580 against 601 us.
__device__ __forceinline__ Trial64 trial64(uint4 w, const ulonglong2 *tab) {
    Trial64 t;
    const uint64_t one = 1ull << 52, half_pi = 0xC90FDAA22168C235ull;  // pi/2 2^63
    const uint64_t iz = bits53(w.x, w.y), iv = bits53(w.z, w.w);
    const bool zneg = iz < one;
    const uint64_t m = zneg ? one - iz : iz - one;  // |z| 2^52
    t.z = fixed_to_double(m, 1033, zneg);
    t.fz = (float)(uint32_t)(m >> 21) * 0x1p-31f;
    t.fz = zneg ? -t.fz : t.fz;

    const uint64_t A = one - m;
    const int sh = __clzll((long long)(A | 1ull)) & ~1;  // 10 .. 62
    const uint64_t W = mulhi_64(A << sh, (one + m) << 10);
    const float wf = (float)(uint32_t)(W >> 32) * 0x1p-32f;
    const float rs = rsqrtf(fmaxf(wf, 0.0625f));
    const uint32_t Y0 = __float2uint_rz(wf * rs * 0x1p32f);
    const int32_t R = __float2int_rz(rs * 0x1p28f);  // (1 / (2 sqrt W)) 2^29
    const int64_t E0 = (int64_t)(W - (uint64_t)Y0 * Y0);  // below 2^43
    const int64_t d0 = (int64_t)(int32_t)(E0 >> 12) * R;  // units of 2^-81
    const uint64_t Y1 = ((uint64_t)Y0 << 32) + (uint64_t)(d0 >> 17);
    const int32_t E1 = (int32_t)(uint32_t)(W - mulhi_64(Y1, Y1));
    const uint64_t r = Y1 + (uint64_t)(((int64_t)E1 * R) >> 29);  // units of 2^-(62 + rexp)
    const int rexp = (sh >> 1) - 5;                               // 0 .. 26

    const uint32_t quad = (uint32_t)(iv >> 51);
    const bool upper = (uint32_t)(iv >> 50) & 1u;  // the quadrant's upper octant: counted down from its end
    const uint64_t g = upper ? (1ull << 51) - (iv & ((1ull << 51) - 1ull)) : iv & ((1ull << 50) - 1ull);
    const uint32_t j = (uint32_t)(g >> 40);  // 0 .. 1024
    const ulonglong2 sc = __ldg(tab + j);
    const uint64_t low = g << 24;
    const uint64_t u = mulhi_64(low, half_pi);  // theta 2^11, units of 2^-63
    const uint64_t s2 = mulhi_64(u, u);         // theta^2 2^22, units of 2^-62
    const uint32_t s2h = (uint32_t)(s2 >> 32);
    // (1 - cos theta) 2^23, units of 2^-62, and sin theta 2^11, units of 2^-63 (1/3 and 1/6 in 32 bits)
    const uint64_t c = s2 - ((uint64_t)__umulhi(__umulhi(s2h, s2h), 0x55555555u) << 10);
    const uint64_t sx = u - ((uint64_t)__umulhi(__umulhi(s2h, (uint32_t)(u >> 32)), 0x2AAAAAABu) << 12);
    uint64_t sn = sc.x + (mulhi_64(sc.y, sx) >> 10) - (mulhi_64(sc.x, c) >> 21);  // units of 2^-(63 + sexp)
    const uint64_t cs = sc.y - (mulhi_64(sc.x, sx) >> 10) - (mulhi_64(sc.y, c) >> 21);
    int sexp = 0;
    if (j == 0u) {  // theta (1 - theta^2/6 + theta^4/120), theta^2/6 and theta^4/120 in units of 2^-84
        const int n = __clzll((long long)(low | 1ull << 24));  // 0 .. 39: low is a multiple of 2^24
        const uint64_t U = mulhi_64(low << n, half_pi);
        const uint64_t q = mulhi_64(s2, 0x2AAAAAAAAAAAAAABull) - ((uint64_t)__umulhi(__umulhi(s2h, s2h), 0x02222222u) << 12);
        sn = U - (mulhi_64(U, q) >> 20);
        sexp = 11 + n;
    }
    // x = -r cos(pi t), y = -r sin(pi t)
    const bool swap = ((quad & 1u) != 0u) != upper;  // x takes the sine
    const uint64_t X = mulhi_64(r, swap ? sn : cs), Y = mulhi_64(r, swap ? cs : sn);
    const int xe = rexp + (swap ? sexp : 0), ye = rexp + (swap ? 0 : sexp);  // units of 2^-(61 + xe), 2^-(61 + ye)
    const bool xneg = quad == 0u || quad == 3u, yneg = quad < 2u;
    t.x = fixed_to_double(X, 1024 - xe, xneg);
    t.y = fixed_to_double(Y, 1024 - ye, yneg);
    t.fx = (float)(uint32_t)(X >> 32) * __uint_as_float((uint32_t)(98 - xe) << 23);
    t.fy = (float)(uint32_t)(Y >> 32) * __uint_as_float((uint32_t)(98 - ye) << 23);
    t.fx = xneg ? -t.fx : t.fx;
    t.fy = yneg ? -t.fy : t.fy;
    return t;
}

// The Philox blocks of one site's FP64 trial: call 0 the orientation, call 1 the acceptance uniform.
__device__ __forceinline__ uint4 trial64_block(uint32_t site, uint32_t sweep, uint32_t colour, uint32_t call,
                                               uint32_t replica, uint32_t k0, uint32_t k1) {
    return philox10(make_uint4(site, sweep, (kTagTrial << 24) | (colour << 8) | call, replica), k0, k1);
}

// A double's value truncated to a float by its bit fields (the conversion
// instruction runs at the FP64 pipe's rate): within 2^-23 of its size for
// 2^-126 <= |v| < 2^128, smaller ones come out below 2^-125.  big collects the
// high word of the largest |v| seen, by which the caller knows the range held.
__device__ __forceinline__ float narrow(double v, int &big) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int u = hi & 0x7FFFFFFF;
    big = max(big, u);
    const uint32_t f = __funnelshift_l((uint32_t)lo, (uint32_t)max(u - 0x38000000, 0), 3);
    return __uint_as_float((f & 0x7FFFFFFFu) | ((uint32_t)hi & 0x80000000u));
}

// ---- FP32 arithmetic of one site (float) or of the two sites of a Philox
// pair (float2, packed sm_100+ instructions).  Every operation is rounded
// explicitly and identically in both forms, so a site's result never depends
// on whether it was processed alone or as a lane of a pair.
__device__ __forceinline__ float f_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float f_sub(float a, float b) { return __fadd_rn(a, -b); }
__device__ __forceinline__ float f_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 f_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f_sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 f_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

template <typename T> __device__ __forceinline__ T splat(float v);
template <> __device__ __forceinline__ float splat<float>(float v) { return v; }
template <> __device__ __forceinline__ float2 splat<float2>(float v) { return make_float2(v, v); }

// 2^x from the hardware base-2 exponential (relative error about 2^-22).
__device__ __forceinline__ float ex2_hw(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_l(float x) { return ex2_hw(x); }
__device__ __forceinline__ float2 ex2_l(float2 x) { return make_float2(ex2_hw(x.x), ex2_hw(x.y)); }
__device__ __forceinline__ float rsqrt_l(float x) { return rsqrtf(x); }
__device__ __forceinline__ float2 rsqrt_l(float2 x) { return make_float2(rsqrtf(x.x), rsqrtf(x.y)); }
__device__ __forceinline__ float pos_or_zero(float w, float r) { return w > 0.0f ? r : 0.0f; }
__device__ __forceinline__ float2 pos_or_zero(float2 w, float2 r) {
    return make_float2(w.x > 0.0f ? r.x : 0.0f, w.y > 0.0f ? r.y : 0.0f);
}
__device__ __forceinline__ void sincos_l(float a, float &s, float &c) { __sincosf(a, &s, &c); }
__device__ __forceinline__ void sincos_l(float2 a, float2 &s, float2 &c) {
    __sincosf(a.x, &s.x, &c.x);
    __sincosf(a.y, &s.y, &c.y);
}
__device__ __forceinline__ float half_round(float x) { return __half2float(__float2half_rn(x)); }
__device__ __forceinline__ float half_round_l(float x) { return half_round(x); }
// both lanes rounded to binary16 by one packed conversion (each lane rounded
// to nearest even, as the scalar form), then widened exactly
__device__ __forceinline__ float2 half_round_l(float2 x) { return __half22float2(__float22half2_rn(x)); }

// c + a for a binary16 a, with one rounding: the mixed-precision add widens a
// exactly, so the result equals f_add(c, (float)a) bit for bit.
__device__ __forceinline__ float add_half(float c, __half a) {
    float d;
    asm("add.rn.f32.f16 %0, %1, %2;" : "=f"(d) : "h"(__half_as_ushort(a)), "f"(c));
    return d;
}

// FP32 schedule: one Philox block serves two sites of the same colour.  The
// site of rank r within its colour class (ascending natural index) uses
// block r >> 1 and the half r & 1: words (a, b) = (x, y) or (z, w).
// u_z and u_phi are the top 21 bits of a and b, P the two low 11-bit fields
// (22 bits).
__device__ __forceinline__ uint4 trial_block(uint32_t rank_pair, uint32_t sweep, uint32_t colour, uint32_t replica,
                                             uint32_t k0, uint32_t k1) {
    return philox10(make_uint4(rank_pair, sweep, (kTagTrial << 24) | (colour << 8), replica), k0, k1);
}

// The three integers of one half (a, b): z index, azimuth index, P index.
__device__ __forceinline__ void half_ints(uint32_t a, uint32_t b, float &zi, float &vi, float &ui) {
    zi = (float)((int)(a >> 11) - (1 << 20));
    vi = (float)((int)(b >> 11) - (1 << 20));
    ui = (float)(((a & 0x7FFu) << 11) | (b & 0x7FFu));
}

// Trial orientation and acceptance uniform (Metropolis step (ii)) from the
// integers: z and v = 2u - 1 are exact, r = w / sqrt(w) with w = (1-z)(1+z)
// >= 0 from the hardware reciprocal square root, the azimuth pi v from the
// hardware sine / cosine on [-pi, pi) (absolute error about 4e-7, below what
// a 21-bit proposal resolves).  FP16 storage renormalises and rounds the trial
// to binary16; the rounded vector is the one tested and stored, so the chain
// samples the stored state.
template <int P, typename T>
__device__ __forceinline__ void trial32(T zi, T vi, T ui, T &tx, T &ty, T &tz, T &u) {
    tz = f_mul(zi, splat<T>(0x1p-20f));
    const T v = f_mul(vi, splat<T>(0x1p-20f));
    u = f_mul(ui, splat<T>(0x1p-22f));
    const T w2 = f_mul(f_sub(splat<T>(1.0f), tz), f_add(splat<T>(1.0f), tz));
    const T r = pos_or_zero(w2, f_mul(w2, rsqrt_l(w2)));
    T sn, cs;
    sincos_l(f_mul(splat<T>(3.14159265358979f), v), sn, cs);
    tx = f_mul(r, cs);
    ty = f_mul(r, sn);
    if constexpr (P == HS_FP16) {
        const T inv = rsqrt_l(f_fma(tz, tz, f_fma(ty, ty, f_mul(tx, tx))));
        tx = half_round_l(f_mul(tx, inv));
        ty = half_round_l(f_mul(ty, inv));
        tz = half_round_l(f_mul(tz, inv));
    }
}

// One site's trial, FP32 / FP16 schedule, from its rank in the colour class.
template <int P>
__device__ __forceinline__ void draw_trial_rank(uint32_t rank, uint32_t sweep, uint32_t colour, uint32_t replica,
                                                uint32_t k0, uint32_t k1, float &tx, float &ty, float &tz, float &u) {
    const uint4 w = trial_block(rank >> 1, sweep, colour, replica, k0, k1);
    float zi, vi, ui;
    if (rank & 1u)
        half_ints(w.z, w.w, zi, vi, ui);
    else
        half_ints(w.x, w.y, zi, vi, ui);
    trial32<P, float>(zi, vi, ui, tx, ty, tz, u);
}

// Metropolis step (iii), FP32 (one site or a pair of lanes): dH of Eq. 1
// restricted to the terms containing S_i, dH = J (S.h - S'.h) +
// K ((S.e)^2 - (S'.e)^2); the dot products are kept for the fused energy.
// Acceptance: dH <= 0 or P <= exp(-beta dH) = 2^(-beta log2(e) dH).
template <typename T>
struct Dots32 {
    T sh, th, se, pe, dH;
    T qs, qt;  // S^T A S and S'^T A S' (tensor term only)
};

// The on-site anisotropy tensor term S^T A S of a general symmetric A (the
// effective shape anisotropy the paper offers in place of dipolar coupling),
// A = (xx, yy, zz, xy, xz, yz): the product A S row by row, then its dot
// product with S.
template <typename T>
__device__ __forceinline__ T quad32(T x, T y, T z, const float (&A)[6]) {
    const T ax = f_fma(splat<T>(A[4]), z, f_fma(splat<T>(A[3]), y, f_mul(splat<T>(A[0]), x)));
    const T ay = f_fma(splat<T>(A[5]), z, f_fma(splat<T>(A[1]), y, f_mul(splat<T>(A[3]), x)));
    const T az = f_fma(splat<T>(A[2]), z, f_fma(splat<T>(A[5]), y, f_mul(splat<T>(A[4]), x)));
    return f_fma(z, az, f_fma(y, ay, f_mul(x, ax)));
}
__device__ __forceinline__ double quad64(double x, double y, double z, const double (&A)[6]) {
    const double ax = A[0] * x + A[3] * y + A[4] * z;
    const double ay = A[3] * x + A[1] * y + A[5] * z;
    const double az = A[4] * x + A[5] * y + A[2] * z;
    return x * ax + y * ay + z * az;
}

// TEN adds the tensor term: dH += S^T A S - S'^T A S'.  ZAX: the easy axis is
// e = (0, 0, 1) exactly, so S.e = S_z (what the three products give for it).
// KZ: K = +0, so the uniaxial term, +0 times a finite number, adds nothing
// (dH may differ only in the sign of a zero, which dH <= 0 does not see).
template <typename T, bool TEN = false, bool ZAX = false, bool KZ = false>
__device__ __forceinline__ Dots32<T> site_math32(T sx, T sy, T sz, T tx, T ty, T tz, T hx, T hy, T hz, float J,
                                                 float K, float ex, float ey, float ez, const float *A = nullptr) {
    Dots32<T> d;
    d.sh = f_fma(sz, hz, f_fma(sy, hy, f_mul(sx, hx)));
    d.th = f_fma(tz, hz, f_fma(ty, hy, f_mul(tx, hx)));
    if constexpr (ZAX) {
        d.se = sz;
        d.pe = tz;
    } else {
        d.se = f_fma(sz, splat<T>(ez), f_fma(sy, splat<T>(ey), f_mul(sx, splat<T>(ex))));
        d.pe = f_fma(tz, splat<T>(ez), f_fma(ty, splat<T>(ey), f_mul(tx, splat<T>(ex))));
    }
    if constexpr (KZ)
        d.dH = f_mul(splat<T>(J), f_sub(d.sh, d.th));
    else
        d.dH = f_fma(splat<T>(K), f_mul(f_sub(d.se, d.pe), f_add(d.se, d.pe)), f_mul(splat<T>(J), f_sub(d.sh, d.th)));
    if constexpr (TEN) {
        const float(&At)[6] = *reinterpret_cast<const float(*)[6]>(A);
        d.qs = quad32<T>(sx, sy, sz, At);
        d.qt = quad32<T>(tx, ty, tz, At);
        d.dH = f_add(d.dH, f_sub(d.qs, d.qt));
    }
    return d;
}

__device__ __forceinline__ bool accept32(float dH, float u, float neg_beta_log2e) {
    return (dH <= 0.0f) || (u <= ex2_hw(f_mul(neg_beta_log2e, dH)));
}

template <typename S, typename C> __device__ __forceinline__ S to_store(C v);
template <> __device__ __forceinline__ double to_store<double, double>(double v) { return v; }
template <> __device__ __forceinline__ float to_store<float, float>(float v) { return v; }
template <> __device__ __forceinline__ __half to_store<__half, float>(float v) { return __float2half_rn(v); }


// Metropolis step (iii) for one site in FP64: dH of Eq. 1 restricted to the
// terms that contain S_i, dH = J (S.h - S'.h) + K ((S.e)^2 - (S'.e)^2), then
// dH <= 0 or P <= exp(-beta dH).  The dot products are returned for the
// fused energy measurement.
template <typename C>
struct SiteDots {
    C sh, th, se, pe;
    C qs, qt;  // tensor term only
    bool acc;
};

// The FP64 acceptance P <= exp(x), x = -beta dH < 0, decided first in FP32:
// e = 2^(x log2(e)) from the hardware base-2 exponential has, for |x| <= 80,
// a relative error of at most 2^-22 (ex2) + 3 |x| 2^-24 (rounding x, log2(e)
// and their product to FP32) < 1.5e-5.  P lies in [uf, uf + 2^-24) (uf its
// top 24 bits, exact in FP32); the bounds e (1 -+ 3e-5), rounded to FP32, keep
// a margin over both errors, so outside that band the outcome of the FP64
// comparison is known.  Inside the band (or for |x| > 80) the FP64
// exponential decides, so the decision always equals the plain FP64 rule.
__device__ __forceinline__ bool accept64(double x, double u, float uf) {
    const float xf = (float)x;
    if (xf >= -80.0f) {
        const float y = __fmul_rn(xf, 1.44269504088896341f);
        float e;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(y));
        if (__fadd_rn(uf, 0x1p-24f) < __fmul_rn(e, 1.0f - 3e-5f)) return true;
        if (uf > __fmul_rn(e, 1.0f + 3e-5f)) return false;
    }
    return u <= exp(x);
}

// The FP64 decision from FP32 values of the spins and the field: x = -beta dH
// is off by at most a.fdelta (PassArgs), beside 2.4e-5 |x| / 80 from five FP32
// roundings and 2^-22 from the hardware 2^x, which the factors 1 -+ 4e-5 cover
// for |x| <= 80; below, P <= e^x < 2^-115 is decided by P's top 24 bits alone,
// and dH <= 0 (e^x >= 1 > P) is the same rule.  1 accepted, 0 rejected, -1
// within the bounds of each other: FP64 decides (1 to 4 sites of 10^5 at T from 0.7
// to 1.7, sc, bcc and fcc).
__device__ __forceinline__ int decide64(float x, float delta, float uf) {
    const float lo = ex2_hw(__fmul_rn(x - delta, 1.44269504088896341f));
    const float hi = ex2_hw(__fmul_rn(x + delta, 1.44269504088896341f));
    if (__fadd_rn(uf, 0x1p-24f) < __fmul_rn(lo, 1.0f - 4e-5f)) return 1;
    return uf > __fmul_rn(hi, 1.0f + 4e-5f) ? 0 : -1;
}

// ZAX: the easy axis is e = (0, 0, 1) exactly, so S.e = S_z (what the three
// products give for that e, without them).
template <typename C, bool TEN = false, bool ZAX = false>
__device__ __forceinline__ SiteDots<C> metropolis(C sx, C sy, C sz, C tx, C ty, C tz, C hx, C hy, C hz, C J, C K,
                                                  C ex, C ey, C ez, C beta, C u, float uf,
                                                  const double *A = nullptr) {
    SiteDots<C> d;
    d.sh = sx * hx + sy * hy + sz * hz;
    d.th = tx * hx + ty * hy + tz * hz;
    if constexpr (ZAX) {
        d.se = sz;
        d.pe = tz;
    } else {
        d.se = sx * ex + sy * ey + sz * ez;
        d.pe = tx * ex + ty * ey + tz * ez;
    }
    // the uniaxial term K ((S.e)^2 - (S'.e)^2): for e = z as S_z^2 - S'_z^2 with one
    // rounding of S'_z^2 (an fma), else as the product of difference and sum
    C dH;
    if constexpr (ZAX)
        dH = fma(K, fma(d.se, d.se, -(d.pe * d.pe)), J * (d.sh - d.th));
    else
        dH = J * (d.sh - d.th) + K * ((d.se - d.pe) * (d.se + d.pe));
    if constexpr (TEN) {
        const double(&At)[6] = *reinterpret_cast<const double(*)[6]>(A);
        d.qs = quad64(sx, sy, sz, At);
        d.qt = quad64(tx, ty, tz, At);
        dH += d.qs - d.qt;
    }
    d.acc = (dH <= C(0)) || accept64(-beta * dH, u, uf);
    return d;
}

__device__ __forceinline__ void load_params(const PassArgs &a, double &J, double &K, double &ex, double &ey,
                                            double &ez, double &beta) {
    J = a.J;
    K = a.K;
    ex = a.e[0];
    ey = a.e[1];
    ez = a.e[2];
    beta = a.beta;
}
__device__ __forceinline__ void load_params(const PassArgs &a, float &J, float &K, float &ex, float &ey, float &ez,
                                            float &beta) {
    J = a.fJ;
    K = a.fK;
    ex = a.fe[0];
    ey = a.fe[1];
    ez = a.fe[2];
    beta = a.fbeta;
}

// ----------------------------------------------------------------- reduction
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Totals of one ring slot (one sweep of a.n_colours passes, or a standalone
// measurement), executed by one whole CTA: every CTA's partials of every
// partial set not in a.skip_sets, summed in a fixed order (so the FP64
// totals do not depend on scheduling); the result is valid in thread 0.
// One warp per quantity: the FP64 pipe takes 16 cycles for a warp's addition,
// so the shuffle trees (5 additions each) are taken once per quantity and not
// once per warp and quantity (120 against 320 such additions for 608 CTAs'
// partials and 8 warps).
template <int NT = kBlock>
__device__ void slot_totals(const PassArgs &a, int slot, double (&tot)[kPartials]) {
    __shared__ double s_fin[kPartials];
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double *base = a.partials + (size_t)slot * a.n_colours * a.n_blocks * kPartials;
    for (int q = warp; q < kPartials; q += NW) {
        double t = 0.0;
        for (int p = 0; p < a.n_colours; ++p) {
            if ((a.skip_sets >> p) & 1ull) continue;
            const double *ps = base + (size_t)p * a.n_blocks * kPartials + q;
#pragma unroll 4
            for (int b = lane; b < a.n_blocks; b += 32) t += __ldcg(ps + (size_t)b * kPartials);
        }
        t = warp_sum(t);
        if (lane == 0) s_fin[q] = t;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPartials; ++q) tot[q] = s_fin[q];
}

// Eq. 2 with |S| = 1 from one sweep's totals: o = E, Mx, My, Mz, |M|, M2, M4,
// |M.e| with M = sum S / N.
__device__ __forceinline__ void sweep_observables(const double (&tot)[kPartials], double n_present,
                                                  const double (&e)[3], double (&o)[8]) {
    const double mx = tot[1] / n_present;
    const double my = tot[2] / n_present;
    const double mz = tot[3] / n_present;
    const double m2 = mx * mx + my * my + mz * mz;
    o[0] = tot[0];
    o[1] = mx;
    o[2] = my;
    o[3] = mz;
    o[4] = sqrt(m2);
    o[5] = m2;
    o[6] = m2 * m2;
    o[7] = fabs(mx * e[0] + my * e[1] + mz * e[2]);
}

// Apply one sweep to an accumulator (one thread): the accepted count, the raw
// sums and, when measured, the observables o of sweep_observables and their
// moments.  Acc is DevAccum in device memory or AccRegs, a register copy of
// its fields.
template <class Acc>
__device__ __forceinline__ void apply_sweep(Acc &A, const double (&tot)[kPartials], const double (&o)[8],
                                            bool measured, bool accumulate) {
    A.accepted += tot[4];
#pragma unroll
    for (int q = 0; q < kPartials; ++q) A.sums[q] = tot[q];
    if (!measured) return;
#pragma unroll
    for (int q = 0; q < 8; ++q) A.last[q] = o[q];
    if (accumulate) {
        A.moments[HS_SUM_E] += o[0];
        A.moments[HS_SUM_E2] += o[0] * o[0];
        A.moments[HS_SUM_ABSM] += o[4];
        A.moments[HS_SUM_M2] += o[5];
        A.moments[HS_SUM_M4] += o[6];
        A.moments[HS_SUM_MX] += o[1];
        A.moments[HS_SUM_MY] += o[2];
        A.moments[HS_SUM_MZ] += o[3];
        A.moments[HS_SUM_ABSME] += o[7];
        A.count += 1.0;
    }
}

// The fields of DevAccum that apply_sweep updates, held in registers while
// one thread applies many sweeps (one read and one write of device memory).
struct AccRegs {
    double moments[HS_N_MOMENTS];
    double count, accepted;
    double last[8];
    double sums[kPartials];
    __device__ __forceinline__ void load(const DevAccum *A) {
#pragma unroll
        for (int q = 0; q < HS_N_MOMENTS; ++q) moments[q] = A->moments[q];
        count = A->count;
        accepted = A->accepted;
#pragma unroll
        for (int q = 0; q < 8; ++q) last[q] = A->last[q];
#pragma unroll
        for (int q = 0; q < kPartials; ++q) sums[q] = A->sums[q];
    }
    __device__ __forceinline__ void store(DevAccum *A) const {
#pragma unroll
        for (int q = 0; q < HS_N_MOMENTS; ++q) A->moments[q] = moments[q];
        A->count = count;
        A->accepted = accepted;
#pragma unroll
        for (int q = 0; q < 8; ++q) A->last[q] = last[q];
#pragma unroll
        for (int q = 0; q < kPartials; ++q) A->sums[q] = sums[q];
    }
};

// Finalise a single colour pass sequence or a standalone measurement inside
// its last kernel: the last of its CTAs to arrive folds the slots.  Every
// earlier launch of the sequence ran on the same stream and has completed
// (griddepcontrol.wait at kernel entry), so only this launch's CTAs count.
template <int NT = kBlock>
__device__ void finish_reduction(const PassArgs &a, bool measured) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned ticket = atomicAdd(&a.acc->done, 1u);
        s_last = (ticket == gridDim.x - 1u);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double tot[kPartials];
    slot_totals<NT>(a, a.slot, tot);
    if (threadIdx.x == 0) {
        double o[8];
        sweep_observables(tot, a.n_present, a.e, o);
        apply_sweep(*a.acc, tot, o, measured, a.accumulate == 1);
        a.acc->done = 0u;
    }
}

// NT = threads of the CTA (a multiple of 32).
template <typename C, bool MEAS, int NT = kBlock>
__device__ __forceinline__ void write_partials(const PassArgs &a, C e, C x, C y, C z, unsigned nacc) {
    __shared__ double s_w[NT / 32][kPartials];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (MEAS) {
        e = warp_sum(e);
        x = warp_sum(x);
        y = warp_sum(y);
        z = warp_sum(z);
    }
    nacc = __reduce_add_sync(0xffffffffu, nacc);
    if (lane == 0) {
        s_w[warp][0] = MEAS ? (double)e : 0.0;
        s_w[warp][1] = MEAS ? (double)x : 0.0;
        s_w[warp][2] = MEAS ? (double)y : 0.0;
        s_w[warp][3] = MEAS ? (double)z : 0.0;
        s_w[warp][4] = (double)nacc;
    }
    __syncthreads();
    if (threadIdx.x < kPartials) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) s += s_w[w][threadIdx.x];
        a.partials[(((size_t)a.slot * a.n_colours + a.pass) * a.n_blocks + blockIdx.x) * kPartials + threadIdx.x] = s;
    }
    if (a.finish) finish_reduction<NT>(a, MEAS);
}

// ----------------------------------------------------------------- stencil pass
// One colour pass of the periodic sc lattice in colour-major SoA layout.
// Work item = V consecutive sites of one row of the updated colour.  Row
// parity p = (y+z+c)&1 fixes where the x neighbours sit in the other colour's
// row: p = 0 -> (xh-1, xh), p = 1 -> (xh, xh+1); the +-y and +-z neighbours
// sit at the same xh in the adjacent rows.  Neighbour order of the local
// field sum: -x, +x, -y, +y, -z, +z.

// Per-thread partial sums of the fused measurement (E, S) and accepted moves.
// FP32 / FP16 accumulate in float2 lanes (even / odd site of a pair).
template <int P>
struct SiteAcc {
    float2 e = make_float2(0.f, 0.f), x = make_float2(0.f, 0.f), y = make_float2(0.f, 0.f),
           z = make_float2(0.f, 0.f);
    unsigned n = 0;
    __device__ __forceinline__ float E(float, float) const { return e.x + e.y; }
    __device__ __forceinline__ float X() const { return x.x + x.y; }
    __device__ __forceinline__ float Y() const { return y.x + y.y; }
    __device__ __forceinline__ float Z() const { return z.x + z.y; }
};
// FP64: the energy as its two sums, scaled once by -K and -J at the end:
// k = sum (S.e)^2 over the sites, j = sum S.h over the later colour's sites,
// e = the tensor term's share.
template <>
struct SiteAcc<HS_FP64> {
    double e = 0.0, k = 0.0, j = 0.0, x = 0.0, y = 0.0, z = 0.0;
    unsigned n = 0;
    __device__ __forceinline__ double E(double J, double K) const { return e - J * j - K * k; }
    __device__ __forceinline__ double X() const { return x; }
    __device__ __forceinline__ double Y() const { return y; }
    __device__ __forceinline__ double Z() const { return z; }
};

// -beta log2(e), rounded once; every FP32 path uses this same value.
__device__ __forceinline__ float neg_beta_log2e(float beta) { return f_mul(-beta, 1.44269504088896341f); }

// Step (i) for the V sites of one work item: the local field h[q][k] of site
// k, the sum of its neighbours in the order -x, +x, -y, +y, -z, +z, from the
// other colour's same row o (+ the edge element ed beyond it; row parity p
// picks (xh-1, xh) or (xh, xh+1) for the x neighbours) and its rows at y-1,
// y+1, z-1, z+1.  FP32 / FP16 add two sites at a time as the lanes of float2
// (identical per lane to the scalar adds).
// FP32 / FP16 here; FP64 in item_fields64.
template <int P, int V>
__device__ __forceinline__ void item_fields(const Vec<typename Tr<P>::S, V> (&o)[3],
                                            const Vec<typename Tr<P>::S, V> (&nym)[3],
                                            const Vec<typename Tr<P>::S, V> (&nyp)[3],
                                            const Vec<typename Tr<P>::S, V> (&nzm)[3],
                                            const Vec<typename Tr<P>::S, V> (&nzp)[3], const typename Tr<P>::C (&ed)[3],
                                            uint32_t p, typename Tr<P>::C (&h)[3][V]) {
    using C = typename Tr<P>::C;
    auto xm_of = [&](int k, int q) -> C { return p ? to_c(o[q].v[k]) : (k == 0 ? ed[q] : to_c(o[q].v[k - 1])); };
    auto xp_of = [&](int k, int q) -> C { return p ? (k == V - 1 ? ed[q] : to_c(o[q].v[k + 1])) : to_c(o[q].v[k]); };
    if constexpr (P == HS_FP16) {
        // binary16 operands added straight into the FP32 sum (add_half: one
        // rounding per add, the same sums as widening each operand first)
#pragma unroll
        for (int k = 0; k < V; ++k)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                float t = xm_of(k, q);
                if (k == V - 1)
                    t = p ? f_add(t, ed[q]) : add_half(t, o[q].v[k]);
                else
                    t = add_half(t, p ? o[q].v[k + 1] : o[q].v[k]);
                t = add_half(t, nym[q].v[k]);
                t = add_half(t, nyp[q].v[k]);
                t = add_half(t, nzm[q].v[k]);
                h[q][k] = add_half(t, nzp[q].v[k]);
            }
    } else if constexpr (V >= 2) {
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            const int k0 = 2 * j, k1 = 2 * j + 1;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float2 xm = make_float2(xm_of(k0, q), xm_of(k1, q));
                const float2 xp = make_float2(xp_of(k0, q), xp_of(k1, q));
                const float2 ym = make_float2(to_c(nym[q].v[k0]), to_c(nym[q].v[k1]));
                const float2 yp = make_float2(to_c(nyp[q].v[k0]), to_c(nyp[q].v[k1]));
                const float2 zm = make_float2(to_c(nzm[q].v[k0]), to_c(nzm[q].v[k1]));
                const float2 zp = make_float2(to_c(nzp[q].v[k0]), to_c(nzp[q].v[k1]));
                const float2 hh = f_add(f_add(f_add(f_add(f_add(xm, xp), ym), yp), zm), zp);
                h[q][k0] = hh.x;
                h[q][k1] = hh.y;
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < 3; ++q)
            h[q][0] = f_add(f_add(f_add(f_add(f_add(xm_of(0, q), xp_of(0, q)), to_c(nym[q].v[0])), to_c(nyp[q].v[0])),
                                  to_c(nzm[q].v[0])),
                            to_c(nzp[q].v[0]));
    }
}

// FP64: the field the decision needs in FP32 (f), and where the energy needs
// it (wide: the later colour's fused measurement, or the tensor term) in FP64
// (d), its FP32 form taken from that.  The 15 FP64 additions a site cost as
// much issue time of their pipe as 480 integer instructions, so the narrow
// form converts every operand by its bit fields instead.  ok: every component
// the FP32 form was made from has a size of at most 1 + 2^-12 (unit vectors),
// which fdelta's error bound rests on.
template <int V>
struct Field64 {
    double d[3][V];
    float f[3][V];
    bool ok;
};

template <int V>
__device__ __forceinline__ void item_fields64(const Vec<double, V> (&o)[3], const Vec<double, V> (&nym)[3],
                                              const Vec<double, V> (&nyp)[3], const Vec<double, V> (&nzm)[3],
                                              const Vec<double, V> (&nzp)[3], const double (&ed)[3], uint32_t p,
                                              bool wide, Field64<V> &F) {
    int big = 0;
    if (wide) {
#pragma unroll
        for (int k = 0; k < V; ++k)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const double xm = p ? o[q].v[k] : (k == 0 ? ed[q] : o[q].v[k == 0 ? 0 : k - 1]);
                const double xp = p ? (k == V - 1 ? ed[q] : o[q].v[k == V - 1 ? 0 : k + 1]) : o[q].v[k];
                F.d[q][k] = ((((xm + xp) + nym[q].v[k]) + nyp[q].v[k]) + nzm[q].v[k]) + nzp[q].v[k];
                F.f[q][k] = narrow(F.d[q][k], big);
            }
        F.ok = big <= 0x40190000;  // 6.25
    } else {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            float x[V];  // the other colour's same row
#pragma unroll
            for (int k = 0; k < V; ++k) x[k] = narrow(o[q].v[k], big);
            const float e = narrow(ed[q], big);
#pragma unroll
            for (int k = 0; k < V; ++k) {
                // p: x neighbours (k, k + 1), else (k - 1, k); beyond the row's end the edge element
                const float other = p ? (k == V - 1 ? e : x[k == V - 1 ? 0 : k + 1]) : (k == 0 ? e : x[k == 0 ? 0 : k - 1]);
                float h = f_add(x[k], other);
                h = f_add(h, narrow(nym[q].v[k], big));
                h = f_add(h, narrow(nyp[q].v[k], big));
                h = f_add(h, narrow(nzm[q].v[k], big));
                F.f[q][k] = f_add(h, narrow(nzp[q].v[k], big));
            }
        }
        F.ok = big <= 0x3FF00100;  // 1 + 2^-12
    }
}

// The trials and acceptance uniforms of a work item's V sites, for a kernel
// that draws them ahead of the item's loads (they need no spin).
template <int P, int V>
struct Trials {
    float x[V], y[V], z[V], u[V];
};
template <int V>
struct Trials<HS_FP64, V> {
    Trial64 t[V];
    uint32_t px[V], py[V];  // the acceptance uniform's words
};

template <int P, int V>
__device__ __forceinline__ void draw_trials(const PassArgs &a, int c, uint32_t site0, uint32_t rank0, Trials<P, V> &d) {
    if constexpr (P == HS_FP64) {
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const uint32_t site = site0 + 2u * k;
            d.t[k] = trial64(trial64_block(site, a.sweep, (uint32_t)c, 0u, a.replica, a.key0, a.key1), a.sc_tab);
            const uint4 w = trial64_block(site, a.sweep, (uint32_t)c, 1u, a.replica, a.key0, a.key1);
            d.px[k] = w.x;
            d.py[k] = w.y;
        }
    } else if constexpr (V >= 2) {  // rank0 is even: rows hold a multiple of V sites
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            const uint4 w = trial_block((rank0 >> 1) + j, a.sweep, (uint32_t)c, a.replica, a.key0, a.key1);
            float2 zi, vi, ui, x, y, z, u;
            half_ints(w.x, w.y, zi.x, vi.x, ui.x);
            half_ints(w.z, w.w, zi.y, vi.y, ui.y);
            trial32<P, float2>(zi, vi, ui, x, y, z, u);
            d.x[2 * j] = x.x, d.x[2 * j + 1] = x.y;
            d.y[2 * j] = y.x, d.y[2 * j + 1] = y.y;
            d.z[2 * j] = z.x, d.z[2 * j + 1] = z.y;
            d.u[2 * j] = u.x, d.u[2 * j + 1] = u.y;
        }
    } else {
        draw_trial_rank<P>(rank0, a.sweep, (uint32_t)c, a.replica, a.key0, a.key1, d.x[0], d.y[0], d.z[0], d.u[0]);
    }
}

// Where a work item's operands lie, for the few sites whose FP32 decision is
// open: the other colour's planes and the item's first element.
struct ItemSource {
    const double *o[3];
    uint32_t b0;
};

// One component of a site's FP64 field, read again from the other colour's
// plane o (which no pass of this colour writes); b = the site's element.
template <bool CG>
__device__ __noinline__ double stencil_field64(const double *o, uint32_t b, uint32_t Lh, uint32_t Ly, uint32_t Lz,
                                               uint32_t par) {
    const uint32_t row = b / Lh, x = b - row * Lh, z = row / Ly, y = row - z * Ly;
    const uint32_t p = (y + z + par) & 1u;
    auto at = [&](uint32_t zz, uint32_t yy, uint32_t xx) {
        const double *q = o + ((size_t)zz * Ly + yy) * Lh + xx;
        if constexpr (CG)
            return __ldcg(q);
        else
            return *q;
    };
    double h = at(z, y, p ? x : (x == 0 ? Lh - 1 : x - 1));
    h += at(z, y, p ? (x == Lh - 1 ? 0 : x + 1) : x);
    h += at(z, y == 0 ? Ly - 1 : y - 1, x);
    h += at(z, y == Ly - 1 ? 0 : y + 1, x);
    h += at(z == 0 ? Lz - 1 : z - 1, y, x);
    h += at(z == Lz - 1 ? 0 : z + 1, y, x);
    return h;
}

// The plain FP64 rule, for a decision that FP32 left open.
template <bool ZAX>
__device__ __noinline__ bool accept_wide(double sx, double sy, double sz, double tx, double ty, double tz, double hx,
                                         double hy, double hz, double J, double K, double ex, double ey, double ez,
                                         double beta, double u, float uf) {
    return metropolis<double, false, ZAX>(sx, sy, sz, tx, ty, tz, hx, hy, hz, J, K, ex, ey, ez, beta, u, uf).acc;
}

// Metropolis steps (ii)-(iii) for the V sites of one FP64 work item (see
// update_item_h); ZAX as in metropolis.  Spins, trials and sums are FP64; the
// decision is the FP64 rule's, taken from FP32 values wherever their error
// bound settles it (decide64).
template <int V, bool MEAS, bool TEN, bool ZAX, bool CG, bool PRE>
__device__ __forceinline__ bool update_fp64(Vec<double, V> (&s)[3], const Field64<V> &F, uint32_t site0, int c,
                                            const PassArgs &a, double J, double K, double ex, double ey, double ez,
                                            double beta, SiteAcc<HS_FP64> &acc, const ItemSource &src,
                                            const Trials<HS_FP64, V> *pre) {
    bool any = false;
#pragma unroll
    for (int k = 0; k < V; ++k) {
        Trial64 t;
        uint2 pw;
        if constexpr (PRE) {
            t = pre->t[k];
            pw = make_uint2(pre->px[k], pre->py[k]);
        } else {
            const uint32_t site = site0 + 2u * k;
            t = trial64(trial64_block(site, a.sweep, (uint32_t)c, 0u, a.replica, a.key0, a.key1), a.sc_tab);
            const uint4 w = trial64_block(site, a.sweep, (uint32_t)c, 1u, a.replica, a.key0, a.key1);
            pw = make_uint2(w.x, w.y);
        }
        const float uf = (float)(pw.x >> 8) * 0x1p-24f;  // P's top 24 bits
        double sx = s[0].v[k], sy = s[1].v[k], sz = s[2].v[k];
        bool ac;
        if constexpr (TEN) {
            const double u = (double)bits53(pw.x, pw.y) * 0x1p-53;
            ac = metropolis<double, true, ZAX>(sx, sy, sz, t.x, t.y, t.z, F.d[0][k], F.d[1][k], F.d[2][k], J, K, ex, ey,
                                               ez, beta, u, uf, a.A)
                     .acc;
        } else {
            int big = 0;
            const float fx = narrow(sx, big), fy = narrow(sy, big), fz = narrow(sz, big);
            const Dots32<float> d =
                site_math32<float, false, ZAX>(fx, fy, fz, t.fx, t.fy, t.fz, F.f[0][k], F.f[1][k], F.f[2][k], a.fJ,
                                               a.fK, a.fe[0], a.fe[1], a.fe[2]);
            int dec = decide64(-a.fbeta * d.dH, a.fdelta, uf);
            if (!F.ok || big > 0x3FF00100) dec = -1;
            if (dec < 0) {
                double h[3];
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    h[q] = stencil_field64<CG>(src.o[q], src.b0 + k, (uint32_t)a.Lh, (uint32_t)a.Ly, (uint32_t)a.Lz,
                                               (uint32_t)(a.colour + a.zpar));
                dec = accept_wide<ZAX>(sx, sy, sz, t.x, t.y, t.z, h[0], h[1], h[2], J, K, ex, ey, ez, beta,
                                       (double)bits53(pw.x, pw.y) * 0x1p-53, uf);
            }
            ac = dec > 0;
        }
        if (ac) {
            s[0].v[k] = sx = t.x;
            s[1].v[k] = sy = t.y;
            s[2].v[k] = sz = t.z;
            any = true;
            ++acc.n;
        }
        if (MEAS) {
            // bond energy counted at the later colour's end: pass 1 owns
            // every sc bond, pass 0 only the anisotropy term
            const double se = ZAX ? sz : sx * ex + sy * ey + sz * ez;
            acc.k = fma(se, se, acc.k);
            if (TEN) acc.e -= quad64(sx, sy, sz, a.A);
            if (c == 1) acc.j = fma(sz, F.d[2][k], fma(sy, F.d[1][k], fma(sx, F.d[0][k], acc.j)));
            acc.x += sx;
            acc.y += sy;
            acc.z += sz;
        }
    }
    return any;
}

// Metropolis steps (ii)-(iii) for the V sites of one work item, given the
// item's own spins s and the local fields h of step (i).  site0 is the
// natural index of the item's first site (the FP64 schedule's counter), rank0
// its rank within its colour class (the FP32 / FP16 schedule's; on a periodic
// sc lattice the natural index halved, kept separately so that it stays exact
// beyond 2^32 sites).  Updates s in place; returns whether any site was
// accepted.
// Metropolis steps (ii)-(iii) for the V sites of one FP32 / FP16 work item
// (see update_item_h); ZAX as in site_math32.
// KZ (with ZAX): K = +0, whose energy share -K (S.e)^2 is -0 (written as such,
// so every sum takes the same values; adding -0 changes none).
template <int P, int V, bool MEAS, bool TEN, bool ZAX, bool KZ = false, bool PRE = false>
__device__ __forceinline__ bool update_f32(Vec<typename Tr<P>::S, V> (&s)[3], const float (&h)[3][V], uint32_t rank0,
                                           int c, const PassArgs &a, float J, float K, float ex, float ey, float ez,
                                           float beta, SiteAcc<P> &acc, const Trials<P, V> *pre = nullptr) {
    using S = typename Tr<P>::S;
    using C = float;
    bool any = false;
    const float nb = neg_beta_log2e(beta);
    // one site in lane x of the accumulators
    auto single = [&](int k, float tx, float ty, float tz, float u) {
        const float sx = to_c(s[0].v[k]), sy = to_c(s[1].v[k]), sz = to_c(s[2].v[k]);
        const Dots32<float> d = site_math32<float, TEN, ZAX, KZ>(sx, sy, sz, tx, ty, tz, h[0][k], h[1][k], h[2][k], J, K,
                                                        ex, ey, ez, a.fA);
        const bool ac = accept32(d.dH, u, nb);
        if (ac) {
            s[0].v[k] = to_store<S, C>(tx);
            s[1].v[k] = to_store<S, C>(ty);
            s[2].v[k] = to_store<S, C>(tz);
            any = true;
            ++acc.n;
        }
        if (MEAS) {
            const float en = ac ? d.pe : d.se;
            float ei = KZ ? -0.0f : f_mul(-K, f_mul(en, en));
            if (TEN) ei = f_sub(ei, ac ? d.qt : d.qs);
            if (c == 1) ei = f_fma(-J, ac ? d.th : d.sh, ei);
            acc.e.x = f_add(acc.e.x, ei);
            acc.x.x = f_add(acc.x.x, ac ? tx : sx);
            acc.y.x = f_add(acc.y.x, ac ? ty : sy);
            acc.z.x = f_add(acc.z.x, ac ? tz : sz);
        }
    };
    // ranks of the item's sites in their colour class: rank0 + k
    if (V >= 2 && (PRE || (rank0 & 1u) == 0u)) {
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {  // one Philox block and packed arithmetic per pair
            const int k0 = 2 * j, k1 = 2 * j + 1;
            float2 tx, ty, tz, u;
            if constexpr (PRE) {
                tx = make_float2(pre->x[k0], pre->x[k1]);
                ty = make_float2(pre->y[k0], pre->y[k1]);
                tz = make_float2(pre->z[k0], pre->z[k1]);
                u = make_float2(pre->u[k0], pre->u[k1]);
            } else {
                const uint4 w = trial_block((rank0 >> 1) + j, a.sweep, (uint32_t)c, a.replica, a.key0, a.key1);
                float2 zi, vi, ui;
                half_ints(w.x, w.y, zi.x, vi.x, ui.x);
                half_ints(w.z, w.w, zi.y, vi.y, ui.y);
                trial32<P, float2>(zi, vi, ui, tx, ty, tz, u);
            }
            float2 hp[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) hp[q] = make_float2(h[q][k0], h[q][k1]);
            const float2 sx = make_float2(to_c(s[0].v[k0]), to_c(s[0].v[k1]));
            const float2 sy = make_float2(to_c(s[1].v[k0]), to_c(s[1].v[k1]));
            const float2 sz = make_float2(to_c(s[2].v[k0]), to_c(s[2].v[k1]));
            const Dots32<float2> d =
                site_math32<float2, TEN, ZAX, KZ>(sx, sy, sz, tx, ty, tz, hp[0], hp[1], hp[2], J, K, ex, ey, ez, a.fA);
            const bool a0 = accept32(d.dH.x, u.x, nb);
            const bool a1 = accept32(d.dH.y, u.y, nb);
            if (a0) {
                s[0].v[k0] = to_store<S, C>(tx.x);
                s[1].v[k0] = to_store<S, C>(ty.x);
                s[2].v[k0] = to_store<S, C>(tz.x);
                ++acc.n;
            }
            if (a1) {
                s[0].v[k1] = to_store<S, C>(tx.y);
                s[1].v[k1] = to_store<S, C>(ty.y);
                s[2].v[k1] = to_store<S, C>(tz.y);
                ++acc.n;
            }
            any = any || a0 || a1;
            if (MEAS) {
                const float2 en = make_float2(a0 ? d.pe.x : d.se.x, a1 ? d.pe.y : d.se.y);
                float2 ei = KZ ? make_float2(-0.0f, -0.0f) : f_mul(splat<float2>(-K), f_mul(en, en));
                if (TEN) ei = f_sub(ei, make_float2(a0 ? d.qt.x : d.qs.x, a1 ? d.qt.y : d.qs.y));
                if (c == 1)
                    ei = f_fma(splat<float2>(-J), make_float2(a0 ? d.th.x : d.sh.x, a1 ? d.th.y : d.sh.y), ei);
                acc.e = f_add(acc.e, ei);
                acc.x = f_add(acc.x, make_float2(a0 ? tx.x : sx.x, a1 ? tx.y : sx.y));
                acc.y = f_add(acc.y, make_float2(a0 ? ty.x : sy.x, a1 ? ty.y : sy.y));
                acc.z = f_add(acc.z, make_float2(a0 ? tz.x : sz.x, a1 ? tz.y : sz.y));
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < V; ++k) {
            float tx, ty, tz, u;
            if constexpr (PRE) {
                tx = pre->x[k], ty = pre->y[k], tz = pre->z[k], u = pre->u[k];
            } else {
                draw_trial_rank<P>(rank0 + k, a.sweep, (uint32_t)c, a.replica, a.key0, a.key1, tx, ty, tz, u);
            }
            single(k, tx, ty, tz, u);
        }
    }
    return any;
}

// A work item's local fields as its precision keeps them.
template <int P, int V>
struct ItemField {
    using T = typename Tr<P>::C[3][V];
};
template <int V>
struct ItemField<HS_FP64, V> {
    using T = Field64<V>;
};

// Step (i) of a work item from its raw operands.
template <int P, int V, bool MEAS, bool TEN>
__device__ __forceinline__ void fields_of(const Vec<typename Tr<P>::S, V> (&o)[3],
                                          const Vec<typename Tr<P>::S, V> (&nym)[3],
                                          const Vec<typename Tr<P>::S, V> (&nyp)[3],
                                          const Vec<typename Tr<P>::S, V> (&nzm)[3],
                                          const Vec<typename Tr<P>::S, V> (&nzp)[3], const typename Tr<P>::C (&ed)[3],
                                          uint32_t p, int c, typename ItemField<P, V>::T &h) {
    if constexpr (P == HS_FP64)
        item_fields64<V>(o, nym, nyp, nzm, nzp, ed, p, TEN || (MEAS && c == 1), h);
    else
        item_fields<P, V>(o, nym, nyp, nzm, nzp, ed, p, h);
}

// AX = 1: the kernel was chosen for e = (0, 0, 1) at launch, so S.e = S_z
// with no branch (the FP32 register stencil's form); AX = 2: the same with
// K = +0 (the FP32 and FP16 batch kernels); AX = 0: FP64 and FP16 decide per
// work item from PassArgs::zaxis, FP32 takes the general products.
// oth, b0: where the item's neighbours lie (FP64 only, which may read them again; CG as in ld_val).  PRE: the
// trials are drawn already (pre).
template <int P, int V, bool MEAS, bool TEN = false, int AX = 0, bool CG = false, bool PRE = false>
__device__ __forceinline__ bool update_item_h(Vec<typename Tr<P>::S, V> (&s)[3],
                                              const typename ItemField<P, V>::T &h, uint32_t site0, uint32_t rank0,
                                              int c, const PassArgs &a, typename Tr<P>::C J, typename Tr<P>::C K,
                                              typename Tr<P>::C ex, typename Tr<P>::C ey, typename Tr<P>::C ez,
                                              typename Tr<P>::C beta, SiteAcc<P> &acc,
                                              const typename Tr<P>::S *const *oth = nullptr, uint32_t b0 = 0,
                                              const Trials<P, V> *pre = nullptr) {
    if constexpr (P == HS_FP64) {
        // one uniform branch per work item: the item body with S.e = S_z
        // (e = (0, 0, 1)) or with the general dot products
        const ItemSource src{{oth[0], oth[1], oth[2]}, b0};
        if constexpr (!TEN)
            if (a.zaxis)
                return update_fp64<V, MEAS, false, true, CG, PRE>(s, h, site0, c, a, J, K, ex, ey, ez, beta, acc, src,
                                                                  pre);
        return update_fp64<V, MEAS, TEN, false, CG, PRE>(s, h, site0, c, a, J, K, ex, ey, ez, beta, acc, src, pre);
    } else {
        if constexpr (AX >= 1 && !TEN)
            return update_f32<P, V, MEAS, false, true, AX == 2, PRE>(s, h, rank0, c, a, J, K, ex, ey, ez, beta, acc,
                                                                     pre);
        // FP16 (bound by instruction issue, its loads decoupled by the
        // pipelined landing slots) takes the same branch; the FP32 register
        // stencil, bound by load latency, measured slower with it (the branch
        // between an item's loads and its arithmetic costs more than the three
        // instructions per site it saves) and keeps the general products
        if constexpr (!TEN && P == HS_FP16)
            if (a.zaxis)
                return update_f32<P, V, MEAS, false, true, false, PRE>(s, h, rank0, c, a, J, K, ex, ey, ez, beta, acc, pre);
        return update_f32<P, V, MEAS, TEN, false, false, PRE>(s, h, rank0, c, a, J, K, ex, ey, ez, beta, acc, pre);
    }
}

// The same from the raw operands: step (i) then steps (ii)-(iii).  EARLY: the
// trials, which need no operand, are drawn first, so that they hide the loads'
// latency (at the price of the registers that hold them: faster in the FP16
// stencil, 464^3 600.1 -> 561.7 us per sweep, the FP32 streaming batches, 64
// replicas 136.5 -> 131.2, and the resident ones, 152 of 24^3 14.1 -> 13.1; slower
// in the FP32 stencil, 256^3 102.5 -> 107.7, the FP16 pipelined one, 96.2 -> 98.6,
// and the FP16 streaming batches, 134.9 -> 137.1).
template <int P, int V, bool MEAS, bool TEN = false, int AX = 0, bool CG = false, bool EARLY = false>
__device__ __forceinline__ bool update_item(Vec<typename Tr<P>::S, V> (&s)[3], const Vec<typename Tr<P>::S, V> (&o)[3],
                                            const Vec<typename Tr<P>::S, V> (&nym)[3],
                                            const Vec<typename Tr<P>::S, V> (&nyp)[3],
                                            const Vec<typename Tr<P>::S, V> (&nzm)[3],
                                            const Vec<typename Tr<P>::S, V> (&nzp)[3], const typename Tr<P>::C (&ed)[3],
                                            uint32_t p, uint32_t site0, uint32_t rank0, int c, const PassArgs &a,
                                            typename Tr<P>::C J, typename Tr<P>::C K, typename Tr<P>::C ex,
                                            typename Tr<P>::C ey, typename Tr<P>::C ez, typename Tr<P>::C beta,
                                            SiteAcc<P> &acc, const typename Tr<P>::S *const *oth = nullptr,
                                            uint32_t b0 = 0) {
    if constexpr (EARLY) {
        Trials<P, V> pre;
        draw_trials<P, V>(a, c, site0, rank0, pre);
        typename ItemField<P, V>::T h;
        fields_of<P, V, MEAS, TEN>(o, nym, nyp, nzm, nzp, ed, p, c, h);
        return update_item_h<P, V, MEAS, TEN, AX, CG, true>(s, h, site0, rank0, c, a, J, K, ex, ey, ez, beta, acc, oth,
                                                            b0, &pre);
    }
    typename ItemField<P, V>::T h;
    fields_of<P, V, MEAS, TEN>(o, nym, nyp, nzm, nzp, ed, p, c, h);
    return update_item_h<P, V, MEAS, TEN, AX, CG>(s, h, site0, rank0, c, a, J, K, ex, ey, ez, beta, acc, oth, b0);
}

// Vector load, optionally L2-only (ld.global.cg).  A kernel that reads data
// other CTAs wrote earlier in the same launch must not be served from a
// stale line of its SM's L1 (L1 is not coherent across SMs).
template <typename T, bool CG>
__device__ __forceinline__ T ld_val(const T *p) {
    if constexpr (!CG) {
        return *p;
    } else {
        T out;
        if constexpr (sizeof(T) == 16) {
            const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(p));
            memcpy(&out, &v, 16);
        } else if constexpr (sizeof(T) == 8) {
            const uint2 v = __ldcg(reinterpret_cast<const uint2 *>(p));
            memcpy(&out, &v, 8);
        } else if constexpr (sizeof(T) == 4) {
            const unsigned int v = __ldcg(reinterpret_cast<const unsigned int *>(p));
            memcpy(&out, &v, 4);
        } else {
            const unsigned short v = __ldcg(reinterpret_cast<const unsigned short *>(p));
            memcpy(&out, &v, 2);
        }
        return out;
    }
}

// Operands of one work item of the register stencil.
template <int P, int V>
struct StencilItem {
    Vec<typename Tr<P>::S, V> s[3], o[3], nym[3], nyp[3], nzm[3], nzp[3];
    typename Tr<P>::C ed[3];
    uint32_t b0, p, site0, rank0;
};

// Element offsets (within a colour plane) of the operands of the work item at
// row (y, z), vector xv: the own vector b0 (and the other colour's same-row
// vector at the same offset), the other colour's rows at y-1, y+1, z-1, z+1,
// and the edge element beyond the row vector on the side parity p picks.
struct ItemOffsets {
    uint32_t b0, bym, byp, bzm, bzp, bed, p, site0, rank0;
};

template <int V>
__device__ __forceinline__ ItemOffsets item_offsets(const PassArgs &a, uint32_t y, uint32_t z, uint32_t xv) {
    const uint32_t Lh = a.Lh, Ly = a.Ly, Lz = a.Lz, Lx = a.Lx;
    const uint32_t row = z * Ly + y;
    const uint32_t xh0 = xv * V;
    const uint32_t ym = (y == 0) ? Ly - 1 : y - 1;
    const uint32_t yp = (y == Ly - 1) ? 0 : y + 1;
    const uint32_t zm = (z == 0) ? Lz - 1 : z - 1;
    const uint32_t zp = (z == Lz - 1) ? 0 : z + 1;
    ItemOffsets o;
    o.p = (y + z + (uint32_t)a.colour + (uint32_t)a.zpar) & 1u;
    o.b0 = row * Lh + xh0;
    o.bym = (z * Ly + ym) * Lh + xh0;
    o.byp = (z * Ly + yp) * Lh + xh0;
    o.bzm = (zm * Ly + y) * Lh + xh0;
    o.bzp = (zp * Ly + y) * Lh + xh0;
    o.bed = row * Lh + (o.p ? ((xh0 + V == Lh) ? 0 : xh0 + V) : ((xh0 == 0) ? Lh - 1 : xh0 - 1));
    o.site0 = row * Lx + 2 * xh0 + o.p + a.site_off;
    o.rank0 = row * Lh + xh0 + a.rank_off;  // (row Lx + 2 xh0 + p) / 2 + the slab's offset
    return o;
}

// Load a work item's operands from their offsets.
template <int P, int V, bool CG = false>
__device__ __forceinline__ void load_item_from(const ItemOffsets &f, const typename Tr<P>::S *const (&own)[3],
                                               const typename Tr<P>::S *const (&oth)[3], StencilItem<P, V> &it) {
    using S = typename Tr<P>::S;
    using VT = Vec<S, V>;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        it.s[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(own[q] + f.b0));
        it.o[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + f.b0));
        it.nym[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + f.bym));
        it.nyp[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + f.byp));
        it.nzm[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + f.bzm));
        it.nzp[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + f.bzp));
        it.ed[q] = to_c(ld_val<S, CG>(oth[q] + f.bed));
    }
    it.b0 = f.b0;
    it.p = f.p;
    it.site0 = f.site0;
    it.rank0 = f.rank0;
}

// Load the operands of the work item at row (y, z), vector xv.
template <int P, int V, bool CG = false>
__device__ __forceinline__ void load_item_at(const PassArgs &a, uint32_t y, uint32_t z, uint32_t xv,
                                             const typename Tr<P>::S *const (&own)[3],
                                             const typename Tr<P>::S *const (&oth)[3], StencilItem<P, V> &it) {
    load_item_from<P, V, CG>(item_offsets<V>(a, y, z, xv), own, oth, it);
}

// The work item with linear index t = (z Ly + y) (Lh/V) + xv (rev - t in a
// descending pass; DIR = false: always ascending, with no reference to rev).
template <int P, int V, bool CG = false, bool DIR = true>
__device__ __forceinline__ void load_item(const PassArgs &a, uint32_t t, const typename Tr<P>::S *const (&own)[3],
                                          const typename Tr<P>::S *const (&oth)[3], StencilItem<P, V> &it) {
    if constexpr (DIR) t = a.rev ? a.rev - t : t;  // a descending pass
    const uint32_t nxv = a.Lh / V;
    const uint32_t r = a.div_nxv.div(t);
    const uint32_t xv = t - r * nxv;
    const uint32_t row = r + (uint32_t)(a.z_off * a.Ly);  // a z-slab's own rows start after its halo plane
    const uint32_t z = a.div_ly.div(row);
    const uint32_t y = row - z * a.Ly;
    load_item_at<P, V, CG>(a, y, z, xv, own, oth, it);
}

// Split loading of the work item with linear index t (see the split
// prefetch of the stencil kernels): part A -- the own row, the other colour's
// same row (+ edge element) and its rows at z-1 and z+1 -- is loaded ahead;
// part B -- the rows at y-1 and y+1 -- when the item is taken up.
template <int P, int V>
struct SplitItem {
    Vec<typename Tr<P>::S, V> s[3], o[3], nzm[3], nzp[3];
    typename Tr<P>::C ed[3];
    ItemOffsets f;
};

template <int P, int V, bool CG = false, bool DIR = true>
__device__ __forceinline__ void load_split_a(const PassArgs &a, uint32_t t, const typename Tr<P>::S *const (&own)[3],
                                             const typename Tr<P>::S *const (&oth)[3], SplitItem<P, V> &A) {
    using S = typename Tr<P>::S;
    using VT = Vec<S, V>;
    if constexpr (DIR) t = a.rev ? a.rev - t : t;  // a descending pass
    const uint32_t nxv = a.Lh / V;
    const uint32_t r = a.div_nxv.div(t);
    const uint32_t xv = t - r * nxv;
    const uint32_t row = r + (uint32_t)(a.z_off * a.Ly);
    const uint32_t z = a.div_ly.div(row);
    A.f = item_offsets<V>(a, row - z * a.Ly, z, xv);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        A.s[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(own[q] + A.f.b0));
        A.o[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + A.f.b0));
        A.nzm[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + A.f.bzm));
        A.nzp[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + A.f.bzp));
        A.ed[q] = to_c(ld_val<S, CG>(oth[q] + A.f.bed));
    }
}

template <int P, int V, bool CG = false>
__device__ __forceinline__ void load_split_b(const SplitItem<P, V> &A, const typename Tr<P>::S *const (&oth)[3],
                                             Vec<typename Tr<P>::S, V> (&nym)[3], Vec<typename Tr<P>::S, V> (&nyp)[3]) {
    using VT = Vec<typename Tr<P>::S, V>;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        nym[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + A.f.bym));
        nyp[q] = ld_val<VT, CG>(reinterpret_cast<const VT *>(oth[q] + A.f.byp));
    }
}

}  // namespace
}  // namespace hs
