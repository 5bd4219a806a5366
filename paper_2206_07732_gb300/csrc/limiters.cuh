// Limiters and helpers of the step's stencils, for the 2D and the 3D tank, in their
// working types R: double, float, or float pairs (df64).
#pragma once

#include <type_traits>

#include "df64.cuh"

namespace wec {
namespace {

template <typename R>
constexpr bool is_f64 = std::is_same<R, double>::value;
template <typename R>
constexpr bool is_df = std::is_same<R, df64>::value;
// v of lane + 1 of the warp (every lane taking part)
template <typename R>
__device__ __forceinline__ R shfl_down1(R v)
{
    if constexpr (is_df<R>)
        return R(__shfl_down_sync(0xffffffffu, v.hi, 1), __shfl_down_sync(0xffffffffu, v.lo, 1));
    else
        return __shfl_down_sync(0xffffffffu, v, 1);
}
// Whether the whole warp (every lane taking part) may read its stencils at fixed
// offsets: inside of every lane that has a face to form (use).  A warp at a row's end
// then runs the clamped form for all its lanes, where the choice by lane ran both
// forms one after the other -- two of a row's warps, and these kernels are bound by
// their arithmetic: 3D FP64 at 256x128x128, a Jacobi sweep of one component went from
// 152 to 131 us and the three momentum systems from 4.70 to 4.01 ms.  The two forms give the
// same values wherever both apply.
__device__ __forceinline__ bool warp_inside(bool inside, bool use) { return __all_sync(0xffffffffu, inside || !use); }
// k x for k a power of two (2 or 1/2 here): exact; for a float pair, both
// floats scaled (the value of the full pair product, in two multiplications)
template <typename R>
__device__ __forceinline__ R scl2(float k, R x)
{
    if constexpr (is_df<R>) return R(k * x.hi, k * x.lo); else return R(k) * x;
}

// Sign and magnitude decisions of the FP64 stencils on the integer pipe: for
// finite doubles the bit pattern orders magnitudes (sign bit shifted out) and
// carries the sign, and this GPU issues FP64 compares, min / max and products
// at 1/64 of its FP32 rate.  Choices, zero tests and sign changes go word by word:
// written on doubles the compiler made the zero tests FP64 compares and the choices
// branches.  Counted per warp in FP64 instructions: upw3 7 -> 5, one direction of the
// ENO-2 / Godunov term 18 -> 9, the PPM face value 49 -> 36; at 256x128x128 a 3D
// reinitialisation stage went from 717 to 440 us, the advection's face values from 1.42
// to 0.97 ms, the momentum systems from 4.01 to 3.09.  The FP32 stencils keep plain
// float compares.
__device__ __forceinline__ unsigned long long mag_bits(double a)
{
    return (unsigned long long)__double_as_longlong(a) << 1;
}
// p ? a : b.  FP64: word by word, so that the choice stays a choice (as a branch, the
// arithmetic on its result was done once per side in every warp that saw both)
template <typename R>
__device__ __forceinline__ R sel(bool p, R a, R b)
{
    if constexpr (is_f64<R>)
        return __hiloint2double(p ? __double2hiint(a) : __double2hiint(b), p ? __double2loint(a) : __double2loint(b));
    else
        return p ? a : b;
}
// a * b <= 0 (opposite signs, or a zero factor; FP64: tested on the two words -- on
// the 64-bit pattern the compiler makes it an FP64 compare with zero)
template <typename R>
__device__ __forceinline__ bool nonpos_prod(R a, R b)
{
    if constexpr (is_f64<R>) {
        const int ah = __double2hiint(a), bh = __double2hiint(b);
        return (ah ^ bh) < 0 || ((ah & 0x7fffffff) | __double2loint(a)) == 0 ||
               ((bh & 0x7fffffff) | __double2loint(b)) == 0;
    } else if constexpr (is_df<R>) {  // the signs of the leading floats
        return (a.hi < 0.f) != (b.hi < 0.f) || a.hi == 0.f || b.hi == 0.f;
    } else {
        return a * b <= R(0);
    }
}
// |a| < |b|
template <typename R>
__device__ __forceinline__ bool abs_lt(R a, R b)
{
    if constexpr (is_f64<R>) return mag_bits(a) < mag_bits(b); else return fabs(a) < fabs(b);
}
// neg ? -a : a.  FP64: the sign bit on the integer pipe (a negation that the compiler
// has to materialise is an FP64 instruction)
template <typename R>
__device__ __forceinline__ R neg_if(bool neg, R a)
{
    if constexpr (is_f64<R>)
        return __hiloint2double(__double2hiint(a) ^ (neg ? (int)0x80000000 : 0), __double2loint(a));
    else
        return neg ? -a : a;
}
// a > 0
template <typename R>
__device__ __forceinline__ bool positive(R a)
{
    if constexpr (is_f64<R>) return __double_as_longlong(a) > 0; else return a > R(0);
}

// twice the van Leer slope of the middle cell: 0 at an extremum, else the smallest of
// 2|dc|, 4|dl|, 4|dr| with the sign of dc -- that of dl and dr, so the smaller of the
// two is chosen first and scaled (exact)
template <typename R>
__device__ __forceinline__ R vl3x2(R am, R a0, R ap)
{
    const R dl = a0 - am, dr = ap - a0;
    if (nonpos_prod(dl, dr)) return R(0);
    const R dc = ap - am, t = scl2<R>(4.f, sel(abs_lt(dl, dr), dl, dr));
    return sel(abs_lt(t, dc), t, dc);
}

// a > b for b >= 0 (FP64 on the integer pipe: the signed bit patterns order
// a against a non-negative b)
template <typename R>
__device__ __forceinline__ bool gt_nonneg(R a, R b)
{
    if constexpr (is_f64<R>) return __double_as_longlong(a) > __double_as_longlong(b); else return a > b;
}

// limited PPM edge values (eL, eR) of the middle cell of a[0..4]
template <typename R>
__device__ __forceinline__ void ppm_edges3(const R *a, R &eL, R &eR)
{
    const R i12 = scl2<R>(0.5f, R(1.0 / 6.0));
    const R dm = vl3x2(a[0], a[1], a[2]), d0 = vl3x2(a[1], a[2], a[3]), dp = vl3x2(a[2], a[3], a[4]);
    const R c = a[2];
    R L = a[1] + scl2<R>(0.5f, c - a[1]) - (d0 - dm) * i12;
    R Rr = c + scl2<R>(0.5f, a[3] - c) - (dp - d0) * i12;
    const R rc = Rr - c, cl = c - L;
    if (nonpos_prod(rc, cl)) {
        L = c;
        Rr = c;
    } else {
        const R dA = Rr - L, m6 = dA * (c - scl2<R>(0.5f, L + Rr)), q = dA * dA * R(1.0 / 6.0);
        if (gt_nonneg(m6, q))
            L = c - scl2<R>(2.f, rc);
        else if (gt_nonneg(neg_if(true, m6), q))
            Rr = c + scl2<R>(2.f, cl);
    }
    eL = L;
    eR = Rr;
}

// time-centred upwind state at the face between a[2] and a[3] (a: cells f-3 .. f+2);
// dtih = dt / h.  The upwind cell's five-cell window is selected first and its
// parabola built once: vel >= 0 takes the right edge of a[2]'s parabola,
// Rr - C/2 (dA - (1 - 2C/3) a6), vel < 0 the left edge of a[3]'s, L + C/2 (dA +
// (1 - 2C/3) a6), with C = |vel| dt / h and a6 = 6 (c - (L + Rr) / 2), so that
// (1 - 2C/3) a6 = (6 - 4C) (c - (L + Rr) / 2) -- one copy of the edge code and no
// divergence between the two cases.
template <typename R>
__device__ __forceinline__ R ppm_face3(const R *a, R vel, R dtih)
{
    bool up;
    if constexpr (is_f64<R>)  // vel >= 0, -0 included
        up = __double_as_longlong(vel) >= 0 || (__double_as_longlong(vel) << 1) == 0;
    else
        up = vel >= R(0);
    R b[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) b[m] = sel(up, a[m], a[m + 1]);
    R L, Rr;
    ppm_edges3(b, L, Rr);
    const R C = neg_if(!up, vel) * dtih, dA = Rr - L;
    const R e = (R(6) - scl2<R>(4.f, C)) * (b[2] - scl2<R>(0.5f, L + Rr)), hc = scl2<R>(0.5f, C);
    return sel(up, Rr, L) + neg_if(up, hc) * (dA + neg_if(up, e));
}

// minmod: 0 for opposite signs, else the smaller in magnitude (a zero of either sign
// where one of them is zero)
template <typename R>
__device__ __forceinline__ R mm3(R a, R b)
{
    if constexpr (is_f64<R>)
        return sel((__double2hiint(a) ^ __double2hiint(b)) < 0, R(0), sel(abs_lt(a, b), a, b));
    else
        return nonpos_prod(a, b) ? R(0) : abs_lt(a, b) ? a : b;
}

// Koren-limited upwind face value: qu at an extremum, else qu + m/2 with m the
// smallest of 2|d2|, (|d1| + 2|d2|)/3, 2|d1| carrying the sign of d1.  d1 and d2 have
// that sign here, so the halves of the three are compared as they stand.
template <typename R>
__device__ __forceinline__ R koren3(R quu, R qu, R qd)
{
    const R d1 = qu - quu, d2 = qd - qu;
    if (nonpos_prod(d1, d2)) return qu;
    const R t = (d1 + scl2<R>(2.f, d2)) * scl2<R>(0.5f, R(1.0 / 3.0)), m = sel(abs_lt(d1, d2), d1, d2);
    return qu + sel(abs_lt(t, m), t, m);
}
template <typename R>
__device__ __forceinline__ R upw3(R q0, R q1, R q2, R q3, R vel)
{
    bool up;
    if constexpr (is_f64<R>)  // vel >= 0, -0 included
        up = __double_as_longlong(vel) >= 0 || (__double_as_longlong(vel) << 1) == 0;
    else
        up = vel >= R(0);
    // the upwind triple selected first: one copy of the limiter, no divergence
    return koren3(sel(up, q0, q3), sel(up, q1, q2), sel(up, q2, q1));
}

// The square of one direction's Godunov term for the sign pos of S: the largest of
// a, -b and 0 (pos) or of -a, b and 0, nb = -b.
template <typename R>
__device__ __forceinline__ R godunov_max(R a, R nb, bool pos)
{
    const R x = neg_if(!pos, a), y = neg_if(!pos, nb);
    const R m = sel(positive(x), x, R(0));
    bool ybig;
    if constexpr (is_f64<R>)
        ybig = positive(y) && mag_bits(y) > mag_bits(m);
    else
        ybig = y > m;
    return sel(ybig, y, m);
}

}  // namespace
}  // namespace wec
