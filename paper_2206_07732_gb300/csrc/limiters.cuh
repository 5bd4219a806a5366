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
// at 1/64 of its FP32 rate.  The FP32 stencils keep plain float compares.
__device__ __forceinline__ unsigned long long mag_bits(double a)
{
    return (unsigned long long)__double_as_longlong(a) << 1;
}
// a * b <= 0 (opposite signs, or a zero factor)
template <typename R>
__device__ __forceinline__ bool nonpos_prod(R a, R b)
{
    if constexpr (is_f64<R>) {
        const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
        return (ia ^ ib) < 0 || (ia << 1) == 0 || (ib << 1) == 0;
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
// a > 0
template <typename R>
__device__ __forceinline__ bool positive(R a)
{
    if constexpr (is_f64<R>) return __double_as_longlong(a) > 0; else return a > R(0);
}

// van Leer slope of the middle cell: 0 at an extremum, else the smallest of
// |dc|, 2|dl|, 2|dr| with the sign of dc (the magnitude choice and the sign on
// the integer pipe in FP64)
template <typename R>
__device__ __forceinline__ R vl3(R am, R a0, R ap)
{
    const R dl = a0 - am, dr = ap - a0;
    if (nonpos_prod(dl, dr)) return R(0);
    const R dc = scl2<R>(0.5f, ap - am), tl = scl2<R>(2.f, dl), tr = scl2<R>(2.f, dr);
    if constexpr (is_f64<R>) {
        unsigned long long m = mag_bits(dc);
        const unsigned long long ml = mag_bits(tl), mr = mag_bits(tr);
        m = ml < m ? ml : m;
        m = mr < m ? mr : m;
        // |result| = the smallest magnitude, sign of dc
        const unsigned long long sgn = (unsigned long long)__double_as_longlong(dc) & 0x8000000000000000ull;
        return __longlong_as_double((long long)((m >> 1) | sgn));
    } else {
        const R m = fmin(fabs(dc), fmin(fabs(tl), fabs(tr)));
        return dc > R(0) ? m : -m;
    }
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
    const R i6 = R(1.0 / 6.0);
    const R dm = vl3(a[0], a[1], a[2]), d0 = vl3(a[1], a[2], a[3]), dp = vl3(a[2], a[3], a[4]);
    R L = a[1] + scl2<R>(0.5f, a[2] - a[1]) - (d0 - dm) * i6;
    R Rr = a[2] + scl2<R>(0.5f, a[3] - a[2]) - (dp - d0) * i6;
    const R c = a[2];
    if (nonpos_prod(Rr - c, c - L)) {
        L = c;
        Rr = c;
    } else {
        const R dA = Rr - L, m6 = dA * (c - scl2<R>(0.5f, L + Rr)), q = dA * dA * i6;
        if (gt_nonneg(m6, q))
            L = R(3) * c - scl2<R>(2.f, Rr);
        else if (gt_nonneg(-m6, q))
            Rr = R(3) * c - scl2<R>(2.f, L);
    }
    eL = L;
    eR = Rr;
}

// time-centred upwind state at the face between a[2] and a[3] (a: cells f-3 .. f+2);
// dtih = dt / h.  The upwind cell's five-cell window is selected first and its
// parabola built once: vel >= 0 takes the right edge of a[2]'s parabola,
// Rr - C/2 (dA - (1 - 2C/3) a6), vel < 0 the left edge of a[3]'s, L + C/2 (dA +
// (1 - 2C/3) a6), with C = |vel| dt / h -- one copy of the edge code and no
// divergence between the two cases.
template <typename R>
__device__ __forceinline__ R ppm_face3(const R *a, R vel, R dtih)
{
    const R t3 = R(2.0 / 3.0);
    bool up;
    if constexpr (is_f64<R>)  // vel >= 0, -0 included
        up = __double_as_longlong(vel) >= 0 || (__double_as_longlong(vel) << 1) == 0;
    else
        up = vel >= R(0);
    R b[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) b[m] = up ? a[m] : a[m + 1];
    R L, Rr;
    ppm_edges3(b, L, Rr);
    const R C = (up ? vel : -vel) * dtih, dA = Rr - L, a6 = R(6) * (b[2] - scl2<R>(0.5f, L + Rr));
    const R e = (R(1) - C * t3) * a6, hc = scl2<R>(0.5f, C);
    return (up ? Rr : L) + (up ? -hc : hc) * (dA + (up ? -e : e));
}

template <typename R>
__device__ __forceinline__ R mm3(R a, R b)
{
    if (nonpos_prod(a, b)) return R(0);
    return abs_lt(a, b) ? a : b;
}

// Koren-limited upwind face value: qu at an extremum, else qu + m/2 with m the
// smallest of 2|d2|, (|d1| + 2|d2|)/3, 2|d1| carrying the sign of d1 (FP64: the
// choice and the sign on the integer pipe)
template <typename R>
__device__ __forceinline__ R koren3(R quu, R qu, R qd)
{
    const R d1 = qu - quu, d2 = qd - qu;
    if (nonpos_prod(d1, d2)) return qu;
    if constexpr (is_f64<R>) {
        const R t2 = scl2<R>(2.f, d2), t1 = scl2<R>(2.f, d1), tm = (fabs(d1) + fabs(t2)) * R(1.0 / 3.0);
        unsigned long long m = mag_bits(t2);
        const unsigned long long mm = mag_bits(tm), m1 = mag_bits(t1);
        m = mm < m ? mm : m;
        m = m1 < m ? m1 : m;
        const unsigned long long sgn = (unsigned long long)__double_as_longlong(d1) & 0x8000000000000000ull;
        return qu + scl2<R>(0.5f, __longlong_as_double((long long)((m >> 1) | sgn)));
    } else {
        const R m = fmin(scl2<R>(2.f, fabs(d2)), fmin((fabs(d1) + scl2<R>(2.f, fabs(d2))) * R(1.0 / 3.0), scl2<R>(2.f, fabs(d1))));
        return d1 > R(0) ? qu + scl2<R>(0.5f, m) : qu - scl2<R>(0.5f, m);
    }
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
    return koren3(up ? q0 : q3, up ? q1 : q2, up ? q2 : q1);
}

// The square of one direction's Godunov term for the sign pos of S: the largest of
// a, -b and 0 (pos) or of -a, b and 0, nb = -b.
template <typename R>
__device__ __forceinline__ R godunov_max(R a, R nb, bool pos)
{
    const R x = pos ? a : -a, y = pos ? nb : -nb;
    R m = positive(x) ? x : R(0);
    bool ybig;
    if constexpr (is_f64<R>)
        ybig = positive(y) && mag_bits(y) > mag_bits(m);
    else
        ybig = y > m;
    return ybig ? y : m;
}

}  // namespace
}  // namespace wec
