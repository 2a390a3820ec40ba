// fmm_df.cuh -- the root of Algorithm 11 for double-precision grids with as
// little as possible on the FP64 pipe, which on GB300 runs at 1/64 of the float
// rate.
//
// df_root takes three FP64 additions, the ones whose operands are of order psi:
// the two shifts delta_i = psi_i - m and t = m + u.  The upwind set and a first
// root come from float arithmetic, then the exact residual of the quadratic about
// that root, in double-float (a value is an unevaluated sum hi + lo of two floats,
// about 46 significant bits), gives the correction.  Where the upwind set is
// recorded and a test is too close for float, df_shifted_root carries the whole
// root in double-float instead (four FP64 additions) and decides on the doubles.
//
// Error-free transformations (Knuth's two-sum, Dekker's fast two-sum, the
// exact product a*b - fl(a*b) from one fused multiply-add) build the
// double-float sums and products.
//
// Accuracy: for a causal root the discriminant is at least q/2 (q the speed
// term (h/F)^2), so no step cancels catastrophically and u carries a relative
// error of at most 3e-14 (against exact arithmetic, ties included), i.e. ~3e-17
// absolute on a grid with h = 1/1024: far below the fp64 parity tolerance of
// 1e-12 max|psi| even summed along a path of a thousand cells.
#pragma once

#include "fmm_fp64.cuh"

namespace fmmgb {

struct dfl {
    float h, l;
};

__device__ __forceinline__ dfl df_fast_two_sum(float a, float b)
{
    const float s = a + b;
    return {s, b - (s - a)};
}

__device__ __forceinline__ dfl df_two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}

// x + y (both of one sign, or a result not far below the operands)
__device__ __forceinline__ dfl df_add(dfl x, dfl y)
{
    const dfl s = df_two_sum(x.h, y.h);
    return df_fast_two_sum(s.h, s.l + (x.l + y.l));
}

__device__ __forceinline__ dfl df_neg(dfl x) { return {-x.h, -x.l}; }

// x * x
__device__ __forceinline__ dfl df_sqr(dfl x)
{
    const float p = x.h * x.h;
    const float e = fmaf(x.h, x.h, -p);
    return df_fast_two_sum(p, fmaf(2.0f * x.h, x.l, e));
}

// x * y
__device__ __forceinline__ dfl df_mul(dfl x, dfl y)
{
    const float p = x.h * y.h;
    const float e = fmaf(x.h, y.h, -p);
    return df_fast_two_sum(p, fmaf(x.h, y.l, fmaf(x.l, y.h, e)));
}

// k * x for a small integer k (exact product of the high part)
__device__ __forceinline__ dfl df_scale(dfl x, float k)
{
    const float p = k * x.h;
    const float e = fmaf(k, x.h, -p);
    return df_fast_two_sum(p, fmaf(k, x.l, e));
}

// sqrt(x), x.h > 0: float estimate and one Newton step in double-float
__device__ __forceinline__ dfl df_sqrt(dfl x)
{
    const float r = rsqrtf(x.h);
    const float s = x.h * r;
    const float res = fmaf(-s, s, x.h) + x.l;
    return df_fast_two_sum(s, res * (0.5f * r));
}

// A non-negative double of magnitude below 1e30 as a double-float: the value
// truncated to 24 significant bits (fmm_fp64.cuh's f32_of) plus the remaining
// fraction bits as a float (the low 29 bits of the double's fraction, of which
// the top 23 are kept), both built with integer operations.  The pair is not
// normalized (lo may reach a whole ulp of hi).  Values below 2^-100 become 0 (an
// absolute error no Algorithm 11 operand of order h notices).
__device__ __forceinline__ dfl df_of(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned E = (unsigned)(b >> 52) & 0x7ffu;
    if (E < 923u)   // below 2^-100, or zero
        return {0.0f, 0.0f};
    const float hi = f32_of(v);
    // 2^(E-1046) * (1 + m/2^23) - 2^(E-1046) with m the fraction bits 6..28
    const unsigned ef = (E - 919u) << 23;
    const unsigned m = ((unsigned)b & 0x1fffffffu) >> 6;
    const float lo = __uint_as_float(ef | m) - __uint_as_float(ef);
    return {hi, lo};
}

// A double-float as a double (one double addition of the exactly converted
// parts; fmm_fp64.cuh's f64_of is exact for normal floats, and a zero part
// is mapped to zero).
__device__ __forceinline__ double df_to_double(dfl x)
{
    const double h = x.h == 0.0f ? 0.0 : f64_of(x.h);
    const double l = x.l == 0.0f ? 0.0 : f64_of(x.l);
    return h + l;
}

// Algorithm 11's root for sorted upwind values m <= v1 <= v2 (nd of them
// present: nd = 1 uses m only), speed term q = (h/F)^2 in [1e-30, 1e30].
// With delta_i = v_i - m the root is t = m + u, u the larger root of
// sum_i (u - delta_i)^2 = q over the set: u = (S + sqrt(k q - P)) / k with
// S = sum delta_i and P = sum_{i<j} (delta_i - delta_j)^2 (Lagrange's form of
// S^2 - k (Q - q), a sum of squares, so nothing cancels), causal when the double
// root t = m + u exceeds the largest value; the largest value is dropped while
// the set is not causal.  Returns the number of values in the causal set (0:
// none, root +inf) and the root in t.
__device__ __forceinline__ int df_shifted_root(double m, double v1, double v2, int nd, double q,
                                               double &t)
{
    const double d1 = nd >= 2 ? v1 - m : 0.0;
    const double d2 = nd >= 3 ? v2 - m : 0.0;
    // operands far above the scale of q cannot be causal: clamp them into
    // the float range (an integer compare: both are >= 0)
    dfl D1 = df_of(__double_as_longlong(d1) < kF64Hi ? d1 : 1e30);
    dfl D2 = df_of(__double_as_longlong(d2) < kF64Hi ? d2 : 1e30);
    const dfl Q = df_of(q);
    const dfl third = {0.333333343267f, -9.93410748e-9f};   // 1/3 = hi + lo
#pragma unroll 1
    for (; nd != 0; --nd) {
        // S, P and k q over the current set (D2 = 0 once axis 2 is dropped,
        // D1 = 0 once axis 1 is)
        const dfl S = df_add(D1, D2);
        dfl P = df_sqr(D1);
        if (nd == 3)
            P = df_add(P, df_add(df_sqr(D2), df_sqr(df_add(D2, df_neg(D1)))));
        const dfl kq = df_scale(Q, (float)nd);
        const dfl disc = df_add(kq, df_neg(P));
        if (disc.h > 0.0f) {
            const dfl r = df_add(S, df_sqrt(disc));
            const dfl u = nd == 3 ? df_mul(r, third) : (nd == 2 ? dfl{0.5f * r.h, 0.5f * r.l} : r);
            // (tested on the doubles the cell and its neighbours will hold: the
            // test on the shifted double-floats can pass by a rounding step while
            // t rounds to that value or below it, and an upwind set recorded for
            // the adjoint must point strictly downhill)
            const double tt = m + df_to_double(u);
            const double vmax = nd == 3 ? v2 : v1;
            if (nd == 1 || __double_as_longlong(vmax) < __double_as_longlong(tt)) {
                t = tt;
                return nd;
            }
        }
        if (nd == 3)
            D2 = {0.0f, 0.0f};
        else
            D1 = {0.0f, 0.0f};
    }
    return 0;
}

// sqrt and reciprocal estimates (about one float ulp; subnormals count as 0,
// sqrt(+inf) = +inf, a negative argument gives NaN)
__device__ __forceinline__ float sqrt_est(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_est(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// A non-negative double as a double-float: the top 24 significant bits and
// the remaining 29 fraction bits, which the conversion rounds to 24.  The
// magnitude is clamped to [2^-100, 2^96] on the exponent (+inf comes out as
// 2^96); below 2^-74 the low part is only an error of at most 2^-97.
__device__ __forceinline__ dfl df_split(double v)
{
    const unsigned lo = (unsigned)__double2loint(v);
    const unsigned hi = umin(umax((unsigned)__double2hiint(v), 923u << 20), 1119u << 20);
    // 2^(E - 1075), the weight of the last fraction bit
    const float ulp = __uint_as_float(((umax(hi, 949u << 20) - (948u << 20)) & 0x7ff00000u) << 3);
    return {__uint_as_float(__funnelshift_l(lo, hi - (896u << 20), 3)),
            __uint2float_rn(lo & 0x1fffffffu) * ulp};
}

// u0 + c as a double, |c| below 1e-6 u0: the bit pattern of u0 moved by c in
// units of four last places (the patterns of adjacent doubles are adjacent
// integers), so no FP64 addition is spent.  A sum that leaves u0's binade
// counts the units beyond it double (below) or half (above).
// c2 is a second, smaller part of c.
__device__ __forceinline__ double df_shift(float u0, float c, float c2 = 0.0f)
{
    const unsigned E = (__float_as_uint(u0) >> 23) & 0xffu;
    const float inv = __uint_as_float((304u - E) << 23);   // 2^(50 - (E - 127))
    const long long d = 4ll * (__float2int_rn(c * inv) + (c2 != 0.0f ? __float2int_rn(c2 * inv) : 0));
    const long long base = (long long)(E + 896u) << 52;
    const long long f = ((long long)(__float_as_uint(u0) & 0x7fffffu) << 29) + d;   // fraction field
    long long t = base + f;
    if ((unsigned)((unsigned long long)f >> 32) >> 20)
        t += f < 0 ? f : -((f - (1ll << 52)) >> 1);
    return __longlong_as_double(t);
}

// What df_root needs of a speed term q = (h/F)^2 in [1e-30, 1e30]: q as a
// double-float, its square root, 2 q and 3 q.
struct DfSpeed {
    float h, l, s, h2, h3;
};
__device__ __forceinline__ DfSpeed df_speed(double q)
{
    const dfl Q = df_split(q);
    return {Q.h, Q.l, sqrt_est(Q.h), 2.0f * Q.h, 3.0f * Q.h};
}

// Algorithm 11's root for sorted upwind values m <= v1 <= v2 (+inf: absent; m
// finite), t = m + u as above: the upwind set and a root u0 in float, then the
// exact root of the quadratic about u0.
//
// The set grows while its root exceeds the next shift (the root of the larger
// set is below that of the smaller one and above the shift it added).  In
// float these tests can err where a root and a shift agree to about 1e-7; the
// two sets' roots then differ by about 1e-14 u, so without a recorded set
// either will do.  kStrict (the set is recorded): a test closer than 1e-5 goes
// to df_shifted_root, which decides on the doubles the cells hold.
//
// With r = q - sum (u0 - delta_i)^2 in double-float and g = sum (u0 -
// delta_i), u - u0 = c - k c^2 / (2 g) + O(c^3), c = r / (2 g); c is about 1e-7
// u0, so its float rounding is about 1e-14 u0 (all in all at most 3e-14).  Three FP64 additions in all
// (two shifts and m + u) on a pipe that takes one warp instruction in 16
// cycles, against four, and about half the float operations, when the root is
// carried in double-float throughout (df_shifted_root).
template <bool kStrict>
__device__ __forceinline__ int df_root(double m, double v1, double v2, const DfSpeed &Q, double q, double &t)
{
    const dfl D1 = df_split(v1 - m), D2 = df_split(v2 - m);
    const float a1 = D1.h, a2 = D2.h, e = a2 - a1, f1 = a1 * a1;
    const bool c1 = a1 < Q.s;
    const float u2 = c1 ? 0.5f * (a1 + sqrt_est(Q.h2 - f1)) : Q.s;
    const bool c2 = a2 < u2;
    if constexpr (kStrict) {
        if (fabsf(a1 - Q.s) < 1e-5f * Q.s || (c1 && fabsf(a2 - u2) < 1e-5f * u2))
            return df_shifted_root(m, v1, v2, v1 < 1e300 ? (v2 < 1e300 ? 3 : 2) : 1, q, t);
    }
    // (products that feed an error-free sum are rounded on their own: a fused
    // multiply-add there would not be the sum whose error is taken)
    const float u0 = c2 ? __fmul_rn((a1 + a2) + sqrt_est(Q.h3 - fmaf(a2, a2, fmaf(e, e, f1))), 0.333333343f) : u2;
    // u0 - delta_i as high + low parts (0 for an axis that is not in the
    // set; u0 is not below a shift of the set, so the difference's error is
    // the two-term one)
    const float b1 = c1 ? a1 : u0, b2 = c2 ? a2 : u0;
    const float x1 = u0 - b1, x2 = u0 - b2;
    const float l1 = ((u0 - x1) - b1) - (c1 ? D1.l : 0.0f), l2 = ((u0 - x2) - b2) - (c2 ? D2.l : 0.0f);
    // r: every partial sum is at least what is subtracted next
    const float p0 = __fmul_rn(u0, u0), p1 = __fmul_rn(x1, x1);
    const float s0 = Q.h - p0, s1 = s0 - p1;
    const float r0 = ((Q.h - s0) - p0) - fmaf(u0, u0, -p0);
    const float r1 = ((s0 - s1) - p1) - fmaf(x1, x1, -p1);
    const float z = fmaf(x1, l1, x2 * l2);
    const float ra = fmaf(-x2, x2, s1), rb = fmaf(-2.0f, z, (r0 + r1) + Q.l);
    const float g = u0 + (x1 + x2), ri = 0.5f * rcp_est(g);
    const float k = c2 ? -3.0f : (c1 ? -2.0f : -1.0f);
    if constexpr (kStrict) {
        // the adjoint divides by sums of t - psi_i, which carry the error of u:
        // c in two parts (4.6e-15 of u off in the mean with one, 2.9e-15 with
        // two; dL/ds of a 125x110x131 grid 3.5e-14 and 2.3e-14 off)
        const dfl r = df_two_sum(ra, rb);
        const float c = r.h * ri;
        t = m + df_shift(u0, c, (fmaf(-2.0f * g, c, r.h) + fmaf(k * c, c, r.l)) * ri);
    } else {
        const float c = (ra + rb) * ri;
        t = m + df_shift(u0, fmaf(k * c, c * ri, c));
    }
    if constexpr (kStrict) {
        // m so large that t rounds to a value of the set
        if (c1 && __double_as_longlong(t) <= __double_as_longlong(c2 ? v2 : v1))
            return df_shifted_root(m, v1, v2, v1 < 1e300 ? (v2 < 1e300 ? 3 : 2) : 1, q, t);
    }
    return c2 ? 3 : (c1 ? 2 : 1);
}

}  // namespace fmmgb
