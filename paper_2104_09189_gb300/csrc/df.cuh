// df.cuh -- double-float arithmetic on the FP32 pipe.
//
// GB300 executes about two FP64 operations per clock per SM against 128 FP32
// ones, and float<->double conversions run at the FP64 rate too.  The fast
// FP64-accuracy kernel therefore keeps values as unevaluated sums hi + lo of
// two floats (48-bit significands) and uses the error-free transformations
// of Knuth (TwoSum), Dekker (FastTwoSum) and the FMA-based exact product:
//   two_sum(a, b)      : s + e = a + b exactly, s = fl(a + b)
//   fast_two_sum(a, b) : the same when |a| >= |b| (or a == 0)
//   two_prod(a, b)     : p + e = a * b exactly (no underflow), p = fl(a * b)
// Intrinsics with explicit rounding stop the compiler from contracting or
// reassociating the error terms.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

namespace sl {

struct df {
    float h, l;
};

__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    float bv = __fsub_rn(s, a);
    float av = __fsub_rn(s, bv);
    e = __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
}

__device__ __forceinline__ void fast_two_sum_f(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

__device__ __forceinline__ df df_make(float h, float l)
{
    df r;
    r.h = h;
    r.l = l;
    return r;
}

// a + b: exact head sum, tails added in float; absolute error about
// 2^-24 (|a.l| + |b.l|) + 2^-48 |a + b|.
__device__ __forceinline__ df df_add(df a, df b)
{
    float s, e;
    two_sum_f(a.h, b.h, s, e);
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    df r;
    fast_two_sum_f(s, e, r.h, r.l);
    return r;
}

__device__ __forceinline__ df df_neg(df a) { return df_make(-a.h, -a.l); }

__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df_neg(b)); }

// a * b with relative error about 2^-46.
__device__ __forceinline__ df df_mul(df a, df b)
{
    float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    df r;
    fast_two_sum_f(p, e, r.h, r.l);
    return r;
}

// cross(a, b) = a.x b.y - a.y b.x for df vectors
__device__ __forceinline__ df df_cross(df ax, df ay, df bx, df by)
{
    return df_sub(df_mul(ax, by), df_mul(ay, bx));
}

// 1 / a, relative error about 2^-45 (a.h != 0)
__device__ __forceinline__ df df_rcp(df a)
{
    float r = __frcp_rn(a.h);
    // residual 1 - a r, computed with an exact product of the heads
    float e = __fmaf_rn(-a.h, r, 1.0f);
    e = __fmaf_rn(-a.l, r, e);
    df q;
    fast_two_sum_f(r, __fmul_rn(r, e), q.h, q.l);
    return q;
}

// Exact sign of orient(p, q, X) = (qx-px)(Xy-py) - (qy-py)(Xx-px) for double
// vertices p, q and a point X given as the exact sums Xx = xh + xl,
// Xy = yh + yl.  Expanded into ten products, each split without error by an
// FMA, and summed into a nonoverlapping expansion (Shewchuk's
// Grow-Expansion with zero elimination).  Exact while every nonzero input has
// magnitude in [2^-450, 2^450].
__device__ __forceinline__ int orient_exact_split(double px, double py, double qx, double qy, double xh, double xl,
                                                  double yh, double yl)
{
    // det = qx Xy - qx py - px Xy - qy Xx + qy px + py Xx
    const double u[10] = {qx, qx, -qx, -px, -px, -qy, -qy, qy, py, py};
    const double v[10] = {yh, yl, py, yh, yl, xh, xl, px, xh, xl};
    double e[20];
    int n = 0;
    for (int k = 0; k < 10; ++k) {
        double p = u[k] * v[k];
        double r = fma(u[k], v[k], -p);
        n = slp::grow(e, n, r);
        n = slp::grow(e, n, p);
    }
    if (n == 0) return 0;
    return e[n - 1] > 0.0 ? 1 : -1;
}

// h + l == p exactly, for a normalised float pair (h, l) and a double p:
// then h = fl32(p) and p - h is exact (Sterbenz), so the test is exact.
__device__ __forceinline__ bool df_equals(float h, float l, double p)
{
    return h == __double2float_rn(p) && (double)l == p - (double)h;
}

// Exact sign of orient(P, Q, X), X = (xh + xl, yh + yl), in three stages:
//  1. X on an axis-parallel edge line, or X equal to P or Q: exactly 0;
//  2. double evaluation of (Qx-Px)(Xy-Py) - (Qy-Py)(Xx-Px) with the
//     differences X - P formed by an error-free TwoSum (so feet a few ulps
//     from a vertex are still resolved), accepted when it clears its
//     forward error bound;
//  3. the full expansion (orient_exact_split).
// `stage` receives the stage that decided.
__device__ __forceinline__ int orient_exact_df(double2 P, double2 Q, float xh, float xl, float yh, float yl, int &stage)
{
    stage = 1;
    if (P.x == Q.x && df_equals(xh, xl, P.x)) return 0;
    if (P.y == Q.y && df_equals(yh, yl, P.y)) return 0;
    if ((df_equals(xh, xl, P.x) && df_equals(yh, yl, P.y)) || (df_equals(xh, xl, Q.x) && df_equals(yh, yl, Q.y)))
        return 0;                                             // X is an endpoint
    stage = 2;
    const double a = Q.x - P.x, b = Q.y - P.y;
    double s, e, r;
    slp::two_sum((double)xh, -P.x, s, e);
    r = e + (double)xl;
    const double c = s + r;                                   // X.x - P.x
    const double ec = 0x1p-52 * (fabs(c) + fabs(r));
    slp::two_sum((double)yh, -P.y, s, e);
    r = e + (double)yl;
    const double d = s + r;                                   // X.y - P.y
    const double ed = 0x1p-52 * (fabs(d) + fabs(r));
    const double t1 = a * d, t2 = b * c;
    const double det = t1 - t2;
    const double E = fabs(a) * ed + fabs(b) * ec + 0x1p-51 * (fabs(t1) + fabs(t2));
    if (fabs(c) + fabs(d) > 0x1p-900 && fabs(a) + fabs(b) > 0x1p-400) {
        if (det > E) return 1;
        if (det < -E) return -1;
    }
    stage = 3;
    return orient_exact_split(P.x, P.y, Q.x, Q.y, xh, xl, yh, yl);
}

// ---------------------------------------------------------------------------
// Values: a double as the (hi, lo) float pair of the double-float kernels and
// back.

// h = v rounded to the nearest float (ties to even) and l = v - h rounded
// to the nearest float, from the bits of v with integer operations, for
// 2^-74 <= |v| < 2^127 (both parts normal floats); false otherwise.  The
// 29 mantissa bits below the float's 23 decide the rounding of h; v - h is
// then the signed integer rem (or rem - 2^29) times 2^(e - 1075), exact, and
// converting that integer to float rounds it once, the scaling by a power of
// two being exact in the normal range.  GB300 converts double to float on its
// slow FP64 pipe, so this keeps the conversion at memory speed.
__device__ __forceinline__ bool split_double_bits(double v, float &h, float &l)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    const int e = (int)((hi >> 20) & 0x7FFu);
    if (e < 1075 - 126 || e > 1023 + 126) return false;
    const uint32_t sign = hi & 0x80000000u;
    const uint32_t top = ((hi & 0xFFFFFu) << 3) | (lo >> 29);   // the float's 23 mantissa bits
    const uint32_t rem = lo & 0x1FFFFFFFu;                       // the 29 bits below them
    const bool up = rem > 0x10000000u || (rem == 0x10000000u && (top & 1u));
    const uint32_t fb = (((uint32_t)(e - 1023 + 127) << 23) | top) + (up ? 1u : 0u);   // a carry bumps the exponent
    h = __uint_as_float(sign | fb);
    const int32_t r = up ? (int32_t)rem - 0x20000000 : (int32_t)rem;
    const float scale = __uint_as_float((uint32_t)(e - 1075 + 127) << 23);   // 2^(e - 1075)
    const float m = __fmul_rn(__int2float_rn(r), scale);
    l = sign ? -m : m;
    return true;
}

__device__ __forceinline__ float2 pair_of_double(double v)
{
    float h, l;
    if (!split_double_bits(v, h, l)) {
        // zero, tiny, huge or not finite: the FP64 pipe
        h = __double2float_rn(v);
        l = __double2float_rn(v - (double)h);
    }
    return make_float2(h, l);
}

// A float as a double from its bits (exact) for zero and normal floats;
// false for subnormal, infinite and NaN ones.
__device__ __forceinline__ bool widen_float_bits(float f, double &d)
{
    const uint32_t u = __float_as_uint(f);
    const uint32_t ef = (u >> 23) & 0xFFu;
    const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
    if ((u & 0x7FFFFFFFu) == 0u) {
        d = __longlong_as_double((long long)sign);
        return true;
    }
    if (ef == 0u || ef == 0xFFu) return false;
    d = __longlong_as_double((long long)(sign | ((unsigned long long)(ef - 127u + 1023u) << 52) |
                                         ((unsigned long long)(u & 0x7FFFFFu) << 29)));
    return true;
}

__device__ __forceinline__ double double_of_pair(float2 v)
{
    double a, b;
    if (!widen_float_bits(v.x, a)) a = (double)v.x;
    if (!widen_float_bits(v.y, b)) b = (double)v.y;
    return a + b;
}

}  // namespace sl
