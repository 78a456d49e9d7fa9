// fch_df.cuh -- double-float arithmetic: a value is the unevaluated sum hi + lo of
// two floats with |lo| <= ulp(hi)/2, about 48 significant bits. The FP64 pipe of
// this GPU runs at a small fraction of the FP32 rate; carrying FP64-class
// precision as float pairs keeps every operation on the FP32 pipe.
//
// Error-free transformations used (classical results, restated here):
//   TwoSum (Knuth): s = fl(a + b), e = (a - (s - b')) + (b - b'), b' = s - a, gives
//     a + b = s + e exactly for any floats a, b;
//   FastTwoSum (Dekker): for |a| >= |b|, s = fl(a + b), e = b - (s - a) is exact;
//   TwoProd with a fused multiply-add: p = fl(a b), e = fma(a, b, -p), a b = p + e.
// Addition sums the high parts with TwoSum and the low parts with one rounding
// (error bounded relative to the operands); multiplication adds the cross terms to
// the exact product of the high parts; division refines a float quotient with two
// correction terms, the reciprocal takes one Newton step. exp and expm1 (the q > 0 well
// and the ETD phi functions) are table-driven on the FP32 pipe.
// Compile without fast-math: the transformations rely on IEEE rounding of each step.
#pragma once
#include <math.h>

namespace fch {

struct df {
    float hi, lo;
    df() = default;
    __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ constexpr df(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ constexpr df(int i) : hi((float)i), lo(0.f) {}
    __host__ __device__ explicit operator double() const { return (double)hi + (double)lo; }
    __host__ __device__ explicit operator float() const { return hi + lo; }
};

struct __align__(16) df2 {
    df x, y;
};

// read-only loads of complex elements
__device__ __forceinline__ float2 ldg(const float2 *p) { return __ldg(p); }
__device__ __forceinline__ double2 ldg(const double2 *p) { return __ldg(p); }
__device__ __forceinline__ df2 ldg(const df2 *p)
{
    const float4 v = __ldg((const float4 *)p);
    df2 r;
    r.x = df(v.x, v.y);
    r.y = df(v.z, v.w);
    return r;
}

// The sums and products of the transformations use the explicitly rounded intrinsics
// (__fadd_rn, __fsub_rn, __fmul_rn): the compiler never contracts those into fused
// multiply-adds, which would break the exactness these steps rely on (a product fused
// into the TwoSum that consumes it counts its rounding error twice).
__device__ __forceinline__ df two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return df(s, e);
}

__device__ __forceinline__ df fast_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return df(s, __fsub_rn(b, __fsub_rn(s, a)));
}

// Sums. The high parts are added exactly (TwoSum), the low parts with one rounding:
// an error of a few u^2 (|a| + |b|), u = 2^-24, relative to the operands rather
// than to a cancelled result. That is the norm-wise accuracy a transform's error
// analysis needs (its output error is bounded by eps log N times the input norm).
//
// The operators renormalise the sum (add_norm, 11 operations). add_lazy / sub_lazy
// leave it unrenormalised (8 operations): |lo| may exceed ulp(hi)/2, and after a
// cancellation of the high parts it may exceed |hi|; the transform butterflies use
// them and renormalise once where a transform ends (renorm restores |lo| <= ulp(hi)/2
// where |hi| >= |lo|, renorm_exact in every case). Whatever reads only the high
// word -- division, reciprocal, comparisons, signs -- renormalises its operands
// first with renorm_exact.
__device__ __forceinline__ df add_lazy(df a, df b)
{
    df s = two_sum(a.hi, b.hi);
    s.lo += a.lo + b.lo;
    return s;
}
__device__ __forceinline__ df sub_lazy(df a, df b)
{
    df s = two_sum(a.hi, -b.hi);
    s.lo += a.lo - b.lo;
    return s;
}
__device__ __forceinline__ df renorm(df a) { return fast_two_sum(a.hi, a.lo); }
__device__ __forceinline__ df renorm_exact(df a) { return two_sum(a.hi, a.lo); }
__device__ __forceinline__ df add_norm(df a, df b)
{
    const df s = add_lazy(a, b);
    return fast_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ df operator+(df a, df b) { return add_norm(a, b); }
__device__ __forceinline__ df operator-(df a) { return df(-a.hi, -a.lo); }
__device__ __forceinline__ df operator-(df a, df b) { return add_norm(a, -b); }

__device__ __forceinline__ df operator*(df a, df b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}

// Product without the final renormalisation (4 operations instead of 7): the exact
// product of the high words and, in one error word, its rounding error and the two
// cross terms. The low word may exceed ulp(hi)/2 by a few units; sums and products
// take such operands (their error stays a few u^2 relative to the operands' size),
// and whatever reads only the high word renormalises first. A product neglects
// lo x lo: an operand whose high word cancelled in an unrenormalised difference (the
// value then sits in lo) is renormalised before it meets another such operand (a
// square of a small difference above all).
__device__ __forceinline__ df mul_lazy(df a, df b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df(p, e);
}

// by +-1 (the DIR factors of the butterflies)
__device__ __forceinline__ df operator*(int s, df a) { return s < 0 ? -a : a; }

// Quotient by long division: three float quotient digits, each remainder
// renormalised before its leading word is read.
__device__ __forceinline__ df operator/(df a, df b)
{
    a = renorm_exact(a);
    b = renorm_exact(b);
    const float rb = 1.0f / b.hi;
    const float q1 = a.hi * rb;
    df r = renorm_exact(sub_lazy(a, b * df(q1, 0.f)));
    const float q2 = r.hi * rb;
    r = renorm_exact(sub_lazy(r, b * df(q2, 0.f)));
    const float q3 = r.hi * rb;
    const df q = fast_two_sum(q1, q2);
    return add_norm(q, df(q3, 0.f));
}

// Reciprocal by one Newton step from the float reciprocal r0 of the leading word:
// 1/d = r0 (1 + e) + O(e^2) with e = 1 - d r0 = O(2^-24), e formed to about 2^-48
// absolute (d.hi r0 split exactly by a fused multiply-add; 1 - p exact since p is
// within 2^-23 of 1), so the result carries a few u^2 relative error.
__device__ __forceinline__ df recip(df d)
{
    d = renorm_exact(d);
    const float r0 = 1.0f / d.hi;
    const float p = __fmul_rn(d.hi, r0);
    const float pe = fmaf(d.hi, r0, -p);
    const float e = ((1.0f - p) - pe) - d.lo * r0;
    return fast_two_sum(r0, r0 * e);
}
__device__ __forceinline__ float recip(float d) { return 1.0f / d; }
__device__ __forceinline__ double recip(double d) { return 1.0 / d; }

// a s for an exact power of two s (both words scale exactly; s.lo is 0)
__device__ __forceinline__ df mul_p2(df a, df s) { return df(a.hi * s.hi, a.lo * s.hi); }
__device__ __forceinline__ float mul_p2(float a, float s) { return a * s; }
__device__ __forceinline__ double mul_p2(double a, double s) { return a * s; }

// Complex product a w for a twiddle factor w, each part a sum of two products
// with one TwoSum: the high products are added exactly, their rounding errors
// (from fused multiply-adds) and the four cross terms with the low words go into
// one error word, left unrenormalised (16 operations a part instead of 25).
__device__ __forceinline__ df2 cmul_lazy(df2 a, df2 w)
{
    df2 r;
    {
        const float p1 = __fmul_rn(a.x.hi, w.x.hi), p2 = __fmul_rn(a.y.hi, w.y.hi);
        r.x = two_sum(p1, -p2);
        float e = fmaf(a.x.hi, w.x.hi, -p1) - fmaf(a.y.hi, w.y.hi, -p2);
        e = fmaf(a.x.hi, w.x.lo, e);
        e = fmaf(a.x.lo, w.x.hi, e);
        e = fmaf(-a.y.hi, w.y.lo, e);
        e = fmaf(-a.y.lo, w.y.hi, e);
        r.x.lo += e;
    }
    {
        const float p1 = __fmul_rn(a.x.hi, w.y.hi), p2 = __fmul_rn(a.y.hi, w.x.hi);
        r.y = two_sum(p1, p2);
        float e = fmaf(a.x.hi, w.y.hi, -p1) + fmaf(a.y.hi, w.x.hi, -p2);
        e = fmaf(a.x.hi, w.y.lo, e);
        e = fmaf(a.x.lo, w.y.hi, e);
        e = fmaf(a.y.hi, w.x.lo, e);
        e = fmaf(a.y.lo, w.x.hi, e);
        r.y.lo += e;
    }
    return r;
}

__device__ __forceinline__ df &operator+=(df &a, df b) { return a = a + b; }
__device__ __forceinline__ df &operator-=(df &a, df b) { return a = a - b; }
__device__ __forceinline__ df &operator*=(df &a, df b) { return a = a * b; }
__device__ __forceinline__ df &operator/=(df &a, df b) { return a = a / b; }

// comparisons (on renormalised operands)
__device__ __forceinline__ bool operator<(df a, df b)
{
    a = renorm_exact(a);
    b = renorm_exact(b);
    return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}
__device__ __forceinline__ bool operator>(df a, df b) { return b < a; }
__device__ __forceinline__ bool operator==(df a, df b)
{
    a = renorm_exact(a);
    b = renorm_exact(b);
    return a.hi == b.hi && a.lo == b.lo;
}
__device__ __forceinline__ bool operator!=(df a, df b) { return !(a == b); }

// float and double forms next to the double-float ones, so unqualified calls in
// namespace fch find every overload
__device__ __forceinline__ float fabs(float a) { return ::fabsf(a); }
__device__ __forceinline__ double fabs(double a) { return ::fabs(a); }
__device__ __forceinline__ float exp(float a) { return ::expf(a); }
__device__ __forceinline__ double exp(double a) { return ::exp(a); }
__device__ __forceinline__ float expm1(float a) { return ::expm1f(a); }
__device__ __forceinline__ double expm1(double a) { return ::expm1(a); }
__device__ __forceinline__ float copysign(float a, float b) { return ::copysignf(a, b); }
__device__ __forceinline__ double copysign(double a, double b) { return ::copysign(a, b); }

__device__ __forceinline__ df fabs(df a)
{
    a = renorm_exact(a);
    return a.hi < 0.f ? -a : a;
}
__device__ __forceinline__ df copysign(df a, df s)
{
    a = renorm_exact(a);
    s = renorm_exact(s);
    return (a.hi < 0.f) != (s.hi < 0.f) ? -a : a;
}

// exp and expm1 on the FP32 pipe, table-driven (P. T. P. Tang, "Table-driven implementation
// of the exponential function in IEEE floating-point arithmetic", 1989): a = n ln2/32 + r,
// |r| <= ln2/64; e^a = 2^(n/32) (1 + p), p = e^r - 1 by the series (terms from r^4/4! on in
// single precision: they are below 2^-30), 2^(n/32) = 2^e T_j from the table. ln2/32 and T_j
// are split in three floats: n L1 cancels against a.hi without rounding (fused multiply-add),
// n L2 is an exact product. Everything is carried to about 2^-52 of the result, so that its
// one rounding to the format (2^-49, the low word's) is the error, as it was of the double
// pipe's exp rounded to double-float: rms 2^-50.6 of both. (With T_j in two floats and sums
// of one rounding a word it was 2^-49.4.) The double exp costs some twenty double operations a
// point, 64 FP32 issue slots each.
__device__ const float4 kExp2Tab[32] = { // 2^(j/32) = x + y + z
    {0x1.0p+0f, 0x0.0p+0f, 0x0.0p+0f, 0.f}, {0x1.059b0ep+0f, -0x1.9d4f52p-25f, 0x1.0eb9f2p-50f, 0.f},
    {0x1.0b5586p+0f, 0x1.9f3122p-25f, -0x1.3ace8ep-53f, 0.f}, {0x1.11301ep+0f, -0x1.fdb496p-25f, 0x1.49d77ep-53f, 0.f},
    {0x1.172b84p+0f, -0x1.c15742p-27f, -0x1.232084p-52f, 0.f}, {0x1.1d4874p+0f, -0x1.d2e8cap-25f, -0x1.61fe92p-50f, 0.f},
    {0x1.2387a6p+0f, 0x1.ceac48p-25f, -0x1.e64f82p-50f, 0.f}, {0x1.29e9ep+0f, -0x1.5c0424p-25f, 0x1.2c25d2p-52f, 0.f},
    {0x1.306fep+0f, 0x1.4636e2p-25f, 0x1.4b7a36p-50f, 0.f}, {0x1.371a74p+0f, -0x1.18aac6p-25f, -0x1.563aeap-50f, 0.f},
    {0x1.3dea64p+0f, 0x1.824684p-25f, 0x1.1ada0ap-51f, 0.f}, {0x1.44e086p+0f, 0x1.8624b4p-30f, 0x1.89b7ap-59f, 0.f},
    {0x1.4bfdaep+0f, -0x1.593abcp-25f, 0x1.c750e6p-50f, 0.f}, {0x1.5342b6p+0f, -0x1.2c561p-25f, 0x1.df0a84p-52f, 0.f},
    {0x1.5ab07ep+0f, -0x1.5bd5ecp-27f, 0x1.58c93p-52f, 0.f}, {0x1.6247ecp+0f, -0x1.f8b55p-25f, 0x1.2c7c3ep-50f, 0.f},
    {0x1.6a09e6p+0f, 0x1.9fcef4p-26f, -0x1.b7ba68p-51f, 0.f}, {0x1.71f75ep+0f, 0x1.1d8beep-25f, 0x1.ee91b8p-51f, 0.f},
    {0x1.7a1148p+0f, -0x1.829fdp-25f, 0x1.b5f544p-50f, 0.f}, {0x1.82589ap+0f, -0x1.accc7cp-26f, 0x1.4567c4p-51f, 0.f},
    {0x1.8ace54p+0f, 0x1.15506ep-27f, -0x1.48b076p-53f, 0.f}, {0x1.93737cp+0f, -0x1.e64744p-25f, 0x1.3d1408p-50f, 0.f},
    {0x1.9c4918p+0f, 0x1.51f848p-27f, 0x1.c7c46cp-56f, 0.f}, {0x1.a5503cp+0f, -0x1.b83b54p-25f, -0x1.ba5edep-51f, 0.f},
    {0x1.ae89fap+0f, -0x1.a94b14p-26f, -0x1.50bc66p-51f, 0.f}, {0x1.b7f77p+0f, -0x1.a09438p-25f, 0x1.baa9ecp-50f, 0.f},
    {0x1.c199bep+0f, -0x1.3d56b2p-27f, 0x1.110658p-55f, 0.f}, {0x1.cb720ep+0f, -0x1.8837ccp-27f, 0x1.1503ccp-52f, 0.f},
    {0x1.d5818ep+0f, -0x1.822dbcp-27f, -0x1.b44bf4p-53f, 0.f}, {0x1.dfc974p+0f, -0x1.908c94p-25f, -0x1.469736p-52f, 0.f},
    {0x1.ea4afap+0f, 0x1.52486cp-27f, 0x1.858f74p-52f, 0.f}, {0x1.f50766p+0f, -0x1.246ebp-26f, 0x1.9d3e12p-54f, 0.f},
};

struct df_exp_parts {
    df T, p;  // 2^(j/32) without its third word, e^r - 1
    float T2; // the third word
    int e;    // binary exponent
};
__device__ __forceinline__ df_exp_parts exp_parts(df a)
{
    const float n = rintf(a.hi * 0x1.715476p+5f); // 32 / ln 2
    const float r1 = fmaf(-n, 0x1.62e43p-6f, a.hi); // exact
    const float p2 = __fmul_rn(n, 0x1.05c61p-34f), pe = fmaf(n, 0x1.05c61p-34f, -p2);
    const df s = two_sum(p2, a.lo);
    df r = two_sum(r1, s.hi);
    r.lo += s.lo + fmaf(n, 0x1.950d88p-59f, pe);
    const float q = fmaf(r.hi, fmaf(r.hi, (float)(1.0 / 720), (float)(1.0 / 120)), (float)(1.0 / 24));
    df c = two_sum((float)(1.0 / 6), __fmul_rn(r.hi, q));
    c.lo += (float)(1.0 / 6 - (double)(float)(1.0 / 6));
    c = mul_lazy(c, r);
    df h = two_sum(0.5f, c.hi);
    h.lo += c.lo;
    df_exp_parts o;
    o.p = add_lazy(r, mul_lazy(mul_lazy(r, r), h)); // r + r^2 (1/2 + r (1/6 + r q))
    const int N = (int)n;
    const float4 t = __ldg(kExp2Tab + (N & 31));
    o.T = df(t.x, t.y);
    o.T2 = t.z;
    o.e = N >> 5;
    return o;
}
// x 2^e for any e (two factors where 2^e is below the normal range)
__device__ __forceinline__ float scale2(float x, int e)
{
    const int e1 = max(e, -126), e2 = max(e - e1, -126);
    return x * __int_as_float((e1 + 127) << 23) * __int_as_float((e2 + 127) << 23);
}
// hi + x + l0 + l1 + rest with one rounding, of the result's low word: |hi| >= |x|, l0 and
// l1 of the size of that sum's rounding or below, rest below theirs
__device__ __forceinline__ df sum_once(float hi, float x, float l0, float l1, float rest)
{
    const df s = two_sum(hi, x), l = two_sum(s.lo, l0), k = two_sum(l.hi, l1);
    df o = fast_two_sum(s.hi, k.hi);
    o.lo += l.lo + k.lo + rest;
    return o;
}
__device__ __forceinline__ df exp(df a)
{
    if (a.hi < -200.0f) return df(0.f, 0.f); // far below the underflow, -inf too (its low word is NaN)
    a = renorm_exact(a);
    if (!(a.hi < 88.0f)) return df(::exp((double)a)); // near and above the overflow of a float, NaN
    const df_exp_parts x = exp_parts(a);
    const df m = mul_lazy(x.T, x.p), y = sum_once(x.T.hi, m.hi, x.T.lo, m.lo, x.T2);
    return df(scale2(y.hi, x.e), scale2(y.lo, x.e));
}
// expm1: the series below 0.1, where e^a - 1 would cancel
__device__ __forceinline__ df expm1(df a)
{
    if (a.hi < -200.0f) return df(-1.f, 0.f);
    a = renorm_exact(a);
    if (!(a.hi < 88.0f)) return df(::expm1((double)a));
    if (::fabsf(a.hi) < 0.1f) {
        // a + a^2 (1/2! + a (1/3! + ...)), terms from a^7/7! on in single precision
        float t = (float)(1.0 / 39916800.0);
        t = fmaf(t, a.hi, (float)(1.0 / 3628800.0));
        t = fmaf(t, a.hi, (float)(1.0 / 362880.0));
        t = fmaf(t, a.hi, (float)(1.0 / 40320.0));
        t = fmaf(t, a.hi, (float)(1.0 / 5040.0));
        df s(t, 0.f);
        const double c[5] = {1.0 / 720, 1.0 / 120, 1.0 / 24, 1.0 / 6, 1.0 / 2};
#pragma unroll
        for (int i = 0; i < 5; i++) s = add_lazy(df(c[i]), mul_lazy(s, a));
        const df w = mul_lazy(mul_lazy(a, a), s);
        return sum_once(a.hi, w.hi, a.lo, w.lo, 0.f);
    }
    const df_exp_parts x = exp_parts(a);
    const df T(scale2(x.T.hi, x.e), scale2(x.T.lo, x.e)), m = mul_lazy(T, x.p), d = two_sum(T.hi, -1.0f);
    const df l = two_sum(d.lo, T.lo);
    return sum_once(d.hi, m.hi, l.hi, m.lo, l.lo + scale2(x.T2, x.e));
}

} // namespace fch
