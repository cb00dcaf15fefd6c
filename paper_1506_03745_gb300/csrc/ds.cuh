// Double-single arithmetic: a number is the unevaluated sum hi + lo of two
// FP32 values with |lo| <= ulp(hi) / 2, about 48 significant bits in the
// FP32 exponent range (magnitudes from about 1e-38 to 1e38; lo loses bits
// below about 1e-31).  Built on the error-free transformations of Knuth
// (two-sum, TAOCP vol. 2, 4.2.2) and Dekker (product error, here by one fused
// multiply-add; Numer. Math. 18, 1971).  The treecode's FP64-class product
// (the outer residual of the refinement) runs in it on the FP32 pipe, which
// GB300 issues 64 times as fast as FP64.  Every operation is written with
// the _rn intrinsics so that the compiler neither fuses nor reorders them.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace pgb {

struct __align__(8) ds {
    float hi, lo;
    ds() = default;
    __host__ __device__ constexpr ds(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ constexpr ds(int i) : hi((float)i), lo(0.f) {}  // exact for |i| < 2^24
};

// Split of a double constant (folded at compile time for literals).
__host__ __device__ constexpr ds ds_const(double d) {
    return ds((float)d, (float)(d - (double)(float)d));
}

__device__ __forceinline__ ds ds_from_double(double d) {
    const float h = __double2float_rn(d);
    return ds(h, __double2float_rn(d - (double)h));
}
__device__ __forceinline__ double ds_to_double(ds a) { return (double)a.hi + (double)a.lo; }

// s + e = a + b exactly (Knuth)
__device__ __forceinline__ ds two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return ds(s, e);
}
// the same when |a| >= |b| (or a == 0)
__device__ __forceinline__ ds fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return ds(s, __fsub_rn(b, __fsub_rn(s, a)));
}

// a + b with error below about 2^-47 (|a| + |b|)
__device__ __forceinline__ ds operator+(ds a, ds b) {
    const ds s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ds operator-(ds a) { return ds(-a.hi, -a.lo); }
__device__ __forceinline__ ds operator-(ds a, ds b) { return a + (-b); }
__device__ __forceinline__ ds& operator+=(ds& a, ds b) {
    a = a + b;
    return a;
}
// a b: the exact product of the high parts by one fused multiply-add, the
// cross terms added to its error (relative error below about 2^-46)
__device__ __forceinline__ ds operator*(ds a, ds b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}
// a b + c in one pass: the product's error term joins the sum (error below
// about 2^-46 (|a b| + |c|)); 15 FP32 operations instead of 18
__device__ __forceinline__ ds ds_fma(ds a, ds b, ds c) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    const ds s = two_sum(p, c.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(e, c.lo)));
}
__device__ __forceinline__ ds mul_f(ds a, float b) {
    const float p = __fmul_rn(a.hi, b);
    float e = __fmaf_rn(a.hi, b, -p);
    e = __fmaf_rn(a.lo, b, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ bool operator>(ds a, ds b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }

// The same operations without the closing renormalisation (3 fewer each): the
// result's lo may reach a few ulps of its hi.  They take such operands
// themselves, as long as no cancellation has made lo large beside hi: products
// drop lo * lo, a few 2^-46 of the result.
__device__ __forceinline__ ds ds_mul_u(ds a, ds b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    return ds(p, __fmaf_rn(a.lo, b.hi, e));
}
__device__ __forceinline__ ds ds_add_u(ds a, ds b) {
    const ds s = two_sum(a.hi, b.hi);
    return ds(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ds ds_fma_u(ds a, ds b, ds c) {
    const ds p = ds_mul_u(a, b);
    const ds s = two_sum(p.hi, c.hi);
    return ds(s.hi, __fadd_rn(s.lo, __fadd_rn(p.lo, c.lo)));
}
__device__ __forceinline__ ds ds_norm(ds a) { return fast_two_sum(a.hi, a.lo); }

// 1/sqrt(x), x > 0 (x = 0 gives a non-finite value; callers mask it): the
// SFU estimate y of 1/sqrt(x.hi) (relative error below 2^-22) and one step of
// Halley's form y + y e (1/2 + 3/8 e), e = 1 - x y^2.  x.hi y = p + q exactly,
// and 1 - p y, of size 2^-21, loses only its own rounding (2^-45) in one fused
// operation, so e costs six operations instead of a double-single chain of 23.
__device__ __forceinline__ ds ds_rsqrt(ds x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x.hi));
    const float p = __fmul_rn(x.hi, y);
    const float q = __fmaf_rn(x.hi, y, -p);
    float e = __fmaf_rn(-p, y, 1.f);
    e = __fmaf_rn(-q, y, e);
    e = __fmaf_rn(-__fmul_rn(x.lo, y), y, e);
    return fast_two_sum(y, __fmul_rn(__fmul_rn(y, e), __fmaf_rn(0.375f, e, 0.5f)));
}

// 2^t for t < 127 (results below 2^-126 are returned as 0), table-driven
// (Tang's reduction, ACM TOMS 15, 1989): t = m / 64 + f with m = rint(64 t.hi)
// and |f| <= 1/128 (t.hi - m/64 is exact), so 2^t = 2^(m >> 6) 2^(j/64) e^s
// with j = m & 63 and s = f ln 2, |s| < 0.0055.  2^(j/64) comes from a 64-entry
// double-single table computed at compile time from the exponential series.
// e^s - 1 = s + s^2/2 + s^3 (1/6 + s/24 + s^2/120): s and s^2 with their error
// terms, the cubic tail (below 2.8e-8) in FP32, whose rounding is below 2e-15
// of the result; the truncation is below 4e-17.  35 FP32 operations (the
// Horner form with double-single steps took 75).
// e^x by its series, for the compile-time table (|x| < 1: 30 terms reach
// double rounding)
__host__ __device__ constexpr double exp_series(double x) {
    double s = 1.0, t = 1.0;
    for (int k = 1; k < 30; ++k) {
        t = t * x / k;
        s += t;
    }
    return s;
}
struct Exp2Table {
    ds v[64];
    __host__ __device__ constexpr Exp2Table() : v() {
        for (int j = 0; j < 64; ++j) v[j] = ds_const(exp_series(j * PGB_LN2 / 64.0));
    }
};
__device__ const Exp2Table kExp2Table = Exp2Table();

__device__ __forceinline__ ds ds_exp2(ds t) {
    constexpr ds ln2 = ds_const(PGB_LN2);
    const float mf = rintf(__fmul_rn(t.hi, 64.f));
    const int m = (int)mf;
    const float fe = __fmaf_rn(mf, -0.015625f, t.hi);  // exact; 0 or at least an ulp of t.hi
    const ds f = fast_two_sum(fe, t.lo);
    const float s = __fmul_rn(f.hi, ln2.hi);
    float sl = __fmaf_rn(f.hi, ln2.hi, -s);
    sl = __fmaf_rn(f.hi, ln2.lo, sl);
    sl = __fmaf_rn(f.lo, ln2.hi, sl);
    const float q = __fmul_rn(s, s);
    const float ql = __fmaf_rn(s, s, -q);  // s^2 = q + ql + 2 s sl
    float tail = __fmaf_rn(s, 1.f / 120.f, 1.f / 24.f);
    tail = __fmul_rn(__fmaf_rn(tail, s, 1.f / 6.f), __fmul_rn(s, q));
    const float a = __fmaf_rn(0.5f, q, s);
    float lo = __fmaf_rn(0.5f, q, -__fsub_rn(a, s));
    lo = __fadd_rn(__fadd_rn(lo, tail), __fmaf_rn(0.5f, ql, __fmaf_rn(s, sl, sl)));
    const float2 tv = __ldg(reinterpret_cast<const float2*>(&kExp2Table.v[m & 63]));
    const float p = __fmul_rn(tv.x, a);
    float pe = __fmaf_rn(tv.x, a, -p);
    pe = __fmaf_rn(tv.x, lo, pe);
    pe = __fmaf_rn(tv.y, a, pe);
    const float h = __fadd_rn(tv.x, p);  // |p| < |tv.x|
    const float l = __fadd_rn(__fsub_rn(p, __fsub_rn(h, tv.x)), __fadd_rn(pe, tv.y));
    const int n = m >> 6;  // floor(m / 64)
    if (n < -126) return ds(0);
    const float sc = __int_as_float((127 + n) << 23);
    return ds(__fmul_rn(h, sc), __fmul_rn(l, sc));
}

// e^x = 2^(x log2 e)
__device__ __forceinline__ ds ds_exp(ds x) {
    constexpr ds log2e = ds_const(1.44269504088896340735992468100189);
    return ds_exp2(x * log2e);
}

}  // namespace pgb
