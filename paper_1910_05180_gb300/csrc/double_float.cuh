// double_float.cuh -- pairs of FP32 numbers as one value, for the diagnostics and
// the constant-volume sums: GB300 issues FP64 at 1/64 of the FP32 rate.
#pragma once

#include <math.h>

namespace spfm {

// ---- double-float arithmetic: a value is hi + lo in two FP32 numbers with
// |lo| <= ulp(hi)/2 (Dekker, Numer. Math. 18, 1971; Knuth, TAOCP 2, 4.2.2).
// About 48 significant bits at the FP32 rate, 64 times the FP64 rate of this
// GPU.  The error-free transforms use the _rn intrinsics, which the compiler
// neither contracts into FMAs nor reassociates.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ DF df_two_sum(float a, float b)   // a + b exactly
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ DF df_fast_sum(float a, float b)  // a + b exactly, |a| >= |b| or a = 0
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DF df_two_prod(float a, float b)  // a b exactly
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
// a + b with absolute error about 2^-48 max(|a|, |b|)
__device__ __forceinline__ DF df_add(DF a, DF b)
{
    const DF s = df_two_sum(a.hi, b.hi);
    return df_fast_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
// a + b with the low parts also added error-free, for running sums
__device__ __forceinline__ DF df_add_acc(DF a, DF b)
{
    DF s = df_two_sum(a.hi, b.hi);
    const DF t = df_two_sum(a.lo, b.lo);
    s = df_fast_sum(s.hi, __fadd_rn(s.lo, t.hi));
    return df_fast_sum(s.hi, __fadd_rn(s.lo, t.lo));
}
__device__ __forceinline__ DF df_neg(DF a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ DF df_mul(DF a, DF b)
{
    const DF p = df_two_prod(a.hi, b.hi);
    return df_fast_sum(p.hi, __fadd_rn(p.lo, __fmaf_rn(a.hi, b.lo, __fmul_rn(a.lo, b.hi))));
}
__device__ __forceinline__ DF df_mul_f(DF a, float b)
{
    const DF p = df_two_prod(a.hi, b);
    return df_fast_sum(p.hi, __fmaf_rn(a.lo, b, p.lo));
}
// a / b, b.hi not 0: the FP32 quotient and two corrections of its remainder
__device__ __forceinline__ DF df_div(DF a, DF b)
{
    const float r = __fdividef(1.0f, b.hi);
    const float q0 = __fmul_rn(a.hi, r);
    const DF p = df_two_prod(q0, b.hi);
    const float e0 = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p.hi), p.lo), __fmaf_rn(-q0, b.lo, a.lo));
    const float q1 = __fmul_rn(e0, r);
    const float e1 = __fmaf_rn(-q1, b.lo, __fmaf_rn(-q1, b.hi, e0));
    const DF q = df_fast_sum(q0, q1);
    return df_fast_sum(q.hi, __fmaf_rn(e1, r, q.lo));
}
__host__ __device__ __forceinline__ DF df_of(double x)
{
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_to_double(DF a) { return (double)a.hi + (double)a.lo; }
// an integer index as an exact pair (|n| < 2^48)
__device__ __forceinline__ DF df_of_int(int n)
{
    const float h = (float)n;
    return {h, (float)(n - (int)h)};
}
// sqrt of a non-negative value: the FP32 root s and one Newton step,
// s + (a - s^2) / (2 s), with s^2 formed exactly
__device__ __forceinline__ DF df_sqrt(DF a)
{
    if (!(a.hi > 0.0f)) return {0.0f, 0.0f};
    const float s = sqrtf(a.hi);
    const DF s2 = df_two_prod(s, s);
    const float r = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, s2.hi), s2.lo), a.lo);
    // the correction is about 2^-24 of s: an approximate reciprocal keeps the pair's accuracy
    return df_fast_sum(s, __fmul_rn(r, __fdividef(0.5f, s)));
}

}  // namespace spfm
