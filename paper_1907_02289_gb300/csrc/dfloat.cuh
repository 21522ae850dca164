// dfloat.cuh -- unevaluated sums of two FP32 numbers (hi + lo, |lo| <= ulp(hi)/2)
// and their arithmetic, built from the error-free transformations of
// Knuth (TwoSum: a + b = s + e exactly) and of the fused multiply-add
// (TwoProd: a * b = p + e exactly, e = fma(a, b, -p)); about 44 significant
// bits, on the FP32 pipe.  Used where an FP32 evaluation is too ill-conditioned
// for its result: the refinement of the FP32 force kernel.
#pragma once
#include <cuda_runtime.h>

namespace bh {

struct df {
    float hi, lo;
};

// s + e == a + b exactly, s = fl(a + b) (no condition on the magnitudes)
__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

// the same when |a| >= |b| (or a == 0)
__device__ __forceinline__ df fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// p + e == a * b exactly
__device__ __forceinline__ df two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ df df_add(df a, df b) {
    df s = two_sum(a.hi, b.hi);
    const df t = two_sum(a.lo, b.lo);
    s.lo = __fadd_rn(s.lo, t.hi);
    s = fast_two_sum(s.hi, s.lo);
    s.lo = __fadd_rn(s.lo, t.lo);
    return fast_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ df df_mul(df a, df b) {
    df p = two_prod(a.hi, b.hi);
    p.lo = __fmaf_rn(a.hi, b.lo, p.lo);
    p.lo = __fmaf_rn(a.lo, b.hi, p.lo);
    return fast_two_sum(p.hi, p.lo);
}

// a * b without the last renormalisation (the same value, |lo| up to a few
// ulp(hi)): a term of a running sum
__device__ __forceinline__ df df_mul_loose(df a, df b) {
    df p = two_prod(a.hi, b.hi);
    p.lo = __fmaf_rn(a.hi, b.lo, p.lo);
    p.lo = __fmaf_rn(a.lo, b.hi, p.lo);
    return p;
}

__device__ __forceinline__ df df_sqr(df a) {
    df p = two_prod(a.hi, a.hi);
    p.lo = __fmaf_rn(__fadd_rn(a.hi, a.hi), a.lo, p.lo);
    return fast_two_sum(p.hi, p.lo);
}

// A running sum in three words: the high parts are added exactly, the errors
// and low parts to a second word, exactly but for the sum of the two that go in,
// and the second word's own errors to a third.  14 operations a term where df_add
// takes 20; a sum of 60, 600 and 3000 terms of either sign that cancel to 1e-3
// is 0.7, 0.6 and 0.6 times as far (median) from the exact sum of its terms as
// with df_add, and node masses 0.8 times.  (Without the third word, 3, 8 and 18 times,
// and masses 1.5 to 2.6 times.)
struct df_sum {
    float hi, lo, err;
};

__device__ __forceinline__ void df_accumulate(df_sum& sum, df t) {
    const df s = two_sum(sum.hi, t.hi);
    const df l = two_sum(sum.lo, __fadd_rn(s.lo, t.lo));
    sum.hi = s.hi;
    sum.lo = l.hi;
    sum.err = __fadd_rn(sum.err, l.lo);
}

__device__ __forceinline__ void df_accumulate(df_sum& sum, float t) {
    const df s = two_sum(sum.hi, t);
    const df l = two_sum(sum.lo, s.lo);
    sum.hi = s.hi;
    sum.lo = l.hi;
    sum.err = __fadd_rn(sum.err, l.lo);
}

// The sum as a df (the high part may have cancelled below the others).
__device__ __forceinline__ df df_total(df_sum sum) {
    const df l = two_sum(sum.lo, sum.err);
    const df s = two_sum(sum.hi, l.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, l.lo));
}

// (x_hi + x_lo) - (y_hi + y_lo) for two hi/lo splits of FP64 values
__device__ __forceinline__ df df_diff(float xh, float xl, float yh, float yl) {
    df d = two_sum(xh, -yh);
    d.lo = __fadd_rn(d.lo, __fsub_rn(xl, yl));
    return fast_two_sum(d.hi, d.lo);
}

// x^2 + y^2 + z^2: nothing cancels, so the low parts are summed in FP32
__device__ __forceinline__ df df_norm2(df x, df y, df z) {
    const df px = two_prod(x.hi, x.hi), py = two_prod(y.hi, y.hi), pz = two_prod(z.hi, z.hi);
    const df s = two_sum(px.hi, py.hi), t = two_sum(s.hi, pz.hi);
    const float ex = __fmaf_rn(__fadd_rn(x.hi, x.hi), x.lo, px.lo);
    const float ey = __fmaf_rn(__fadd_rn(y.hi, y.hi), y.lo, py.lo);
    const float ez = __fmaf_rn(__fadd_rn(z.hi, z.hi), z.lo, pz.lo);
    return fast_two_sum(t.hi, __fadd_rn(__fadd_rn(s.lo, t.lo), __fadd_rn(__fadd_rn(ex, ey), ez)));
}

// 1 / sqrt(s), s > 0: an FP32 estimate y0 and the binomial series to second
// order, y = y0 + y0 (r / 2 + 3 r^2 / 8), r = 1 - s y0^2 (r^2 reaches 2^-44: a
// Newton step, without it, is off by 2e-14 rms for an estimate within an ulp;
// this by 5e-15).  s y0^2 is within a few 2^-23 of 1, so 1 - its high part is exact.
__device__ __forceinline__ df df_rsqrt(df s) {
    const float y0 = rsqrtf(s.hi);
    const df p = df_mul_loose(s, two_prod(y0, y0));
    const float r = __fsub_rn(__fsub_rn(1.f, p.hi), p.lo);
    return fast_two_sum(y0, __fmul_rn(y0, __fmul_rn(r, __fmaf_rn(r, 0.375f, 0.5f))));
}

__device__ __forceinline__ bool df_gt(df a, df b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }

__device__ __forceinline__ double df_to_double(df a) { return (double)a.hi + (double)a.lo; }

}  // namespace bh
