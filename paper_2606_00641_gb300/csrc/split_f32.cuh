// split_f32.cuh -- more than single precision from FP32 operations.
//
// A GB300 SM issues 64 FP32 operations for every FP64 one, so the passes that
// need more than 24 bits per cell but read and write memory at full rate (the
// channel's initial populations and its moments) carry values as unevaluated
// sums of floats.  The error-free transformations are those of Dekker (1971,
// "A floating-point technique for extending the available precision") and
// Knuth (TAOCP vol. 2, sec. 4.2.2); products are split with a fused
// multiply-add.  Rounding intrinsics throughout, so that nothing is contracted
// or reordered.
#pragma once

namespace vlbm {

// s + e = a + b exactly, s = fl(a + b).
__device__ __forceinline__ float two_sum(float a, float b, float &e)
{
    const float s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
    return s;
}

// A running sum of floats in three floats: s takes the sum, e the rounding errors of
// s, r those of e.  Its value as a double carries at least the accuracy of adding the
// same floats in FP64.
struct Sum3 {
    float s = 0.f, e = 0.f, r = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        float d, d2;
        s = two_sum(s, x, d);
        e = two_sum(e, d, d2);
        r = __fadd_rn(r, d2);
    }
    // a term that overflows, an infinity or a NaN leaves s itself not finite
    __device__ __forceinline__ bool finite() const { return fabsf(s) <= 3.402823466e38f; }
    __device__ __forceinline__ double value() const { return (double)s + ((double)e + (double)r); }
};

// A value as hi + lo, |lo| at most half a unit in the last place of hi: about 46 bits.
struct Split {
    float hi, lo;
};

__device__ __forceinline__ Split split(double v)
{
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ Split renorm(float s, float e)  // |e| small against s
{
    const float h = __fadd_rn(s, e);
    return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ Split operator+(Split a, Split b)
{
    float e, f;
    const float s = two_sum(a.hi, b.hi, e);
    const float t = two_sum(a.lo, b.lo, f);
    const Split c = renorm(s, __fadd_rn(e, t));
    return renorm(c.hi, __fadd_rn(c.lo, f));
}
__device__ __forceinline__ Split operator-(Split a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ Split operator-(Split a, Split b) { return a + (-b); }
__device__ __forceinline__ Split operator*(Split a, Split b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
    return renorm(p, e);
}
// 1 / a: the FP32 quotient and one Newton correction with the residual in full.
__device__ __forceinline__ Split reciprocal(Split a)
{
    const float q = __fdiv_rn(1.f, a.hi);
    const float r = __fmaf_rn(-q, a.lo, __fmaf_rn(-q, a.hi, 1.f));
    return renorm(q, __fmul_rn(q, r));
}

// Whether a value within `off` (>= 0) of a rounds to a.hi whatever it is.
__device__ __forceinline__ bool rounds_surely(Split a, float off)
{
    return __fadd_rn(a.hi, __fadd_ru(a.lo, off)) == a.hi && __fadd_rn(a.hi, __fsub_rd(a.lo, off)) == a.hi;
}

}  // namespace vlbm
