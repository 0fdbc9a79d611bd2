// Double-float arithmetic shared by the field kernels.
#pragma once
#include "gp_common.cuh"

namespace gp {
namespace {

// A value carried as an unevaluated sum hi + lo of two FP32 numbers (about 48
// significant bits; Dekker 1971, Knuth's two-sum). The per-point sums of the
// density and its force run in this form: a few FP32 instructions replace an
// FP64 instruction that costs 64 FP32 issue slots on this GPU.
struct df { float hi, lo; };

__device__ __forceinline__ df df_from(double v) {
    const float2 p = split_to_float2(v);      // the casts' result, without the FP64 pipe
    return {p.x, p.y};
}
__device__ __forceinline__ double df_to(df a) { return f32_to_f64(a.hi) + f32_to_f64(a.lo); }
__device__ __forceinline__ df as_df(float2 v) { return df{v.x, v.y}; }

// (s, c): a compensated pair (value s + c) summed across the warp in place (Knuth two-sum per step)
__device__ __forceinline__ void warp_sum_df(float& s, float& c) {
    for (int o = 16; o > 0; o >>= 1) {
        const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
        const float c2 = __shfl_xor_sync(0xffffffffu, c, o);
        const float t = s + s2;
        const float z = t - s;
        c += c2 + ((s - (t - z)) + (s2 - z));
        s = t;
    }
}

__device__ __forceinline__ df df_quick(float s, float e) {   // |s| >= |e|
    const float t = s + e;
    return {t, e - (t - s)};
}
__device__ __forceinline__ df df_mul(df a, df b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df_quick(p, e);
}
__device__ __forceinline__ df df_add(df a, df b) {
    const float s = a.hi + b.hi;
    const float v = s - a.hi;
    float e = (a.hi - (s - v)) + (b.hi - v);
    e += a.lo + b.lo;
    return df_quick(s, e);
}

// s += a * b with the product formed exactly to ~2^-48 (df64) and the sum
// compensated (Neumaier): the FP32 pipe does the work of an FP64 FMA.
__device__ __forceinline__ void df_acc(float& s, float& c, df a, df b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    const float t = s + p;
    const float z = t - s;
    c += ((s - (t - z)) + (p - z)) + e;
    s = t;
}

// the same, renormalised after every term: c stays below half an ulp of s, so a long sum of one
// sign loses 2^-48 of itself a term (with a growing c it loses that times the number of terms)
__device__ __forceinline__ void df_acc_norm(float& s, float& c, df a, df b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    const float t = s + p;
    const float z = t - s;
    e += ((s - (t - z)) + (p - z)) + c;
    s = t + e;
    c = e - (s - t);
}

}  // namespace
}  // namespace gp
