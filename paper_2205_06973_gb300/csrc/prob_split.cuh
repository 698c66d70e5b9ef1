// |a|^2 on the FP32 pipes as an unevaluated sum of two floats.
//
// GB300 has about two FP64 lanes per SM, so a probability computed in FP64
// costs more than the HBM time of its amplitude. Here the squares are taken
// exactly as high part and FMA remainder (the error-free product), added
// with Knuth's error-free TwoSum, and only the remainders' sum is rounded:
// hi + lo is |a|^2 to about 2^-48, hi + lo rounded to float is the float that
// FP64 arithmetic gives (but for a tie's neighbourhood of 2^-24 ulp), and the
// roundings of lo are unbiased, so that a norm of 2^11 and more amplitudes
// keeps the accuracy of its final FP64 sums (measured: the same to the last
// bits of the FP64 kernels' norm).
#pragma once
#include <cuda_runtime.h>

namespace hisv {

// The remainders are exact and nothing overflows while the larger component
// of an amplitude is zero or in [2^-50, 2^60); other amplitudes (and
// infinities) go through FP64. A NaN may take either path: both give NaN.
__device__ __forceinline__ bool split_range1(float x, float y) {
    const float m = fmaxf(fabsf(x), fabsf(y));
    return m < 0x1p60f && (m >= 0x1p-50f || m == 0.0f);
}
// A double-float pair is taken as normalised (|lo| within 2^-22 |hi|).
template <bool DF>
__device__ __forceinline__ bool split_range(const float4 &v) {
    if constexpr (DF)
        return split_range1(v.x, v.z) && fabsf(v.y) <= 0x1p-22f * fabsf(v.x) && fabsf(v.w) <= 0x1p-22f * fabsf(v.z);
    else return split_range1(v.x, v.y) && split_range1(v.z, v.w);
}

// s + e = a + b exactly (Knuth, TAOCP vol. 2, 4.2.2).
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// x^2 + y^2 as (hi, lo).
__device__ __forceinline__ float2 split_prob(float x, float y) {
    const float h = __fmul_rn(x, x), k = __fmul_rn(y, y);   // never contracted into the sum below
    const float r = fmaf(x, x, -h), t = fmaf(y, y, -k);
    float e;
    const float s = two_sum(h, k, e);
    return make_float2(s, e + (r + t));
}

// The same for a double-float amplitude (re.hi, re.lo, im.hi, im.lo): the
// cross terms 2 hi lo join the remainders, lo^2 (below 2^-48) is dropped.
__device__ __forceinline__ float2 split_prob_df(const float4 &v) {
    const float h = __fmul_rn(v.x, v.x), k = __fmul_rn(v.z, v.z);
    const float r = fmaf(2.0f * v.x, v.y, fmaf(v.x, v.x, -h)), t = fmaf(2.0f * v.z, v.w, fmaf(v.z, v.z, -k));
    float e;
    const float s = two_sum(h, k, e);
    return make_float2(s, e + (r + t));
}

// (S, T) += p: high parts by TwoSum, its error and the low part into T.
__device__ __forceinline__ void split_add(float &S, float &T, float2 p) {
    float e;
    S = two_sum(S, p.x, e);
    T += e + p.y;
}

}  // namespace hisv
