// |a|^2 and its sums on the FP32 pipes, to no less than FP64's accuracy.
//
// GB300 has about two FP64 lanes per SM, so a probability computed in FP64
// costs more than the HBM time of its amplitude. Here the squares are taken
// exactly as high part and FMA remainder (the error-free product), and a
// thread sums them in three floats per component: the high parts, then the
// first sum's errors and the remainders, then the second sum's errors. The
// first two sums start at a large number (NormSum), so that the error of an
// addition is exact in two more operations (Dekker's FastTwoSum, Numer. Math.
// 18, 1971) whatever the order of magnitudes. What is dropped is below 2^-57
// of the largest square; the FP64 additions that join threads and blocks
// round as FP64 arithmetic does. Largest relative error of a norm in units of
// 2^-53 (complex64 and double-float, 256 states of one, three and ten nonzero
// amplitudes, random states of 2^11 to 2^20): one 1.6 (in FP64 2.0), three 3.0
// (3.0), ten 2.0 (2.0), random 2.0 (2.0). With the remainders and errors in
// one float, summed plainly, it was 69, 82, 34 and 16.
// re and im are the halves of packed operations: 13 per amplitude of
// complex64, 20 of double-float.
#pragma once
#include <cuda_runtime.h>

#include "packed.cuh"

namespace hisv {

// s + e = a + b exactly (Knuth, TAOCP vol. 2, 4.2.2).
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}
// re^2 and im^2 of an amplitude as -neg + rem; for a double-float one (hi, lo)
// with the cross terms 2 hi lo = -cross + small, small also holding lo^2.
struct Squares {
    float2 neg, rem;
    __device__ __forceinline__ explicit Squares(float2 v) {
        neg = mul2(make_float2(-v.x, -v.y), v);
        rem = fma2(v, v, neg);
    }
    // |a|^2 rounded to float, but for ties' neighbourhoods of 2^-22 ulp
    __device__ __forceinline__ float prob() const { return join(rem.x + rem.y); }
    // re^2 + im^2 + low; the sum of two numbers of known order is exact in two
    // more operations (Dekker)
    __device__ __forceinline__ float join(float low) const {
        const float a = -fminf(neg.x, neg.y), b = -fmaxf(neg.x, neg.y), s = __fadd_rn(a, b);
        return s + (__fsub_rn(b, __fsub_rn(s, a)) + low);
    }
    // within 2^-23 of it
    __device__ __forceinline__ float rough() const { return -(neg.x + neg.y); }
};
struct SquaresDf : Squares {
    float2 cross, small;
    __device__ __forceinline__ explicit SquaresDf(const float4 &v) : Squares(make_float2(v.x, v.z)) {
        const float2 hi = make_float2(v.x, v.z), lo = make_float2(v.y, v.w), two = add2(hi, hi);
        cross = mul2(make_float2(-two.x, -two.y), lo);
        small = fma2(lo, lo, fma2(two, lo, cross));
    }
    __device__ __forceinline__ float prob() const { return join((rem.x - cross.x) + (rem.y - cross.y)); }
    __device__ __forceinline__ float rough() const { return -((neg.x + cross.x) + (neg.y + cross.y)); }
};

// A thread's sum, re and im apart. lim: a power of two above every component
// of the warp so far. s starts at 3/2 of 2^5 lim^2, which the sum of PROB_SUM
// squares keeps within its binade, so s is never smaller than what is added to
// it; t at 3/2 of 2^-13 lim^2, likewise for the errors of s (2^-19 lim^2 each)
// and the remainders (2^-24, of double-floats also 2^-21). What u rounds off
// is below 2^-60 lim^2 a time (with sums of 64 2^-56: an amplitude alone was
// off by up to 1.3 instead of 1.0 units of 2^-53).
constexpr int PROB_SUM = 16;
struct NormSum {
    float lim = 0x1p-46f;
    float2 s, t, u;
    __device__ __forceinline__ float s0() const { return 48.0f * lim * lim; }
    __device__ __forceinline__ float t0() const { return 0x1.8p-13f * lim * lim; }
    __device__ __forceinline__ NormSum() { clear(); }
    __device__ __forceinline__ void clear() {
        s = make_float2(s0(), s0());
        t = make_float2(t0(), t0());
        u = make_float2(0.0f, 0.0f);
    }
    // a += b, with the error of the addition; |a| >= |b|
    __device__ __forceinline__ static float2 fast(float2 &a, float2 b) {
        const float2 n = add2(a, b), e = sub2(b, sub2(n, a));
        a = n;
        return e;
    }
    __device__ __forceinline__ void add(const Squares &q) {
        const float2 e = fast(s, make_float2(-q.neg.x, -q.neg.y));
        u = add2(u, fast(t, e));
        u = add2(u, fast(t, q.rem));
    }
    __device__ __forceinline__ void add(const SquaresDf &q) {
        add(static_cast<const Squares &>(q));
        u = add2(u, fast(t, make_float2(-q.cross.x, -q.cross.y)));
        u = add2(u, q.small);
    }
    // the sum in FP64, reset: after at most PROB_SUM amplitudes
    __device__ __forceinline__ double take() {
        const float a = s0(), b = t0();
        float e, f, g;   // joined in FP32: three conversions and two FP64 additions
        const float hi = two_sum(s.x - a, s.y - a, e);
        const float lo = two_sum(two_sum(t.x - b, t.y - b, f), e, g);
        const double d = (double)hi + ((double)lo + (double)((f + g) + (u.x + u.y)));
        clear();
        return d;
    }
    // Whether the split takes the amplitudes of v, one test for all. The
    // remainders are exact to 2^-150 and nothing overflows while the larger
    // component of an amplitude is zero or in [2^-46, 2^56) and a double-float
    // pair normalised (|lo| within 2^-22 |hi|); other amplitudes (and
    // infinities) go through FP64. A NaN may take either path: both give NaN.
    // Where one of the warp's (all lanes call this together) is not below lim
    // yet, lim grows and the sums so far join acc: about once a warp (a limit
    // of each thread's own grew in most of a warp's first rounds, 25 us more
    // at 2^25 amplitudes).
    template <bool DF, int U> __device__ __forceinline__ bool fits(const float4 (&v)[U], double &acc) {
        float top = 0.0f;
        uint32_t low = ~0u;   // bits of the smallest larger component less 1: zeros wrap to the top
        bool norm = true;
        auto amp = [&](float x, float y) {
            const float m = fmaxf(fabsf(x), fabsf(y));
            top = fmaxf(top, m);
            low = min(low, __float_as_uint(m) - 1u);
        };
#pragma unroll
        for (int u = 0; u < U; u++) {
            if constexpr (DF) {
                amp(v[u].x, v[u].z);
                norm = norm && fabsf(v[u].y) <= 0x1p-22f * fabsf(v[u].x) && fabsf(v[u].w) <= 0x1p-22f * fabsf(v[u].z);
            } else {
                amp(v[u].x, v[u].y);
                amp(v[u].z, v[u].w);
            }
        }
        const bool exact = norm && low >= 0x28800000u - 1u;   // 2^-46
        if (__all_sync(0xffffffffu, exact && top < lim)) return true;
        const bool ok = exact && top < 0x1p56f;
        float most = ok ? top : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, o));
        if (most >= lim) {
            if (lim > 0x1p-46f) acc += take();   // else only zeros so far
            lim = __uint_as_float((__float_as_uint(most) & 0x7f800000u) + 0x00800000u);   // 2^e <= most: 2^(e + 1)
            clear();
        }
        return ok;
    }
};

}  // namespace hisv
