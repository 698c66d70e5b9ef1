// sm_103a kernels of the hierarchical state-vector simulator.
//
//  k_gate1 / k_gate2 : the plain per-gate pass of Sec. III-A (comparator).
//  k_probs / k_sum   : |a_x|^2 and the norm with FP64 accumulation.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "kernels.hpp"
#include "ops.cuh"
#include "prob_split.cuh"

namespace hisv {

// ------------------------------------------------------------------------
// plain per-gate kernels
// ------------------------------------------------------------------------
template <typename Real> struct M2 { Real m[8]; };
template <typename Real> struct M4 { Real m[32]; };

template <typename Real>
__global__ void __launch_bounds__(256) k_gate1(typename CT<Real>::T *__restrict__ sv, int q, uint64_t npairs,
                                                const __grid_constant__ M2<Real> g) {
    typedef typename CT<Real>::T C;
    const uint64_t lomask = (1ull << q) - 1;
    for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < npairs;
         p += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t x0 = ((p & ~lomask) << 1) | (p & lomask);
        const uint64_t x1 = x0 | (1ull << q);
        const C x = sv[x0], y = sv[x1];
        C u, v;
        u.x = g.m[0] * x.x - g.m[1] * x.y + g.m[2] * y.x - g.m[3] * y.y;
        u.y = g.m[0] * x.y + g.m[1] * x.x + g.m[2] * y.y + g.m[3] * y.x;
        v.x = g.m[4] * x.x - g.m[5] * x.y + g.m[6] * y.x - g.m[7] * y.y;
        v.y = g.m[4] * x.y + g.m[5] * x.x + g.m[6] * y.y + g.m[7] * y.x;
        sv[x0] = u;
        sv[x1] = v;
    }
}

template <typename Real>
__global__ void __launch_bounds__(256) k_gate2(typename CT<Real>::T *__restrict__ sv, int q0, int q1,
                                                uint64_t nquads, const __grid_constant__ M4<Real> g) {
    typedef typename CT<Real>::T C;
    const int lo = q0 < q1 ? q0 : q1, hi = q0 < q1 ? q1 : q0;
    const uint64_t m_lo = (1ull << lo) - 1, m_hi = (1ull << hi) - 1;
    for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nquads;
         p += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t x = ((p & ~m_lo) << 1) | (p & m_lo);   // insert a zero bit at lo
        x = ((x & ~m_hi) << 1) | (x & m_hi);              // then at hi
        uint64_t idx[4];
        idx[0] = x;
        idx[1] = x | (1ull << q0);
        idx[2] = x | (1ull << q1);
        idx[3] = x | (1ull << q0) | (1ull << q1);
        C in[4];
#pragma unroll
        for (int l = 0; l < 4; l++) in[l] = sv[idx[l]];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            Real re = 0, im = 0;
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const Real mr = g.m[2 * (4 * r + c)], mi = g.m[2 * (4 * r + c) + 1];
                re += mr * in[c].x - mi * in[c].y;
                im += mr * in[c].y + mi * in[c].x;
            }
            C o;
            o.x = re;
            o.y = im;
            sv[idx[r]] = o;
        }
    }
}

static unsigned grid_for(uint64_t work, int threads) {
    uint64_t b = (work + threads - 1) / threads;
    const uint64_t cap = 152ull * 16;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

cudaError_t launch_gate1(bool fp64, void *sv, int n, int q, const double *m, cudaStream_t st) {
    const uint64_t np = 1ull << (n - 1);
    if (!fp64) {
        M2<float> g;
        for (int i = 0; i < 8; i++) g.m[i] = (float)m[i];
        k_gate1<float><<<grid_for(np, 256), 256, 0, st>>>((float2 *)sv, q, np, g);
    } else {
        M2<double> g;
        for (int i = 0; i < 8; i++) g.m[i] = m[i];
        k_gate1<double><<<grid_for(np, 256), 256, 0, st>>>((double2 *)sv, q, np, g);
    }
    return cudaGetLastError();
}

cudaError_t launch_gate2(bool fp64, void *sv, int n, int q0, int q1, const double *m, cudaStream_t st) {
    const uint64_t nq = 1ull << (n - 2);
    if (!fp64) {
        M4<float> g;
        for (int i = 0; i < 32; i++) g.m[i] = (float)m[i];
        k_gate2<float><<<grid_for(nq, 256), 256, 0, st>>>((float2 *)sv, q0, q1, nq, g);
    } else {
        M4<double> g;
        for (int i = 0; i < 32; i++) g.m[i] = m[i];
        k_gate2<double><<<grid_for(nq, 256), 256, 0, st>>>((double2 *)sv, q0, q1, nq, g);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------------
// probabilities and norm
// ------------------------------------------------------------------------
// Real and imaginary part of a stored amplitude, in FP64: complex64
// (float2), complex128 (double2) or double-float complex128 (float4: re.hi,
// re.lo, im.hi, im.lo; each part is the sum of its two floats).
__device__ __forceinline__ void amp_parts(const float2 &v, double &re, double &im) {
    re = (double)v.x;
    im = (double)v.y;
}
__device__ __forceinline__ void amp_parts(const double2 &v, double &re, double &im) {
    re = v.x;
    im = v.y;
}
__device__ __forceinline__ void amp_parts(const float4 &v, double &re, double &im) {
    re = (double)v.x + (double)v.y;
    im = (double)v.z + (double)v.w;
}

// The sum of a block's FP64 partials into partials[blockIdx.x]; the block that
// ends last (ticket: blocks done, back at zero afterwards) also adds all
// partials up, in the same order as k_sum, and writes the norm: one launch
// less per measurement. ticket null: k_sum follows.
__device__ __forceinline__ bool last_block(uint32_t *ticket, uint32_t &flag) {
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t t = atomicAdd(ticket, 1u);
        flag = t + 1 == gridDim.x;
        if (flag) {
            *ticket = 0u;
            __threadfence();
        }
    }
    __syncthreads();
    return flag != 0;
}

// 256 threads: the sum of v[0..nb) in a fixed order, valid in thread 0.
__device__ __forceinline__ double sum_partials(const double *v, int nb, double *red) {
    double s = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) s += __ldcg(v + i);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    return red[0];
}

__device__ __forceinline__ void finish_norm(double acc, double *partials, uint32_t *ticket, double *out) {
    __shared__ double red[256];
    __shared__ uint32_t flag;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += red[w];
        partials[blockIdx.x] = s;
    }
    if (!ticket || !last_block(ticket, flag)) return;
    const double s = sum_partials(partials, gridDim.x, red);
    if (threadIdx.x == 0) *out = s;
}

template <typename E, typename Out>
__global__ void __launch_bounds__(256) k_probs(const E *__restrict__ sv, uint64_t N, Out *__restrict__ out,
                                                double *__restrict__ partials, uint32_t *ticket, double *norm) {
    double acc = 0.0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (uint64_t)gridDim.x * blockDim.x) {
        const E v = __ldcs(sv + i);
        double re, im;
        amp_parts(v, re, im);
        const double p = re * re + im * im;
        if (out) out[i] = (Out)p;
        acc += p;
    }
    finish_norm(acc, partials, ticket, norm);
}

__global__ void k_sum(const double *__restrict__ partials, int nb, double *__restrict__ out) {
    __shared__ double red[256];
    const double s = sum_partials(partials, nb, red);
    if (threadIdx.x == 0) *out = s;
}

// k_probs_fast: the same for float outputs of complex64 and double-float
// states, on the FP32 pipes (prob_split.cuh). In FP64 the two conversions,
// the product, the multiply-add and the add of an amplitude made the kernel
// FP64-bound on a GPU with ~2 FP64 lanes per SM (2^28 complex64 amplitudes:
// 3.05 ms against 0.47 ms of HBM time for the 3.2 GB; 0.49 ms here).
// Each thread takes 16 bytes at a time, U of them in flight, and sends the
// FP64 pipe three conversions and three adds per PROB_SUM amplitudes at most.
// Probabilities leave with streaming stores. Two loads and six blocks per SM:
// 469 us of kernel; two loads and plain stores 494, four loads and four blocks
// 492, eight and two 478. Four loads and four blocks up to 2^25 amplitudes
// (63 us of kernel there against 68; 2^20: 19.7 us a call against 22.5) and
// for double-floats (2^27: 450 us a call against 466).
constexpr int SUMMARY_U = 4;   // loads in flight per thread of k_summary_fast

template <bool DF, int U, int BLOCKS>
__global__ void __launch_bounds__(256, BLOCKS)
k_probs_fast(const float4 *__restrict__ sv, uint64_t n_chunks, float *__restrict__ out, double *__restrict__ partials,
             uint32_t *ticket, double *norm) {
    double acc = 0.0;
    NormSum sum;
    uint32_t it = 0;
    for (uint64_t c = blockIdx.x; c < n_chunks; c += gridDim.x) {
        const uint64_t at = c * (256 * U) + threadIdx.x;
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = __ldcs(sv + at + 256 * u);
        if (sum.fits<DF>(v, acc)) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                if constexpr (DF) {
                    const SquaresDf q(v[u]);
                    sum.add(q);
                    if (out) __stcs(out + at + 256 * u, q.prob());
                } else {
                    const Squares q(make_float2(v[u].x, v[u].y)), r(make_float2(v[u].z, v[u].w));
                    sum.add(q);
                    sum.add(r);
                    if (out) __stcs(reinterpret_cast<float2 *>(out) + at + 256 * u, make_float2(q.prob(), r.prob()));
                }
            }
        } else {   // outside the split's range: FP64
#pragma unroll
            for (int u = 0; u < U; u++) {
                if constexpr (DF) {
                    double re, im;
                    amp_parts(v[u], re, im);
                    const double p = re * re + im * im;
                    if (out) out[at + 256 * u] = (float)p;
                    acc += p;
                } else {
                    const double p = (double)v[u].x * v[u].x + (double)v[u].y * v[u].y;
                    const double q = (double)v[u].z * v[u].z + (double)v[u].w * v[u].w;
                    if (out) reinterpret_cast<float2 *>(out)[at + 256 * u] = make_float2((float)p, (float)q);
                    acc += p;
                    acc += q;
                }
            }
        }
        if (++it % (PROB_SUM / ((DF ? 1 : 2) * U)) == 0) acc += sum.take();
    }
    finish_norm(acc + sum.take(), partials, ticket, norm);
}

template <bool DF, int U, int BLOCKS>
static int probs_fast(const void *sv, uint64_t loads, void *out, double *partials, int nblocks, uint32_t *ticket,
                      double *d_norm, cudaStream_t st) {
    const uint64_t chunks = loads / (256 * U), wave = std::min<uint64_t>(nblocks, 152 * BLOCKS);
    const int nb = (int)std::min(chunks, wave);
    k_probs_fast<DF, U, BLOCKS><<<nb, 256, 0, st>>>((const float4 *)sv, chunks, (float *)out, partials, ticket, d_norm);
    return nb;
}

// The FP32 kernels take whole chunks of at most 1024 16-byte loads, and an output of pairs aligned to 8 bytes (one float per load otherwise).
static bool fast_prob_ok(const void *sv, uint64_t N, bool fp64, bool df, int out_fp64, const void *out) {
    const uint64_t loads = df ? N : N / 2;
    return (!fp64 || df) && !(out && out_fp64) && loads >= 1024 &&
           (reinterpret_cast<uintptr_t>(sv) & 15) == 0 && (df || (reinterpret_cast<uintptr_t>(out) & 7) == 0);
}
cudaError_t launch_probs(bool fp64, const void *sv, int n, void *out, int out_fp64, double *partials,
                         int nblocks, double *d_norm, cudaStream_t st, bool df, uint32_t *ticket) {
    const uint64_t N = 1ull << n;
    uint64_t need = (N + 255) / 256;
    int nb = (int)(need < (uint64_t)nblocks ? need : (uint64_t)nblocks);
    if (nb < 1) nb = 1;
    if (fast_prob_ok(sv, N, fp64, df, out_fp64, out)) {
        const uint64_t loads = df ? N : N / 2;
        nb = df ? probs_fast<true, 4, 4>(sv, loads, out, partials, nblocks, ticket, d_norm, st)
             : loads <= 1ull << 24 ? probs_fast<false, 4, 4>(sv, loads, out, partials, nblocks, ticket, d_norm, st)
                                             : probs_fast<false, 2, 6>(sv, loads, out, partials, nblocks, ticket, d_norm, st);
    } else if (df) {
        if (out_fp64) k_probs<float4, double><<<nb, 256, 0, st>>>((const float4 *)sv, N, (double *)out, partials, ticket, d_norm);
        else k_probs<float4, float><<<nb, 256, 0, st>>>((const float4 *)sv, N, (float *)out, partials, ticket, d_norm);
    } else if (!fp64) {
        if (out_fp64) k_probs<float2, double><<<nb, 256, 0, st>>>((const float2 *)sv, N, (double *)out, partials, ticket, d_norm);
        else k_probs<float2, float><<<nb, 256, 0, st>>>((const float2 *)sv, N, (float *)out, partials, ticket, d_norm);
    } else {
        if (out_fp64) k_probs<double2, double><<<nb, 256, 0, st>>>((const double2 *)sv, N, (double *)out, partials, ticket, d_norm);
        else k_probs<double2, float><<<nb, 256, 0, st>>>((const double2 *)sv, N, (float *)out, partials, ticket, d_norm);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || ticket) return e;
    k_sum<<<1, 256, 0, st>>>(partials, nb, d_norm);
    return cudaGetLastError();
}

// Summary of the probability distribution without writing it: per block the
// FP64 sum of |a_x|^2 and the largest |a_x|^2 with its index (ties to the
// smaller index); the block that ends last combines them.
__device__ __forceinline__ void better(double &p, uint64_t &i, double q, uint64_t j) {
    if (q > p || (q == p && j < i)) {
        p = q;
        i = j;
    }
}

// out[0] = sum |a|^2, out[1] = |a_0|^2, out[2] = max |a_x|^2, out[3] = its index (bits)
template <typename E>
__device__ __forceinline__ void finish_summary(const E *sv, double acc, double best, uint64_t bi, double *sums,
                                               double *maxs, uint64_t *idxs, uint32_t *ticket, double *out) {
    __shared__ double rs[256], rm[256];
    __shared__ uint64_t ri[256];
    __shared__ uint32_t flag;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const double q = __shfl_xor_sync(0xffffffffu, best, o);
        const uint64_t j = __shfl_xor_sync(0xffffffffu, bi, o);
        better(best, bi, q, j);
    }
    if ((threadIdx.x & 31) == 0) {
        rs[threadIdx.x >> 5] = acc;
        rm[threadIdx.x >> 5] = best;
        ri[threadIdx.x >> 5] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0, m = -1.0;
        uint64_t mi = ~0ull;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            s += rs[w];
            better(m, mi, rm[w], ri[w]);
        }
        sums[blockIdx.x] = s;
        maxs[blockIdx.x] = m;
        idxs[blockIdx.x] = mi;
    }
    if (!last_block(ticket, flag)) return;
    double s = 0.0, m = -1.0;
    uint64_t mi = ~0ull;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        s += __ldcg(sums + i);
        better(m, mi, __ldcg(maxs + i), __ldcg(reinterpret_cast<const unsigned long long *>(idxs) + i));
    }
    rs[threadIdx.x] = s;
    rm[threadIdx.x] = m;
    ri[threadIdx.x] = mi;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            rs[threadIdx.x] += rs[threadIdx.x + w];
            better(rm[threadIdx.x], ri[threadIdx.x], rm[threadIdx.x + w], ri[threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double re, im;
        amp_parts(sv[0], re, im);
        out[0] = rs[0];
        out[1] = re * re + im * im;
        out[2] = rm[0];
        out[3] = __longlong_as_double((long long)ri[0]);
    }
}

template <typename E>
__global__ void __launch_bounds__(256) k_summary(const E *__restrict__ sv, uint64_t N,
                                                  double *__restrict__ sums, double *__restrict__ maxs,
                                                  uint64_t *__restrict__ idxs, uint32_t *ticket, double *out) {
    double acc = 0.0, best = -1.0;
    uint64_t bi = ~0ull;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (uint64_t)gridDim.x * blockDim.x) {
        const E v = __ldcs(sv + i);
        double re, im;
        amp_parts(v, re, im);
        const double p = re * re + im * im;
        acc += p;
        better(best, bi, p, i);
    }
    finish_summary(sv, acc, best, bi, sums, maxs, idxs, ticket, out);
}

// The norm on the FP32 pipes as in k_probs_fast. The maximum stays exact: an
// amplitude goes through the FP64 comparison only if its FP32 probability
// (within 2^-22 of the true one) comes within 2^-21 of the warp's largest so
// far, so nothing that could win or tie is passed over. For random states
// that is a few amplitudes per warp (2^28 complex64 amplitudes: 3.57 ms with
// every amplitude in FP64, against 0.32 ms of HBM time; 2^25: 0.48 ms, 0.16 ms
// with whole groups of loads in FP64, 0.074 ms here); for a state of equal
// probabilities it is every amplitude, as before. At most 48 registers for
// complex64: a block then fits on an SM beside a block of a tensor-core pass
// (53,248 of 65,536 registers), so that the summary of one state need not wait
// for the end of another's long pass.
constexpr int summary_blocks(bool df) { return df ? 4 : 5; }   // per SM
template <bool DF>
__global__ void __launch_bounds__(256, summary_blocks(DF))
k_summary_fast(const float4 *__restrict__ sv, uint64_t n_chunks, double *__restrict__ sums, double *__restrict__ maxs,
               uint64_t *__restrict__ idxs, uint32_t *ticket, double *out) {
    constexpr int PER = DF ? 1 : 2;   // amplitudes per load
    double acc = 0.0, best = -1.0;
    uint64_t bi = ~0ull;
    float least = -1.0f;   // below this a probability cannot win (warp-wide)
    NormSum sum;
    uint32_t it = 0;
    for (uint64_t c = blockIdx.x; c < n_chunks; c += gridDim.x) {
        const uint64_t at = c * (256 * SUMMARY_U) + threadIdx.x;
        float4 v[SUMMARY_U];
#pragma unroll
        for (int u = 0; u < SUMMARY_U; u++) v[u] = __ldcs(sv + at + 256 * u);
        const bool ok = sum.fits<DF>(v, acc);
        float p[SUMMARY_U * PER], top = -1.0f;
        if (ok) {
#pragma unroll
            for (int u = 0; u < SUMMARY_U; u++) {
                if constexpr (DF) {
                    const SquaresDf q(v[u]);
                    sum.add(q);
                    p[u] = q.rough();
                } else {
                    const Squares q(make_float2(v[u].x, v[u].y)), r(make_float2(v[u].z, v[u].w));
                    sum.add(q);
                    sum.add(r);
                    p[2 * u] = q.rough();
                    p[2 * u + 1] = r.rough();
                }
            }
#pragma unroll
            for (int j = 0; j < SUMMARY_U * PER; j++) top = fmaxf(top, p[j]);
        }
        if (__any_sync(0xffffffffu, !ok || top >= least)) {
            float w = top;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w = fmaxf(w, __shfl_xor_sync(0xffffffffu, w, o));
            least = fmaxf(least, w * (1.0f - 0x1p-21f));
#pragma unroll
            for (int j = 0; j < SUMMARY_U * PER; j++) {
                if (ok && p[j] < least) continue;
                const float4 x = v[j / PER];
                double re, im;
                if constexpr (DF) amp_parts(x, re, im);
                else amp_parts(j % 2 ? make_float2(x.z, x.w) : make_float2(x.x, x.y), re, im);
                const double q = re * re + im * im;
                if (!ok) acc += q;
                better(best, bi, q, PER * (at + 256 * (j / PER)) + j % PER);
            }
        }
        if (++it % (PROB_SUM / (PER * SUMMARY_U)) == 0) acc += sum.take();
    }
    acc += sum.take();
    const typename std::conditional<DF, float4, float2>::type *amps =
        reinterpret_cast<const typename std::conditional<DF, float4, float2>::type *>(sv);
    finish_summary(amps, acc, best, bi, sums, maxs, idxs, ticket, out);
}

cudaError_t launch_summary(bool fp64, const void *sv, int n, double *scratch, int nblocks, double *out,
                           cudaStream_t st, bool df, uint32_t *ticket) {
    const uint64_t N = 1ull << n;
    uint64_t need = (N + 255) / 256;
    int nb = (int)(need < (uint64_t)nblocks ? need : (uint64_t)nblocks);
    if (nb < 1) nb = 1;
    double *sums = scratch, *maxs = scratch + nblocks;
    uint64_t *idxs = reinterpret_cast<uint64_t *>(scratch + 2 * nblocks);
    if (fast_prob_ok(sv, N, fp64, df, 0, nullptr)) {
        const uint64_t chunks = (df ? N : N / 2) / (256 * SUMMARY_U);
        nb = (int)std::min<uint64_t>(chunks, std::min(nblocks, 152 * summary_blocks(df)));
        if (df) k_summary_fast<true><<<nb, 256, 0, st>>>((const float4 *)sv, chunks, sums, maxs, idxs, ticket, out);
        else k_summary_fast<false><<<nb, 256, 0, st>>>((const float4 *)sv, chunks, sums, maxs, idxs, ticket, out);
    } else if (df) {
        k_summary<float4><<<nb, 256, 0, st>>>((const float4 *)sv, N, sums, maxs, idxs, ticket, out);
    } else if (fp64) {
        k_summary<double2><<<nb, 256, 0, st>>>((const double2 *)sv, N, sums, maxs, idxs, ticket, out);
    } else {
        k_summary<float2><<<nb, 256, 0, st>>>((const float2 *)sv, N, sums, maxs, idxs, ticket, out);
    }
    return cudaGetLastError();
}

// ALU peak probe: 8 independent FMA chains per thread (enough to cover the
// FMA latency), over a grid that fills every SM; the result is stored so the
// chains are not removed.
template <typename T>
__global__ void __launch_bounds__(256) k_fma_probe(T *__restrict__ out, int iters, T b, T c) {
    T x[8];
#pragma unroll
    for (int j = 0; j < 8; j++) x[j] = (T)(threadIdx.x + j);
    for (int i = 0; i < iters; i++) {
#pragma unroll
        for (int j = 0; j < 8; j++) x[j] = fma(x[j], b, c);
    }
    T s = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) s += x[j];
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

cudaError_t alu_probe(bool fp64, double *flops_per_s, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int blocks = sms * 8, threads = 256;
    void *out = nullptr;
    e = cudaMallocAsync(&out, (size_t)blocks * threads * 8, st);
    if (e != cudaSuccess) return e;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    double best = 0.0;
    int iters = 256;
    for (int rep = 0; rep < 8 && e == cudaSuccess; rep++) {
        cudaEventRecord(e0, st);
        if (fp64) k_fma_probe<double><<<blocks, threads, 0, st>>>((double *)out, iters, 0.999999, 1e-7);
        else k_fma_probe<float><<<blocks, threads, 0, st>>>((float *)out, iters, 0.999999f, 1e-7f);
        cudaEventRecord(e1, st);
        e = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e != cudaSuccess) break;
        const double flops = 2.0 * 8.0 * iters * (double)blocks * threads;
        if (ms > 0.f) best = flops / (ms * 1e-3) > best ? flops / (ms * 1e-3) : best;
        if (ms < 20.f && iters < (1 << 24)) iters *= 4;   // grow to a launch of tens of milliseconds
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFreeAsync(out, st);
    if (e != cudaSuccess) return e;
    *flops_per_s = best;
    return cudaGetLastError();
}

template <typename Real>
__global__ void k_set_one(typename CT<Real>::T *sv, uint64_t idx) {
    typename CT<Real>::T v;
    v.x = Real(1);
    v.y = Real(0);
    sv[idx] = v;
}

__global__ void k_set_one_df(float4 *sv, uint64_t idx) { sv[idx] = make_float4(1.f, 0.f, 0.f, 0.f); }

cudaError_t launch_set_basis(bool fp64, void *sv, int n, uint64_t idx, cudaStream_t st, bool df) {
    const size_t bytes = (fp64 || df ? 16ull : 8ull) << n;
    cudaError_t e = cudaMemsetAsync(sv, 0, bytes, st);
    if (e != cudaSuccess) return e;
    if (df) k_set_one_df<<<1, 1, 0, st>>>((float4 *)sv, idx);
    else if (fp64) k_set_one<double><<<1, 1, 0, st>>>((double2 *)sv, idx);
    else k_set_one<float><<<1, 1, 0, st>>>((float2 *)sv, idx);
    return cudaGetLastError();
}

// Double-float representation (Dekker 1971): a double d is held as the
// unevaluated sum hi + lo of two floats, hi = d rounded to float and lo =
// (d - hi) rounded to float (d - hi is exact in FP64). In place: each element
// is read before it is written.
__global__ void __launch_bounds__(256) k_to_df(double2 *__restrict__ sv, uint64_t N) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (uint64_t)gridDim.x * blockDim.x) {
        const double2 v = sv[i];
        const float rh = __double2float_rn(v.x), ih = __double2float_rn(v.y);
        const float rl = __double2float_rn(v.x - (double)rh), il = __double2float_rn(v.y - (double)ih);
        reinterpret_cast<float4 *>(sv)[i] = make_float4(rh, rl, ih, il);
    }
}

// hi + lo back to FP64 (exact: lo lies below hi's last bit, the sum fits 53 bits).
__global__ void __launch_bounds__(256) k_from_df(const float4 *__restrict__ src, double2 *__restrict__ dst,
                                                 uint64_t N) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (uint64_t)gridDim.x * blockDim.x) {
        const float4 v = src[i];
        dst[i] = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
    }
}

cudaError_t launch_to_df(void *sv, uint64_t n_amps, cudaStream_t st) {
    k_to_df<<<grid_for(n_amps, 256), 256, 0, st>>>((double2 *)sv, n_amps);
    return cudaGetLastError();
}

cudaError_t launch_from_df(const void *src, void *dst, uint64_t n_amps, cudaStream_t st) {
    k_from_df<<<grid_for(n_amps, 256), 256, 0, st>>>((const float4 *)src, (double2 *)dst, n_amps);
    return cudaGetLastError();
}

}  // namespace hisv
