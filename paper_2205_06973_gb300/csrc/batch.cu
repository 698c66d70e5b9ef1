// Batched persistent kernel: thousands of small, uneven circuits in one launch.
//
// Every circuit's plan is compiled for 2^9-amplitude tiles (32 lanes x 16
// amplitudes), so one warp executes one tile of one part with warp-private
// shared memory and no CTA-wide barrier. A device work list holds items
// (circuit, part, range of tiles) in wave order: the first parts of all
// circuits, then the second parts, and so on. Warps take items with an
// atomic ticket; an item of part w of circuit c starts once the circuit's
// tile counter shows that all tiles of its parts 0..w-1 are done (a bounded
// acquire spin), and bumps the counter with release semantics when it ends.
// An item only waits on items with smaller tickets, which running warps
// already hold, so the queue cannot deadlock.
#include <cuda_runtime.h>

#include <cstdint>

#include "batch.hpp"
#include "ops.cuh"
#include "prob_split.cuh"

namespace hisv {

namespace {

constexpr int BT = BATCH_TILE_QUBITS;   // tile qubits
constexpr int BR = BATCH_REG_BITS;      // register bits per lane
constexpr int BNR = 1 << BR;
constexpr uint32_t BATCH_WAIT_LIMIT = 1u << 22;

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add(uint32_t *p, uint32_t v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ uint64_t deposit_b(uint64_t v, uint64_t mask) {
    uint64_t out = 0;
    while (mask) {
        const uint64_t low = mask & (~mask + 1);
        if (v & 1) out |= low;
        v >>= 1;
        mask ^= low;
    }
    return out;
}

}  // namespace

__global__ void __launch_bounds__(256) k_batch(float2 *__restrict__ svbase, const BatchItem *__restrict__ items,
                                              uint32_t n_items, const uint64_t *__restrict__ circ_off,
                                              const PartLaunch *__restrict__ parts,
                                              const uint4 *__restrict__ stream, const IWindow *__restrict__ windows,
                                              uint32_t *__restrict__ done, uint32_t *__restrict__ head,
                                              int *__restrict__ err) {
    extern __shared__ __align__(16) float2 bsm[];
    const int lane = threadIdx.x & 31;
    float2 *const wsm = bsm + (threadIdx.x >> 5) * (1 << BT);
    float2 a[BNR];
    while (true) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(head, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_items) break;
        const BatchItem I = items[it];
        if (I.wait) {
            int ok = 1;
            if (lane == 0) {
                uint32_t k = 0;
                while (ld_acquire(done + I.circuit) < I.wait) {
                    if (++k > BATCH_WAIT_LIMIT) {
                        ok = 0;
                        break;
                    }
                    __nanosleep(64);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                if (lane == 0) atomicExch(err, 1);
                break;
            }
        }
        const PartLaunch &P = parts[I.part];
        float2 *const sv = svbase + circ_off[I.circuit];
        // copy layout: tile element = lane (slots 0..4) | i << 5 (slots 5..9)
        uint64_t c_thr = 0;
        uint32_t s_cthr = 0;
#pragma unroll
        for (int j = 0; j < BT - BR; j++)
            if ((lane >> j) & 1) {
                c_thr |= 1ull << P.tile_q[j];
                s_cthr ^= swz<float>(j);
            }
        for (uint32_t tile = I.tile_begin; tile < I.tile_begin + I.tile_count; tile++) {
            const uint64_t base = deposit_b(tile, P.outer_mask) | c_thr;
#pragma unroll
            for (int i = 0; i < BNR; i++) {
                uint64_t go = 0;
                uint32_t so = s_cthr;
#pragma unroll
                for (int b = 0; b < BR; b++)
                    if (i & (1 << b)) {
                        go |= 1ull << P.tile_q[BT - BR + b];
                        so ^= swz<float>(BT - BR + b);
                    }
                wsm[so] = __ldcg(sv + (base | go));
            }
            __syncwarp();
            float tpr = 1.0f, tpi = 0.0f;
            uint32_t tsg = 0u;
            Slots<BR, BT - BR> S;
            for (uint32_t w = 0; w < P.n_phases; w++) {   // read in place: a warp's items share few programs
                const IWindow W = windows[P.phase_begin + w];
                run_window<float, BR, BT - BR>(a, wsm, S, reinterpret_cast<const char *>(stream + W.at), W.phases, w == 0,
                                               lane, tpr, tpi, tsg, [] { __syncwarp(); });
            }
            if (P.flags & PL_STORE_FACTOR) {
                const float gr = (float)P.gr, gi = (float)P.gi;
                const float fr = gr * tpr - gi * tpi, fi = gr * tpi + gi * tpr;
#pragma unroll
                for (int i = 0; i < BNR; i++) cmul_in(a[i], fr, fi);
            }
            {
                uint64_t toff = deposit_b(tile, P.outer_mask);
#pragma unroll
                for (int j = 0; j < BT - BR; j++)
                    if ((lane >> j) & 1) toff ^= P.store_thr[j];
#pragma unroll
                for (int i = 0; i < BNR; i++) {
                    uint64_t off = toff;
#pragma unroll
                    for (int b = 0; b < BR; b++)
                        if (i & (1 << b)) off ^= P.store_reg[b];
                    __stcg(sv + off, a[i]);
                }
            }
            __syncwarp();   // the warp's shared tile is reused by the next tile
        }
        if (lane == 0) {
            __threadfence();
            red_release_add(done + I.circuit, I.tile_count);
        }
        __syncwarp();
    }
    pdl_wait();   // done when the kernel before is (BatchLaunch::beside)
}

// Whole circuits of T qubits, one CTA each: the state stays in shared memory
// and registers from the first gate to the last (the planner's program of the
// circuit as one part). On 2^9-amplitude tiles such a circuit is a chain of
// parts of a few tiles each, every part a trip through L2 and the work queue
// with little for the other warps to do: 45 parameterised circuits of 10 to
// 12 qubits took 3.2 ms.
// The kernels of a batch's sizes and the one after them share nothing: each
// lets the next launch as soon as its own CTAs have started, and ends when the
// one before has ended, so that they run beside each other and still form a
// chain (BatchLaunch::beside).
template <int T, int R>
__global__ void __launch_bounds__(1 << (T - R))
k_batch_whole(float2 *__restrict__ svbase, const BatchWhole *__restrict__ circuits,
              const PartLaunch *__restrict__ parts, const uint4 *__restrict__ stream,
              const IWindow *__restrict__ windows) {
    constexpr int TB = T - R, NR = 1 << R;
    extern __shared__ __align__(16) float2 bsm[];
    char *const prog = reinterpret_cast<char *>(bsm + (1 << T));   // INTERP_WINDOW bytes
    const uint32_t tid = threadIdx.x;
    const BatchWhole C = circuits[blockIdx.x];
    const PartLaunch &P = parts[C.part];
    pdl_launch();   // the next kernel of the graph shares nothing with this one
    float2 *const sv = svbase + C.sv_off;
    uint32_t s_cthr = 0;
#pragma unroll
    for (int j = 0; j < TB; j++)
        if ((tid >> j) & 1) s_cthr ^= swz<float>(j);
#pragma unroll
    for (int i = 0; i < NR; i++) {
        uint32_t so = s_cthr;
#pragma unroll
        for (int b = 0; b < R; b++)
            if (i & (1 << b)) so ^= swz<float>(TB + b);
        bsm[so] = __ldcg(sv + (tid | ((uint32_t)i << TB)));
    }
    float2 a[NR];
    float tpr = 1.0f, tpi = 0.0f;
    uint32_t tsg = 0u;
    Slots<R, TB> S;
    for (uint32_t w = 0; w < P.n_phases; w++) {
        const IWindow W = windows[P.phase_begin + w];
        if (w > 0) __syncthreads();   // every thread is done with the previous window
        copy_window(prog, stream, W, tid, 1u << TB);
        __syncthreads();
        run_window<float, R, TB>(a, bsm, S, prog, W.phases, w == 0, tid, tpr, tpi, tsg, [] { __syncthreads(); });
    }
    if (P.flags & PL_STORE_FACTOR) {
        const float gr = (float)P.gr, gi = (float)P.gi;
        const float fr = gr * tpr - gi * tpi, fi = gr * tpi + gi * tpr;
#pragma unroll
        for (int i = 0; i < NR; i++) cmul_in(a[i], fr, fi);
    }
    uint32_t toff = 0;
#pragma unroll
    for (int j = 0; j < TB; j++)
        if ((tid >> j) & 1) toff ^= (uint32_t)P.store_thr[j];
#pragma unroll
    for (int i = 0; i < NR; i++) {
        uint32_t off = toff;
#pragma unroll
        for (int b = 0; b < R; b++)
            if (i & (1 << b)) off ^= (uint32_t)P.store_reg[b];
        __stcg(sv + off, a[i]);
    }
    pdl_wait();   // done when the kernel before is
}

// p[i] = |a_i|^2 over the concatenated states, 2^10 amplitudes per block and
// iteration (the smallest circuit, and every circuit's offset is a multiple
// of it), on the FP32 pipes as in k_probs_fast; partials (may be null)
// receives each chunk's FP64 sum. One block per circuit with FP64 arithmetic
// left a batch's largest circuits to single SMs: 2.83 ms for 160 circuits of
// 10 to 20 qubits (28.5 M amplitudes), the time of one 20-qubit circuit;
// 0.06 ms here, 0.12 with norms.
constexpr int BPROB_CHUNK = 1 << BATCH_MIN_QUBITS;
constexpr int BPROB_THREADS = 128;
constexpr int BPROB_U = 4;   // 16-byte loads in flight per thread: a chunk in one round
static_assert(BPROB_CHUNK == 2 * BPROB_THREADS * BPROB_U && 2 * BPROB_U <= PROB_SUM, "a chunk per block");

__global__ void __launch_bounds__(BPROB_THREADS, 10)
k_batch_probs(const float4 *__restrict__ sv, uint64_t n_chunks, float *__restrict__ out, bool pairs,
              double *__restrict__ partials) {
    __shared__ double red[BPROB_THREADS / 32];
    for (uint64_t c = blockIdx.x; c < n_chunks; c += gridDim.x) {
        const uint64_t at = c * (BPROB_CHUNK / 2) + threadIdx.x;
        float4 v[BPROB_U];
#pragma unroll
        for (int u = 0; u < BPROB_U; u++) v[u] = __ldcs(sv + at + BPROB_THREADS * u);
        NormSum sum;
        double acc = 0.0;
        const bool ok = sum.fits<false>(v, acc);
#pragma unroll
        for (int u = 0; u < BPROB_U; u++) {
            float p, q;
            if (ok) {
                const Squares a(make_float2(v[u].x, v[u].y)), b(make_float2(v[u].z, v[u].w));
                sum.add(a);
                sum.add(b);
                p = a.prob();
                q = b.prob();
            } else {
                const double a = (double)v[u].x * v[u].x + (double)v[u].y * v[u].y;
                const double b = (double)v[u].z * v[u].z + (double)v[u].w * v[u].w;
                acc += a;
                acc += b;
                p = (float)a;
                q = (float)b;
            }
            if (out) {
                const uint64_t i = 2 * (at + BPROB_THREADS * u);
                if (pairs) *reinterpret_cast<float2 *>(out + i) = make_float2(p, q);
                else {
                    out[i] = p;
                    out[i + 1] = q;
                }
            }
        }
        if (!partials) continue;
        acc += sum.take();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < BPROB_THREADS / 32; w++) s += red[w];
            partials[c] = s;
        }
        __syncthreads();
    }
}

// A circuit's norm: its chunks' sums in a fixed order, one block per circuit.
__global__ void __launch_bounds__(256) k_batch_norms(const double *__restrict__ partials,
                                                     const uint64_t *__restrict__ circ_off,
                                                     const uint32_t *__restrict__ circ_n, double *__restrict__ norms) {
    __shared__ double red[8];
    const uint32_t c = blockIdx.x;
    const double *const v = partials + circ_off[c] / BPROB_CHUNK;
    const uint32_t m = 1u << (circ_n[c] - BATCH_MIN_QUBITS);
    double acc = 0.0;
    for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) acc += v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < 8; w++) s += red[w];
        norms[c] = s;
    }
}

__global__ void k_batch_reset(float2 *__restrict__ svbase, const uint64_t *__restrict__ circ_off,
                              uint32_t n_circ, uint64_t total) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (uint64_t)gridDim.x * blockDim.x)
        svbase[i] = make_float2(0.f, 0.f);
}

__global__ void k_batch_basis(float2 *__restrict__ svbase, const uint64_t *__restrict__ circ_off, uint32_t n_circ) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n_circ) svbase[circ_off[c]] = make_float2(1.f, 0.f);
}

cudaError_t batch_prepare(int warps_per_cta, int *n_ctas) {
    const size_t smem = (size_t)warps_per_cta * (1u << BT) * sizeof(float2);
    cudaError_t e = cudaFuncSetAttribute(k_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * 8192);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch, warps_per_cta * 32, smem)) != cudaSuccess)
        return e;
    *n_ctas = sms * (per_sm < 1 ? 1 : per_sm);
    return cudaSuccess;
}

cudaError_t launch_batch(const BatchLaunch &B, int warps_per_cta, int n_ctas, cudaStream_t st) {
    BatchConfig c(n_ctas, warps_per_cta * 32, (size_t)warps_per_cta * (1u << BT) * sizeof(float2), st, B.beside);
    cudaError_t e = cudaLaunchKernelEx(&c.cfg, k_batch, B.svbase, B.items, B.n_items, B.circ_off, B.parts, B.stream,
                                       B.windows, B.done, B.head, B.err);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <int T>
static cudaError_t whole_t(const BatchLaunch &B, const BatchWhole *circuits, uint32_t n, cudaStream_t st) {
    constexpr int R = batch_whole_R(T);
    BatchConfig c(n, 1u << (T - R), (sizeof(float2) << T) + INTERP_WINDOW, st, B.beside);
    cudaError_t e = cudaLaunchKernelEx(&c.cfg, k_batch_whole<T, R>, B.svbase, circuits, B.parts, B.stream, B.windows);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_batch_whole(int t, const BatchLaunch &B, const BatchWhole *circuits, uint32_t n, cudaStream_t st) {
    switch (t) {
    case 10: return whole_t<10>(B, circuits, n, st);
    case 11: return whole_t<11>(B, circuits, n, st);
    case 12: return whole_t<12>(B, circuits, n, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_batch_probs(float2 *svbase, uint64_t total, const uint64_t *circ_off, const uint32_t *circ_n,
                               uint32_t n_circ, float *out, double *partials, double *norms, cudaStream_t st) {
    const uint64_t chunks = total / BPROB_CHUNK;
    const uint64_t blocks = chunks < 152 * 10 ? chunks : 152 * 10;
    if (out || norms) {
        k_batch_probs<<<(unsigned)blocks, BPROB_THREADS, 0, st>>>(reinterpret_cast<const float4 *>(svbase), chunks, out,
                                                        (reinterpret_cast<uintptr_t>(out) & 7) == 0,
                                                        norms ? partials : nullptr);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (norms) k_batch_norms<<<n_circ, 256, 0, st>>>(partials, circ_off, circ_n, norms);
    return cudaGetLastError();
}

cudaError_t launch_batch_reset(float2 *svbase, const uint64_t *circ_off, uint32_t n_circ, uint64_t total,
                               cudaStream_t st) {
    uint64_t blocks = (total + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    k_batch_reset<<<(unsigned)blocks, 256, 0, st>>>(svbase, circ_off, n_circ, total);
    k_batch_basis<<<(n_circ + 255) / 256, 256, 0, st>>>(svbase, circ_off, n_circ);
    return cudaGetLastError();
}

}  // namespace hisv
