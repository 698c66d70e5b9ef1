// Circuits on fewer than 10 qubits (a state of at most 8 KiB, below the part
// kernels' smallest tile): one CTA keeps the state in shared memory and runs
// the whole gate list in one launch.
//
// Gate by gate, such a circuit is one launch of a few hundred threads per
// gate, bound by the launches: 2.5 us each, 347 us for the 138 gates of a
// 8-qubit parameterised circuit (complex64). Here an op costs a shared-memory
// round trip of its pairs and a barrier, about 0.12 us of latency, so the host
// makes fewer ops of the gates: the product of a run of one-qubit gates on a
// qubit, and one permutation of a run of CX and SWAP gates (GF(2)-linear in
// the index): 12.3 us, 22.5 us with one op per gate. One thread per pair (2^(n-1) threads,
// at least a warp); the op records are staged in shared memory a block at a
// time, so that an op's coefficients are broadcast reads. Ops do only the
// arithmetic their form needs (a real matrix, a diagonal, a permutation): in
// complex128 the SM's two FP64 lanes would otherwise set the time.
// The records are kernel parameters, so that a launch (also one in a captured
// graph) needs nothing of the plan afterwards, and a first apply uploads
// nothing.
#include "small.hpp"

#include "ops.cuh"

namespace hisv {
namespace {

constexpr int STAGE = 64;   // op records staged per block of the list

template <typename Real, uint32_t CAP> struct SmallList {
    SmallOp<Real> op[CAP];
};

template <typename Real, uint32_t CAP>
__global__ void __launch_bounds__(256) k_small(typename CT<Real>::T *__restrict__ sv, int n, uint32_t n_ops,
                                                const __grid_constant__ SmallList<Real, CAP> list) {
    typedef typename CT<Real>::T C;
    __shared__ C a[1 << SMALL_MAX_QUBITS];
    __shared__ __align__(16) unsigned char stage_raw[STAGE * sizeof(SmallOp<Real>)];
    const SmallOp<Real> *const stage = reinterpret_cast<const SmallOp<Real> *>(stage_raw);
    const uint32_t tid = threadIdx.x, N = 1u << n;
    for (uint32_t x = tid; x < N; x += blockDim.x) a[x] = sv[x];
    for (uint32_t g0 = 0; g0 < n_ops; g0 += STAGE) {
        const uint32_t m = min((uint32_t)STAGE, n_ops - g0);
        __syncthreads();
        // by its generic address: a constant-bank load takes a warp's 32
        // addresses one after another (13.3 instead of 12.3 us)
        const uint4 *src;
        asm volatile("mov.b64 %0, %1;" : "=l"(src) : "l"(list.op + g0));
        for (uint32_t i = tid; i < m * (uint32_t)(sizeof(SmallOp<Real>) / 16); i += blockDim.x)
            reinterpret_cast<uint4 *>(stage_raw)[i] = src[i];
        __syncthreads();
        for (uint32_t g = 0; g < m; g++) {
            const SmallOp<Real> &G = stage[g];
            const int kind = G.kind;
            if (kind < SMALL_PHASE) {
                const uint32_t lo = (1u << G.q0) - 1, x0 = ((tid & ~lo) << 1) | (tid & lo), x1 = x0 | (1u << G.q0);
                if (tid < N / 2) {
                    const C x = a[x0], y = a[x1];
                    C u, v;
                    if (kind == SMALL_REAL) {
                        u.x = G.m[0] * x.x + G.m[1] * y.x;
                        u.y = G.m[0] * x.y + G.m[1] * y.y;
                        v.x = G.m[2] * x.x + G.m[3] * y.x;
                        v.y = G.m[2] * x.y + G.m[3] * y.y;
                    } else if (kind == SMALL_DIAG) {
                        u.x = G.m[0] * x.x - G.m[1] * x.y;
                        u.y = G.m[0] * x.y + G.m[1] * x.x;
                        v.x = G.m[2] * y.x - G.m[3] * y.y;
                        v.y = G.m[2] * y.y + G.m[3] * y.x;
                    } else if (kind == SMALL_CROSS) {
                        u.x = G.m[0] * x.x - G.m[1] * y.y;
                        u.y = G.m[0] * x.y + G.m[1] * y.x;
                        v.x = G.m[3] * y.x - G.m[2] * x.y;
                        v.y = G.m[3] * y.y + G.m[2] * x.x;
                    } else {
                        u.x = G.m[0] * x.x - G.m[1] * x.y + G.m[2] * y.x - G.m[3] * y.y;
                        u.y = G.m[0] * x.y + G.m[1] * x.x + G.m[2] * y.y + G.m[3] * y.x;
                        v.x = G.m[4] * x.x - G.m[5] * x.y + G.m[6] * y.x - G.m[7] * y.y;
                        v.y = G.m[4] * x.y + G.m[5] * x.x + G.m[6] * y.y + G.m[7] * y.x;
                    }
                    a[x0] = u;
                    a[x1] = v;
                }
            } else if (kind == SMALL_PHASE) {
                const int ql = min(G.q0, G.q1), qh = max(G.q0, G.q1);
                const uint32_t ml = (1u << ql) - 1, mh = (1u << qh) - 1;
                if (tid < N / 4) {
                    uint32_t x = ((tid & ~ml) << 1) | (tid & ml);   // zero bits inserted at ql, then qh
                    x = ((x & ~mh) << 1) | (x & mh) | (1u << ql) | (1u << qh);
                    C v = a[x];
                    cmul_in(v, G.m[0], G.m[1]);
                    a[x] = v;
                }
            } else {   // every amplitude is read before any is written
                const uint32_t x = 2 * tid;
                uint32_t y = G.perm[n];
                for (int b = 1; b < n; b++) y ^= (x >> b) & 1 ? G.perm[b] : 0u;
                C u{}, v{};
                if (x < N) {
                    u = a[y];
                    v = a[y ^ G.perm[0]];
                }
                __syncthreads();
                if (x < N) {
                    a[x] = u;
                    a[x + 1] = v;
                }
            }
            __syncthreads();
        }
    }
    for (uint32_t x = tid; x < N; x += blockDim.x) sv[x] = a[x];
}

template <typename Real, uint32_t CAP>
cudaError_t launch_list(void *sv, int n, const SmallOp<Real> *ops, uint32_t n_ops, cudaStream_t st) {
    static_assert(sizeof(SmallList<Real, CAP>) <= 30720, "kernel parameters");
    const unsigned threads = n > 6 ? 1u << (n - 1) : 32u;
    void *args[4] = {&sv, &n, &n_ops, const_cast<SmallOp<Real> *>(ops)};   // the list is copied
    cudaError_t e = cudaLaunchKernel(reinterpret_cast<const void *>(k_small<Real, CAP>), dim3(1), dim3(threads), args, 0, st);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// The parameters' copy is part of a launch's time, so short lists go in a
// smaller record (up to 3.75 and 12 KiB).
template <typename Real>
cudaError_t launch_ops(void *sv, int n, const SmallOp<Real> *ops, uint32_t n_ops, cudaStream_t st) {
    constexpr bool W = sizeof(Real) == 8;
    constexpr uint32_t A = W ? 48 : 80, B = W ? 152 : 256, C = small_most(W);
    for (uint32_t at = 0; at < n_ops; at += C) {
        const uint32_t m = n_ops - at < C ? n_ops - at : C;
        cudaError_t e = m <= A   ? launch_list<Real, A>(sv, n, ops + at, m, st)
                        : m <= B ? launch_list<Real, B>(sv, n, ops + at, m, st)
                                 : launch_list<Real, C>(sv, n, ops + at, m, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_small(bool fp64, void *sv, int n, const void *ops, uint32_t n_ops, cudaStream_t st) {
    if (n < 1 || n > SMALL_MAX_QUBITS) return cudaErrorInvalidValue;
    return fp64 ? launch_ops(sv, n, static_cast<const SmallOp<double> *>(ops), n_ops, st)
                : launch_ops(sv, n, static_cast<const SmallOp<float> *>(ops), n_ops, st);
}

}  // namespace hisv
