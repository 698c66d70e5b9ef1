// Whole circuits on fewer than 10 qubits in one launch (see small.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace hisv {

constexpr int SMALL_MAX_QUBITS = 9;   // below the part kernels' smallest tile

// What an op does to the state: a 2x2 matrix on an amplitude pair, a phase, or
// a permutation of the amplitudes.
enum SmallKind : int32_t {
    SMALL_GENERAL = 0,   // m: m00 m01 m10 m11 (re, im each)
    SMALL_DIAG,          // m: d0 (re, im), d1 (re, im)
    SMALL_REAL,          // m: m00 m01 m10 m11, real
    SMALL_CROSS,         // m: a, b, c, d of [[a, ib], [ic, d]] (RX)
    SMALL_PHASE,         // m: d (re, im) on |11> of q0, q1
    SMALL_PERM           // new[x] = old[perm[n] ^ XOR of perm[b] over the set bits b of x] (CX, SWAP)
};

template <typename Real> struct alignas(16) SmallOp {
    union {
        Real m[8];
        uint16_t perm[SMALL_MAX_QUBITS + 1];
    };
    int32_t kind, q0, q1, pad;
};

// Op records that one launch takes (30 KiB of kernel parameters).
constexpr uint32_t small_most(bool fp64) { return fp64 ? 384u : 640u; }

// Apply n_ops ops to the n-qubit state. ops (host memory) holds
// small_most(fp64) records behind them that are never run; the launch takes
// a copy.
cudaError_t launch_small(bool fp64, void *sv, int n, const void *ops, uint32_t n_ops, cudaStream_t st);

}  // namespace hisv
