// Whole circuits on fewer than 10 qubits in one launch (see small.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace hisv {

constexpr int SMALL_MAX_QUBITS = 9;   // below the part kernels' smallest tile

// What a gate does to an amplitude pair (one qubit) or quad (two qubits).
enum SmallKind : int32_t {
    SMALL_GENERAL = 0,   // m: m00 m01 m10 m11 (re, im each)
    SMALL_DIAG,          // m: d0 (re, im), d1 (re, im)
    SMALL_REAL,          // m: m00 m01 m10 m11, real
    SMALL_RX,            // m: c, s of [[c, -is], [-is, c]]
    SMALL_CX,            // q0 control, q1 target
    SMALL_PHASE,         // m: d (re, im) on |11>
    SMALL_SWAP
};

template <typename Real> struct SmallGate {
    Real m[8];
    int32_t kind, q0, q1, pad;
};

// Apply n_gates gates (device memory, 16-byte aligned) to the n-qubit state.
cudaError_t launch_small(bool fp64, void *sv, int n, const void *gates, uint32_t n_gates, cudaStream_t st);

}  // namespace hisv
