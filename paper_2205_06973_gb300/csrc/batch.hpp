// Batched persistent launch over many small circuits (device side).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "interp.hpp"
#include "program.hpp"

namespace hisv {

// One queue item: tiles [tile_begin, tile_begin + tile_count) of part `part`
// (index into the concatenated PartLaunch array) of circuit `circuit`; it may
// start once done[circuit] >= wait (tiles of the circuit's earlier parts).
struct BatchItem {
    uint32_t circuit;
    uint32_t part;
    uint32_t tile_begin;
    uint32_t tile_count;
    uint32_t wait;
};

// A circuit that one CTA runs from start to end (its program is one part).
struct BatchWhole {
    uint64_t sv_off;             // first amplitude of its state
    uint32_t part;
    uint32_t pad;
};

struct BatchLaunch {
    float2 *svbase;              // concatenated complex64 states
    const BatchItem *items;
    uint32_t n_items;
    const uint64_t *circ_off;    // first amplitude of each circuit's state
    const PartLaunch *parts;     // all circuits' parts (tile of 2^9 amplitudes)
    const uint4 *stream;         // lowered programs (interp.hpp)
    const IWindow *windows;
    uint32_t *done;              // per-circuit finished-tile counters (zeroed per run)
    uint32_t *head;              // queue ticket (zeroed per run)
    int *err;                    // bounded-wait failure flag
    bool beside;                 // the kernel before on the stream is one of the whole circuits: launched
                                 // without waiting for it, ends after it
};

// Launch configuration of a batch's kernel; beside: as a dependent that may run
// with the kernel before (griddepcontrol.wait at its end).
struct BatchConfig {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    BatchConfig(unsigned grid, unsigned threads, size_t smem, cudaStream_t st, bool beside) {
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = beside ? 1 : 0;
    }
    BatchConfig(const BatchConfig &) = delete;   // cfg points into it
};

constexpr int BATCH_TILE_QUBITS = 9;   // one warp's tile: 32 lanes x 16 amplitudes
constexpr int BATCH_REG_BITS = 4;      // tile qubits held in registers (16 amplitudes per lane)
constexpr int BATCH_MIN_QUBITS = 10;
// Circuits of at most this many qubits run on one CTA each: a 12-qubit state
// is 32 KiB of shared memory for 256 threads, so several share an SM.
constexpr int BATCH_WHOLE_QUBITS = 12;
// Their register bits: a 10-qubit state on 2^4 amplitudes per thread would
// leave two of the SM's four schedulers without a warp.
constexpr int batch_whole_R(int n) { return n < 12 ? 3 : BATCH_REG_BITS; }

// Raise the shared-memory limit and return the persistent grid size (CTAs
// resident on all SMs) for a CTA of warps_per_cta warps.
cudaError_t batch_prepare(int warps_per_cta, int *n_ctas);
cudaError_t launch_batch(const BatchLaunch &B, int warps_per_cta, int n_ctas, cudaStream_t st);
// n circuits of t qubits (BATCH_MIN_QUBITS..BATCH_WHOLE_QUBITS), one CTA each.
cudaError_t launch_batch_whole(int t, const BatchLaunch &B, const BatchWhole *circuits, uint32_t n, cudaStream_t st);
// Probabilities of all states (out, may be null) and, with norms, each
// circuit's norm: partials then holds total / 2^BATCH_MIN_QUBITS doubles.
cudaError_t launch_batch_probs(float2 *svbase, uint64_t total, const uint64_t *circ_off, const uint32_t *circ_n,
                               uint32_t n_circ, float *out, double *partials, double *norms, cudaStream_t st);
cudaError_t launch_batch_reset(float2 *svbase, const uint64_t *circ_off, uint32_t n_circ, uint64_t total,
                               cudaStream_t st);

}  // namespace hisv
