// k_part: one HBM pass of one part (Algorithm 1, Gather-Execute-Scatter), with
// the part's gates interpreted from a stream (interp.hpp) whose window the
// CTA copies into shared memory before the first tile. Persistent CTAs walk the
// tiles (outer assignments) with a two-stage pipeline: while tile i is
// computed from registers, the cp.async copy of tile i + 1 streams into the
// other shared buffer. The tile's register phases (2^R amplitudes per thread)
// are separated by transposes through XOR-swizzled shared memory; the last
// phase's layout scatters the tile back from registers.
//
// Consecutive passes use programmatic dependent launch: a CTA that starts its
// last tile lets the next pass's CTAs launch, and they wait for this grid
// before they touch the state, so the launch and the prologue of a pass do
// not stand between two passes of a small state.
#pragma once
#include <atomic>
#include <mutex>

#include "kernels.hpp"
#include "ops.cuh"

namespace hisv {

// Asynchronous global -> shared copies (sm_80+ cp.async); 8-byte elements use
// the L1-allocating form, 16-byte elements the L2-only form.
template <int BYTES>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Deposit the bits of v, lowest first, into the set bits of mask.
__device__ __forceinline__ uint64_t deposit64(uint64_t v, uint64_t mask) {
    uint64_t out = 0;
    while (mask) {
        const uint64_t low = mask & (~mask + 1);
        if (v & 1) out |= low;
        v >>= 1;
        mask ^= low;
    }
    return out;
}

// Resident CTAs the launch bound asks for: two tile buffers of 2^T amplitudes
// in shared memory, and the registers per thread that avoid spills (at 80,
// three CTAs of 256 threads, a 20-qubit circuit took 242 us against 175 us).
template <typename Real, int T, int R>
struct PartCfg {
    static constexpr int NT = 1 << (T - R);
    static constexpr int SMEM = 2 * (1 << T) * 2 * (int)sizeof(Real) + (int)INTERP_WINDOW;
    static constexpr int REGS = sizeof(Real) == 8 ? (R == 4 ? 168 : 120) : (R == 5 ? 168 : R == 4 ? 104 : 64);
    static constexpr int BY_REG = 65536 / (REGS * NT);
    static constexpr int BY_SMEM = (227 * 1024) / (SMEM + 1024);
    static constexpr int MINB0 = BY_REG < BY_SMEM ? BY_REG : BY_SMEM;
    static constexpr int MINB = MINB0 < 1 ? 1 : MINB0 > 24 ? 24 : MINB0;
};

template <typename Real, int T, int R>
__global__ void __launch_bounds__(PartCfg<Real, T, R>::NT, PartCfg<Real, T, R>::MINB)
k_part(typename CT<Real>::T *__restrict__ sv, const __grid_constant__ PartLaunch L,
       const uint4 *__restrict__ stream, const IWindow *__restrict__ windows, uint64_t n_tiles) {
    typedef typename CT<Real>::T C;
    constexpr int NR = 1 << R;
    constexpr int TB = T - R;
    constexpr int TILE = 1 << T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *const buf0 = reinterpret_cast<C *>(smem_raw);
    C *const buf1 = buf0 + TILE;
    char *const prog = reinterpret_cast<char *>(buf1 + TILE);   // INTERP_WINDOW bytes
    const uint32_t tid = threadIdx.x;
    IWindow W = windows[L.phase_begin];
    copy_window(prog, stream, W, tid, 1u << TB);   // ordered by the first tile's barriers

    // copy layout: tile index = tid | (c << TB); thread bits on the lowest slots
    uint64_t c_thr = 0, s_thr = 0;
    uint32_t s_cthr = 0;
#pragma unroll
    for (int j = 0; j < TB; j++)
        if ((tid >> j) & 1) {
            c_thr |= 1ull << L.tile_q[j];
            s_cthr ^= swz<Real>(j);
            s_thr ^= L.store_thr[j];
        }
    auto issue = [&](uint64_t base, C *dst) {
        const C *src = sv + (base | c_thr);
#pragma unroll
        for (int i = 0; i < NR; i++) {
            uint64_t go = 0;
            uint32_t so = s_cthr;
#pragma unroll
            for (int b = 0; b < R; b++)
                if (i & (1 << b)) {
                    go |= 1ull << L.tile_q[TB + b];
                    so ^= swz<Real>(TB + b);
                }
            cp_async<(int)sizeof(C)>(dst + so, src + go);
        }
    };

    C a[NR];
    uint64_t tile = blockIdx.x;
    const uint64_t dgrid = deposit64(gridDim.x, L.outer_mask);
    const uint64_t flip = L.flags & PL_REVERSE ? L.outer_mask : 0ull;
    uint64_t base = deposit64(tile, L.outer_mask);
    pdl_wait();   // the previous pass has written the state
    if (tile < n_tiles) issue(base ^ flip, buf0);
    cp_async_commit();
    for (uint32_t it = 0; tile < n_tiles; tile += gridDim.x, it++) {
        C *const cur = (it & 1) ? buf1 : buf0;
        C *const nxt = (it & 1) ? buf0 : buf1;
        __syncthreads();   // every thread is done with nxt (it was cur two stages ago)
        // the next tile's outer bits: an add whose carries run over the tile's qubits
        const uint64_t nbase = ((base | ~L.outer_mask) + dgrid) & L.outer_mask;
        if (tile + gridDim.x < n_tiles) issue(nbase ^ flip, nxt);
        else pdl_launch();
        cp_async_commit();
        cp_async_wait<1>();  // this tile's copies have landed
        __syncthreads();

        Real tpr = Real(1), tpi = Real(0);   // per-thread phase of diagonal gates on thread bits
        uint32_t tsg = 0u;                   // and its sign
        Slots<R, TB> S;
        for (uint32_t w = 0; w < L.n_phases; w++) {
            if (L.n_phases > 1 && (w > 0 || it > 0)) {   // a program of several windows
                __syncthreads();
                W = windows[L.phase_begin + w];
                copy_window(prog, stream, W, tid, 1u << TB);
                __syncthreads();
            }
            run_window<Real, R, TB>(a, cur, S, prog, W.phases, w == 0, tid, tpr, tpi, tsg, [] { __syncthreads(); });
        }
        // Scatter: the last phase's layout, with SWAP relabels applied; the
        // part factor and the last phase's per-thread phase are applied here
        if (L.flags & PL_STORE_FACTOR) {
            const Real gr = (Real)L.gr, gi = (Real)L.gi;
            const Real fr = gr * tpr - gi * tpi, fi = gr * tpi + gi * tpr;
#pragma unroll
            for (int i = 0; i < NR; i++) cmul_in(a[i], fr, fi);
        }
        const uint64_t dst = (base ^ flip) | s_thr;
#pragma unroll
        for (int i = 0; i < NR; i++) {
            uint64_t off = dst;
#pragma unroll
            for (int b = 0; b < R; b++)
                if (i & (1 << b)) off ^= L.store_reg[b];
            __stcs(sv + off, a[i]);
        }
        base = nbase;
    }
    cp_async_wait<0>();
}

template <typename Real, int T, int R>
static cudaError_t launch_part_t(void *sv, const PartLaunch &L, const void *stream, const IWindow *windows,
                                 uint64_t n_tiles, cudaStream_t st) {
    typedef typename CT<Real>::T C;
    typedef PartCfg<Real, T, R> Cfg;
    auto kern = k_part<Real, T, R>;
    const size_t smem = Cfg::SMEM;
    // per instantiation: devices on which the shared-memory limit was raised,
    // and the resident CTAs per SM found there
    // (set once under a lock; a thread that sees the device's bit sees its counts)
    static std::atomic<uint64_t> attr_set{0};
    static std::mutex mu;
    static int resident[64];
    static int sms[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64) return cudaErrorInvalidDevice;
    if (!((attr_set.load(std::memory_order_acquire) >> dev) & 1)) {
        std::lock_guard<std::mutex> lk(mu);
        if (!((attr_set.load(std::memory_order_relaxed) >> dev) & 1)) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            int nb = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, Cfg::NT, smem);
            if (e != cudaSuccess) return e;
            e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            resident[dev] = nb < 1 ? 1 : nb;
            attr_set.fetch_or(1ull << dev, std::memory_order_release);
        }
    }
    uint64_t grid = (uint64_t)sms[dev] * resident[dev];
    if (grid > n_tiles) grid = n_tiles;
    if (grid < 1) grid = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(Cfg::NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // not where the grid leaves many slots of a second or third CTA per SM
    // free: the early CTAs of the next pass would share SMs while others idle
    // (20 qubits, 2^12 tiles, three slots: 157 us against 184)
    const uint64_t slots = (uint64_t)sms[dev] * resident[dev];
    cfg.numAttrs = grid > (uint64_t)sms[dev] && slots - grid > grid / 2 ? 0 : 1;
    e = cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<C *>(sv), L, reinterpret_cast<const uint4 *>(stream), windows,
                           n_tiles);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace hisv
