// C ABI of the library (declared in include/hisvsim.h).
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/hisvsim.h"
#include "abi_internal.hpp"
#include "dense.hpp"
#include "kernels.hpp"
#include "partition.hpp"
#include "planner.hpp"
#include "small.hpp"

using namespace hisv;

namespace {
thread_local std::string g_err = "no error";

sv_status fail(sv_status st, const std::string &msg) {
    g_err = msg;
    return st;
}

#define CUDA_TRY(call)                                                                        \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return fail(SV_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));    \
    } while (0)

constexpr int kProbBlocks = 152 * 8;
// per-state reduction scratch: kProbBlocks partial sums and the norm
// (sv_measure_probs), then 3 * kProbBlocks block results and 4 outputs
// (sv_measure_summary)
constexpr int kSummaryAt = kProbBlocks + 1;
constexpr int kPartialsLen = kSummaryAt + 3 * kProbBlocks + 4;
// per-state device words: the error word of bounded waits, then the block
// tickets of the two measurements
constexpr int kErrWords = 3;

// Result slots in pinned host memory that the measurement kernels write
// themselves: a copy of a few bytes to pageable memory costs more than the
// reduction of a small state (summary of 2^10 amplitudes 29 -> 18 us a call,
// 2^20 54 -> 28 us with the reduction's own gain). One page for the process,
// allocated at the first measurement; a state holds a slot from its first
// measurement to its end. A state that finds none copies its results.
constexpr int kSlots = 64, kSlotDoubles = 8;
struct ResultSlots {
    std::mutex mu;
    double *page = nullptr;
    bool tried = false;
    uint64_t used = 0;
    double *take() {
        std::lock_guard<std::mutex> lk(mu);
        if (!tried) {
            tried = true;
            // another thread may be capturing: the allocation is no part of it
            cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
            const bool swapped = cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess;
            if (cudaHostAlloc(reinterpret_cast<void **>(&page), sizeof(double) * kSlots * kSlotDoubles,
                              cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess)
                page = nullptr;
            if (swapped) cudaThreadExchangeStreamCaptureMode(&mode);
            cudaGetLastError();
        }
        if (!page || !~used) return nullptr;
        const int i = __builtin_ctzll(~used);
        used |= 1ull << i;
        return page + i * kSlotDoubles;
    }
    void give(double *slot) {
        if (!slot) return;
        std::lock_guard<std::mutex> lk(mu);
        used &= ~(1ull << ((slot - page) / kSlotDoubles));
    }
};
ResultSlots &result_slots() {
    static ResultSlots *s = new ResultSlots();   // never destroyed: states may outlive static objects
    return *s;
}
}  // namespace

namespace hisv {
void set_last_error(const std::string &msg) { g_err = msg; }
}

static size_t amp_bytes(sv_precision p) { return p == SV_C64 ? 8 : 16; }
// complex128 and its double-float form share the FP64 program (tile, register bits)
static bool is_fp64(const sv_state *s) { return s->prec != SV_C64; }
static bool is_df(const sv_state *s) { return s->prec == SV_C128DF; }
constexpr uint64_t kStageAmps = 1ull << 21;   // 32 MiB of double2 per staged download chunk

// Default tile: 2^12 complex64 / 2^11 complex128 amplitudes per CTA (two
// 64 KiB shared buffers, three CTAs per SM), grown so that the tile holds
// the plan's largest part and, where the limit allows, enough of the lowest
// free qubits that every contiguous run of a gathered tile fills a 32-byte
// sector: two qubits (4 amplitudes) for complex64, one for the 16-byte
// complex128 forms. A part without the state's low qubits otherwise reads
// runs of one amplitude, and the shared-memory fill of the tile, not the
// HBM traffic, sets the pace (measured at k = 12: 1.4-1.8x slower per pass
// with the 2^12 tile than with 2^13).
static int default_tile(bool fp64, int max_part) {
    int t = fp64 ? 11 : 12;
    const int fill = fp64 ? 1 : 2;
    if (max_part + fill > t) t = max_part + fill;
    return t > part_tmax(fp64) ? part_tmax(fp64) : t;
}

extern "C" {

const char *sv_last_error(void) { return g_err.c_str(); }
const char *sv_version(void) { return "hisvsim-gb300 0.1 (sm_103a)"; }

}  // extern "C"

// Copy v to new device memory (stream-ordered).
template <typename V> static cudaError_t upload_vec(void **d, const V &v, cudaStream_t st) {
    if (v.empty()) return cudaSuccess;
    const size_t bytes = v.size() * sizeof(v[0]);
    cudaError_t e = dev_alloc(d, bytes, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(*d, v.data(), bytes, cudaMemcpyHostToDevice, st);
    return e;
}
static cudaError_t upload_lowered(const Program &prog, DevProgram &d, cudaStream_t st) {
    Lowered lo;
    lower_program(prog, lo);
    d.parts = lo.parts;
    cudaError_t e = upload_vec(&d.d_stream, lo.stream, st);
    if (e == cudaSuccess) e = upload_vec(reinterpret_cast<void **>(&d.d_windows), lo.windows, st);
    cudaError_t se = cudaStreamSynchronize(st);   // lo goes out of scope
    return e == cudaSuccess ? se : e;
}

// The ops of a small circuit in the kernel's precision: runs of one-qubit
// gates on a qubit as one matrix (any gate on other qubits between them
// commutes with them), runs of CX and SWAP gates as one permutation.
template <typename Real> static std::vector<SmallOp<Real>> small_ops(const sv_plan *p) {
    std::vector<SmallOp<Real>> out;
    const int n = p->n;
    std::vector<std::array<double, 8>> pend(n);   // product of the qubit's pending gates
    std::vector<char> has(n, 0);
    auto flush = [&](int q) {
        if (!has[q]) return;
        has[q] = 0;
        const double *u = pend[q].data();
        SmallOp<Real> r;
        std::memset(&r, 0, sizeof(r));
        r.q0 = q;
        double m[8] = {0};
        if (u[2] == 0 && u[3] == 0 && u[4] == 0 && u[5] == 0) {
            r.kind = SMALL_DIAG;
            m[0] = u[0]; m[1] = u[1]; m[2] = u[6]; m[3] = u[7];
        } else if (u[1] == 0 && u[3] == 0 && u[5] == 0 && u[7] == 0) {
            r.kind = SMALL_REAL;
            for (int j = 0; j < 4; j++) m[j] = u[2 * j];
        } else if (u[1] == 0 && u[2] == 0 && u[4] == 0 && u[7] == 0) {
            r.kind = SMALL_CROSS;
            m[0] = u[0]; m[1] = u[3]; m[2] = u[5]; m[3] = u[6];
        } else {
            r.kind = SMALL_GENERAL;
            std::memcpy(m, u, sizeof(m));
        }
        for (int j = 0; j < 8; j++) r.m[j] = (Real)m[j];
        out.push_back(r);
    };
    // the pending permutation new[x] = old[L x]: columns of L
    std::vector<uint16_t> cols(n);
    bool perm = false;
    auto flush_perm = [&]() {
        if (!perm) return;
        perm = false;
        SmallOp<Real> r;
        std::memset(&r, 0, sizeof(r));
        r.kind = SMALL_PERM;
        for (int b = 0; b < n; b++) r.perm[b] = cols[b];
        out.push_back(r);
    };
    for (const GateRef &g : p->gates) {
        if (g.arity == 1) {
            // gates on qubits that the permutation moves come after it
            const int q = g.q[0];
            if (perm) flush_perm();
            double u[8];
            gate_matrix_1q(g.kind, g.theta, u);
            if (!has[q]) {
                std::copy(u, u + 8, pend[q].begin());
                has[q] = 1;
                continue;
            }
            std::array<double, 8> t;
            for (int r = 0; r < 2; r++)
                for (int c = 0; c < 2; c++) {
                    double re = 0, im = 0;
                    for (int k = 0; k < 2; k++) {
                        const double ar = u[2 * (2 * r + k)], ai = u[2 * (2 * r + k) + 1];
                        const double br = pend[q][2 * (2 * k + c)], bi = pend[q][2 * (2 * k + c) + 1];
                        re += ar * br - ai * bi;
                        im += ar * bi + ai * br;
                    }
                    t[2 * (2 * r + c)] = re;
                    t[2 * (2 * r + c) + 1] = im;
                }
            pend[q] = t;
            continue;
        }
        flush(g.q[0]);
        flush(g.q[1]);
        if (g.kind == SV_GATE_CX || g.kind == SV_GATE_SWAP) {
            if (!perm)
                for (int b = 0; b < n; b++) cols[b] = (uint16_t)(1u << b);
            perm = true;
            // new state y[x] = old[L x]; the gate then maps z[x] = y[G x], so L <- L G
            if (g.kind == SV_GATE_CX) cols[g.q[0]] ^= cols[g.q[1]];   // G e_c = e_c + e_t
            else std::swap(cols[g.q[0]], cols[g.q[1]]);
            continue;
        }
        flush_perm();
        SmallOp<Real> r;
        std::memset(&r, 0, sizeof(r));
        r.kind = SMALL_PHASE;
        r.q0 = g.q[0];
        r.q1 = g.q[1];
        r.m[0] = (Real)(g.kind == SV_GATE_CZ ? -1.0 : std::cos(g.theta));
        r.m[1] = (Real)(g.kind == SV_GATE_CZ ? 0.0 : std::sin(g.theta));
        out.push_back(r);
    }
    flush_perm();
    for (int q = 0; q < n; q++) flush(q);
    return out;
}

static sv_status create_state(int n, sv_precision prec, void *dev_buf, size_t dev_buf_bytes, void *stream, bool init,
                              sv_state **out) {
    if (!out) return fail(SV_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (n < 1 || n > 36) return fail(SV_ERR_ARG, "n_qubits must be in [1, 36]");
    if (prec != SV_C64 && prec != SV_C128 && prec != SV_C128DF) return fail(SV_ERR_ARG, "bad precision");
    const size_t bytes = amp_bytes(prec) << n;
    if (dev_buf && dev_buf_bytes < bytes) return fail(SV_ERR_ARG, "dev_buf smaller than 2^n amplitudes");
    if (dev_buf && (reinterpret_cast<uintptr_t>(dev_buf) & 15)) return fail(SV_ERR_ARG, "dev_buf must be 16-byte aligned");
    std::unique_ptr<sv_state> s(new sv_state());
    s->n = n;
    s->prec = prec;
    s->bytes = bytes;
    s->stream = reinterpret_cast<cudaStream_t>(stream);
    CUDA_TRY(cudaGetDevice(&s->dev));
    if (dev_buf) {
        s->buf = dev_buf;
    } else {
        cudaError_t e = dev_alloc(&s->buf, bytes, s->stream);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(SV_ERR_OOM, std::string("state allocation: ") + cudaGetErrorString(e));
        }
        s->owns = true;
    }
    cudaError_t e = dev_alloc(reinterpret_cast<void **>(&s->d_partials), sizeof(double) * kPartialsLen, s->stream);
    if (e == cudaSuccess) e = dev_alloc(reinterpret_cast<void **>(&s->d_err), sizeof(int) * kErrWords, s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->d_err, 0, sizeof(int) * kErrWords, s->stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (s->owns) dev_free(s->buf, s->stream);
        dev_free(s->d_partials, s->stream);
        dev_free(s->d_err, s->stream);
        return fail(SV_ERR_OOM, std::string("scratch allocation: ") + cudaGetErrorString(e));
    }
    if (init) e = launch_set_basis(is_fp64(s.get()), s->buf, n, 0, s->stream, is_df(s.get()));
    if (e != cudaSuccess) {
        if (s->owns) dev_free(s->buf, s->stream);
        dev_free(s->d_partials, s->stream);
        dev_free(s->d_err, s->stream);
        return fail(SV_ERR_CUDA, std::string("init: ") + cudaGetErrorString(e));
    }
    *out = s.release();
    return SV_OK;
}

extern "C" {

sv_status sv_create(int n, sv_precision prec, void *dev_buf, size_t dev_buf_bytes, void *stream, sv_state **out) {
    return create_state(n, prec, dev_buf, dev_buf_bytes, stream, true, out);
}

sv_status sv_attach(int n, sv_precision prec, void *dev_buf, size_t dev_buf_bytes, void *stream, sv_state **out) {
    if (!dev_buf) return fail(SV_ERR_ARG, "sv_attach needs dev_buf");
    return create_state(n, prec, dev_buf, dev_buf_bytes, stream, false, out);
}

sv_status sv_destroy(sv_state *s) {
    if (!s) return fail(SV_ERR_ARG, "state is NULL");
    cudaError_t e = cudaStreamSynchronize(s->stream);
    if (s->owns) dev_free(s->buf, s->stream);
    dev_free(s->d_partials, s->stream);
    dev_free(s->d_err, s->stream);
    dev_free(s->d_dnorm, s->stream);
    dev_free(s->d_stage, s->stream);
    result_slots().give(s->h_slot);   // the stream is idle
    delete s;
    if (e != cudaSuccess) return fail(SV_ERR_CUDA, std::string("pending work failed: ") + cudaGetErrorString(e));
    return SV_OK;
}

sv_status sv_set_basis(sv_state *s, uint64_t index) {
    if (!s) return fail(SV_ERR_ARG, "state is NULL");
    if (index >> s->n) return fail(SV_ERR_ARG, "basis index >= 2^n");
    CUDA_TRY(launch_set_basis(is_fp64(s), s->buf, s->n, index, s->stream, is_df(s)));
    return SV_OK;
}

sv_status sv_upload(sv_state *s, const void *src, size_t bytes) {
    if (!s || !src) return fail(SV_ERR_ARG, "NULL argument");
    if (bytes != s->bytes) return fail(SV_ERR_ARG, "bytes must equal the state size");
    CUDA_TRY(cudaMemcpyAsync(s->buf, src, bytes, cudaMemcpyHostToDevice, s->stream));
    if (is_df(s)) CUDA_TRY(launch_to_df(s->buf, 1ull << s->n, s->stream));   // double2 -> hi + lo, in place
    return SV_OK;
}

// Device -> host copy of the state (stream-ordered). A double-float state
// goes through a staging buffer in chunks, each converted to double2 first.
static sv_status copy_out(sv_state *s, void *dst) {
    if (!is_df(s)) {
        CUDA_TRY(cudaMemcpyAsync(dst, s->buf, s->bytes, cudaMemcpyDeviceToHost, s->stream));
        return SV_OK;
    }
    const uint64_t N = 1ull << s->n, chunk = std::min<uint64_t>(N, kStageAmps);
    if (!s->d_stage) {
        cudaError_t e = dev_alloc(&s->d_stage, 16 * chunk, s->stream);
        if (e != cudaSuccess) {
            cudaGetLastError();
            s->d_stage = nullptr;
            return fail(SV_ERR_OOM, std::string("download staging: ") + cudaGetErrorString(e));
        }
    }
    for (uint64_t i = 0; i < N; i += chunk) {
        const uint64_t m = std::min(chunk, N - i);
        CUDA_TRY(launch_from_df(static_cast<char *>(s->buf) + 16 * i, s->d_stage, m, s->stream));
        CUDA_TRY(cudaMemcpyAsync(static_cast<char *>(dst) + 16 * i, s->d_stage, 16 * m, cudaMemcpyDeviceToHost,
                                 s->stream));
    }
    return SV_OK;
}

sv_status sv_copy_state(sv_state *s, void *dst, size_t bytes) {
    if (!s || !dst) return fail(SV_ERR_ARG, "NULL argument");
    if (bytes != s->bytes) return fail(SV_ERR_ARG, "bytes must equal the state size");
    sv_status st = copy_out(s, dst);
    if (st != SV_OK) return st;
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    return SV_OK;
}

sv_status sv_download(sv_state *s, void *dst, size_t bytes) {
    if (!s || !dst) return fail(SV_ERR_ARG, "NULL argument");
    if (bytes != s->bytes) return fail(SV_ERR_ARG, "bytes must equal the state size");
    return copy_out(s, dst);
}

sv_status sv_export_c128(sv_state *s, void *dev_dst, size_t bytes) {
    if (!s || !dev_dst) return fail(SV_ERR_ARG, "NULL argument");
    if (s->prec == SV_C64) return fail(SV_ERR_ARG, "sv_export_c128 needs a complex128 state");
    if (bytes != s->bytes) return fail(SV_ERR_ARG, "bytes must equal the state size");
    if (is_df(s)) CUDA_TRY(launch_from_df(s->buf, dev_dst, 1ull << s->n, s->stream));
    else CUDA_TRY(cudaMemcpyAsync(dev_dst, s->buf, bytes, cudaMemcpyDeviceToDevice, s->stream));
    return SV_OK;
}

sv_status sv_device_ptr(sv_state *s, void **ptr, size_t *bytes) {
    if (!s) return fail(SV_ERR_ARG, "state is NULL");
    if (ptr) *ptr = s->buf;
    if (bytes) *bytes = s->bytes;
    return SV_OK;
}

static sv_status check_device_error(sv_state *s) {
    int h = 0;
    CUDA_TRY(cudaMemcpyAsync(&h, s->d_err, sizeof(int), cudaMemcpyDeviceToHost, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    if (h) {
        CUDA_TRY(cudaMemsetAsync(s->d_err, 0, sizeof(int), s->stream));
        return fail(SV_ERR_TIMEOUT, "a bounded device wait of the tensor-core kernel gave up");
    }
    return SV_OK;
}

sv_status sv_sync(sv_state *s) {
    if (!s) return fail(SV_ERR_ARG, "state is NULL");
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    return check_device_error(s);
}

sv_status sv_set_tile(sv_state *s, int t) {
    if (!s) return fail(SV_ERR_ARG, "state is NULL");
    if (t != 0 && (t < part_tmin() || t > part_tmax(is_fp64(s))))
        return fail(SV_ERR_ARG, "tile_qubits out of range");
    s->tile = t;
    return SV_OK;
}

sv_status sv_plan_build(const sv_gate *gates, size_t n_gates, int n, sv_method m, int k, uint64_t seed,
                        int dfs_trials, sv_plan **out) {
    if (!out) return fail(SV_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (n < 1 || n > 36) return fail(SV_ERR_ARG, "n_qubits must be in [1, 36]");
    if (n_gates && !gates) return fail(SV_ERR_ARG, "gates is NULL");
    if (m < SV_PART_NONE || m > SV_PART_BEAM) return fail(SV_ERR_ARG, "bad method");
    std::unique_ptr<sv_plan> p(new sv_plan());
    p->n = n;
    p->method = m;
    p->k = k;
    p->gates.resize(n_gates);
    int max_arity = 0;
    for (size_t i = 0; i < n_gates; i++) {
        const sv_gate &g = gates[i];
        if (g.kind >= SV_GATE_COUNT) return fail(SV_ERR_ARG, "gate " + std::to_string(i) + ": bad kind");
        const int want = gate_is_two_qubit(g.kind) ? 2 : 1;
        if (g.arity != want) return fail(SV_ERR_ARG, "gate " + std::to_string(i) + ": arity does not match kind");
        GateRef &r = p->gates[i];
        r.kind = g.kind;
        r.arity = g.arity;
        r.theta = g.theta;
        for (int j = 0; j < 3; j++) r.q[j] = j < g.arity ? (int)g.q[j] : 0;
        for (int j = 0; j < g.arity; j++)
            if (g.q[j] >= (uint32_t)n) return fail(SV_ERR_ARG, "gate " + std::to_string(i) + ": qubit out of range");
        if (g.arity == 2 && g.q[0] == g.q[1]) return fail(SV_ERR_ARG, "gate " + std::to_string(i) + ": repeated qubit");
        max_arity = std::max(max_arity, (int)g.arity);
    }
    if (m != SV_PART_NONE) {
        if (k < 1) return fail(SV_ERR_ARG, "k must be >= 1");
        if (max_arity > k) return fail(SV_ERR_PARTITION, "a gate has more qubits than k");
        Dag dag;
        std::string err;
        if (!build_dag(p->gates, n, dag, err)) return fail(SV_ERR_ARG, err);
        if (m == SV_PART_NAT) p->pog = part_nat(dag, k);
        else if (m == SV_PART_DFS) p->pog = part_dfs(dag, k, seed, dfs_trials);
        else if (m == SV_PART_DAGP) p->pog = part_dagp(dag, k);
        else if (m == SV_PART_BEAM) p->pog = part_beam(dag, k, dfs_trials);
        else if (!part_exact(dag, k, p->pog, err)) return fail(SV_ERR_ARG, err);
        for (uint32_t x : p->pog) p->n_parts = std::max(p->n_parts, x + 1);
        std::vector<uint64_t> pm(p->n_parts, 0), nd(p->n_parts, 0);
        for (size_t i = 0; i < n_gates; i++) {
            pm[p->pog[i]] |= dag.qmask[i];
            nd[p->pog[i]] |= tile_need(p->gates[i]);
        }
        for (uint64_t m : pm) p->max_part = std::max(p->max_part, __builtin_popcountll(m));
        for (uint64_t m : nd) p->max_tile = std::max(p->max_tile, __builtin_popcountll(m));
    } else {
        p->pog.resize(n_gates);
        for (size_t i = 0; i < n_gates; i++) p->pog[i] = (uint32_t)i;
        p->n_parts = (uint32_t)n_gates;
    }
    *out = p.release();
    return SV_OK;
}

sv_status sv_plan_build_ml(const sv_gate *gates, size_t n_gates, int n, sv_method m1, int k1, sv_method m2, int k2,
                           uint64_t seed, int dfs_trials, sv_plan **out) {
    if (!out) return fail(SV_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (m1 == SV_PART_NONE || m2 < SV_PART_NAT || m2 > SV_PART_BEAM)
        return fail(SV_ERR_ARG, "both levels need a part builder");
    if (k2 < 1 || k2 > k1) return fail(SV_ERR_ARG, "k2 must be in [1, k1]");
    sv_plan *p = nullptr;
    sv_status st = sv_plan_build(gates, n_gates, n, m1, k1, seed, dfs_trials, &p);
    if (st != SV_OK) return st;
    std::unique_ptr<sv_plan> hold(p);
    for (const GateRef &g : p->gates)
        if (g.arity > k2) return fail(SV_ERR_PARTITION, "a gate has more qubits than k2");
    std::vector<uint32_t> outer, inner;
    std::string err;
    if (!part_multilevel(p->gates, n, (int)m1, k1, (int)m2, k2, seed, dfs_trials, outer, inner, err))
        return fail(SV_ERR_ARG, err);
    if (outer != p->pog) return fail(SV_ERR_INTERNAL, "first-level partition differs from the plan's");
    p->inner = std::move(inner);
    for (uint32_t x : p->inner) p->n_inner = std::max(p->n_inner, x + 1);
    p->k2 = k2;
    *out = hold.release();
    return SV_OK;
}

sv_status sv_plan_export_inner(const sv_plan *p, uint32_t *inner, size_t n_gates, uint32_t *n_inner) {
    if (!p) return fail(SV_ERR_ARG, "plan is NULL");
    if (n_gates != p->gates.size()) return fail(SV_ERR_ARG, "n_gates does not match the plan");
    if (p->inner.empty() && n_gates) return fail(SV_ERR_ARG, "the plan has one level");
    if (inner && n_gates) std::memcpy(inner, p->inner.data(), sizeof(uint32_t) * n_gates);
    if (n_inner) *n_inner = p->n_inner;
    return SV_OK;
}

sv_status sv_plan_export(const sv_plan *p, uint32_t *pog, size_t n_gates, uint32_t *n_parts) {
    if (!p) return fail(SV_ERR_ARG, "plan is NULL");
    if (n_gates != p->gates.size()) return fail(SV_ERR_ARG, "n_gates does not match the plan");
    if (pog && n_gates) std::memcpy(pog, p->pog.data(), sizeof(uint32_t) * n_gates);
    if (n_parts) *n_parts = p->n_parts;
    return SV_OK;
}

// Program variants of a plan (besides precision and tile): bit 0 = tensor-core
// dense parts (complex64 only), bit 1 = two of them per pass where they fit
// one tile, bits 4-7 = register bits per thread (the flags' whole field: what
// compile_program has no program for it refuses), and the bits below.
constexpr int kModeWhole = 4;   // all gates as one part (the tile is the whole state)
constexpr int kModeJit = 8;     // for the specialised kernels (outer_diag), no interpreter stream
constexpr int kModeRefine = 256;   // the plan's parts cut and joined (refine_parts)
static int mode_R(int mode) { return (mode >> 4) & 15; }

static sv_status get_host_program(sv_plan *p, bool fp64, int t, int mode, const Program **out) {
    std::lock_guard<std::recursive_mutex> lk(p->mu);
    auto key = std::make_tuple(fp64, t, mode);
    auto it = p->host_progs.find(key);
    if (it == p->host_progs.end()) {
        std::unique_ptr<Program> prog(new Program());
        std::string err;
        const bool refined = (mode & kModeRefine) && p->max_part <= t;   // else refused below
        const bool own = (mode & kModeWhole) || refined;
        std::vector<uint32_t> pog;
        uint32_t n_parts = p->n_parts;
        if (mode & kModeWhole) {
            pog.assign(p->gates.size(), 0u);
            n_parts = 1;
        } else if (refined) {
            n_parts = refine_parts(p->gates, p->n, p->pog, p->n_parts, fp64, t, pog);
        }
        if (!compile_program(p->gates, p->n, own ? pog : p->pog, n_parts, fp64, t, mode_R(mode),
                             mode & 3, *prog, err, p->inner.empty() ? nullptr : &p->inner, (mode & kModeJit) != 0,
                             refined))
            return fail(SV_ERR_PARTITION, err);
        it = p->host_progs.emplace(key, std::move(prog)).first;
    }
    *out = it->second.get();
    return SV_OK;
}

// A smaller tile for a state that gives fewer than two tiles per SM, down to
// 2^8 amplitudes and the plan's largest part.
static int small_tiles(const sv_plan *p, int t) {
    while (t > 8 && t > p->max_part && (p->n <= t || (1ull << (p->n - t)) < 2 * 152)) t--;
    return t;
}

// The variant of the flags with the precision's default register bits unless
// given (sources; without kModeJit, what stats_mode says).
static int dense_mode(uint32_t flags, bool fp64) {
    const bool tc = (flags & SV_FLAG_TC_DENSE) && !fp64;
    const int R = (int)((flags >> 8) & 0xFu);
    return (tc ? 1 : 0) | ((tc && (flags & SV_FLAG_TC_PAIRS)) ? 2 : 0) | kModeJit | ((R ? R : part_R(fp64)) << 4);
}

// Tile (t_user, 0 = the default) and variant of the kernels that an apply (or
// sv_plan_specialise) compiles for a plan. With tile and register bits left to the library they go by the
// state's size (measured on layered and parameterised circuits, 20 layers):
//  * complex64 up to 19 qubits: 2^4 amplitudes per thread instead of 2^5 give
//    the SMs twice the warps where a pass is a tile or less per SM (14 to 19
//    qubits: 8 to 17 % shorter applies; even at 20 and 21, 5 to 13 % longer
//    above), and up to 17 qubits half the tile (15 to 30 % shorter at 12 to
//    16 qubits; even at 18); at 20 qubits twice the tile, 128 tiles of 152
//    SMs in one wave (k = 10: 130 -> 90 us layered, 155 -> 133 parameterised;
//    at 19 and 21 even to 60 % longer);
//  * double-float: 2^3 amplitudes per thread; with 2^4 the straight-line code
//    (about 40 instructions per amplitude and gate) outran the instruction
//    cache (4.6 of 7 stall cycles; 25 qubits: 12.6 against 8.3 ms, on 2^12
//    tiles, which above 21 qubits are 8 to 14 % faster than 2^11);
//  * complex128: small states in tiles down to 2^8 amplitudes until there
//    are two per SM (14 qubits, 20 layers: 385 -> 173 us), since an SM has
//    about two FP64 lanes and its tiles' arithmetic sets the time.
// Multi-level plans keep the register bits their second level may use.
static int spec_mode(const sv_plan *p, sv_precision prec, uint32_t flags, int t_user, int &t) {
    const bool fp64 = prec != SV_C64;
    t = t_user ? t_user : default_tile(fp64, p->max_part);
    int mode = dense_mode(flags, fp64);
    // a part's controls and two-qubit phases need not be in its tile
    if (!t_user && p->inner.empty()) t = std::max(default_tile(fp64, p->max_tile), p->max_part);
    if (t > part_tmax(fp64)) t = part_tmax(fp64);
    // (a complex128 state in L2 is bound by FP64 work alone: a 20-qubit QFT
    // takes 455 us on joined parts, 445 on its own)
    if (p->inner.empty() && !(mode & 3) && !(prec == SV_C128 && p->n <= 21)) mode |= kModeRefine;
    if (t_user || ((flags >> 8) & 0xFu) || !p->inner.empty()) return mode;
    int R = part_R(fp64);
    if (!fp64) {
        if (p->n <= 20) R = 4;
        if (p->n <= 17 && t == 12 && p->max_part < 12) t = 11;
        if (p->n == 20) t = 13;
    } else if (prec == SV_C128DF) {
        R = 3;
        if (p->n >= 22) t = part_tmax(true);
    } else if (small_tiles(p, t) < t) {
        t = small_tiles(p, t);
        R = 3;
    }
    return (mode & ~(15 << 4)) | (R << 4);
}

// Tile and variant of an apply on the interpreter (no register bits given).
//  * Multi-level plans keep the register bits their second level may use.
//  * A complex64 state of at most 13 qubits on its default tile is one tile:
//    all gates become one part, in their order, so the apply is one launch
//    that keeps the state on chip from the first gate to the last. At 10
//    qubits 2^3 amplitudes per thread (15 layers: 34 -> 31 us, parameterised
//    52 -> 49; at 11 and 12 qubits 38 -> 38, 82 -> 92). At 12 and 13 qubits
//    one SM's issue (about 0.17 and 0.25 us a gate) takes longer than the
//    passes of a plan with enough gates to a part (about 2 us a pass and 0.13
//    us a gate on 2^10 tiles): k = 10, 12 qubits 54 -> 47 us, parameterised
//    82 -> 70, but with k = 6 and 33 gates to a part 82 -> 92; 13 qubits 78 ->
//    50 and 134 -> 78, with k = 6 and 31 gates to a part 134 -> 104.
//  * A small complex128 state is cut into tiles down to 2^8 amplitudes until
//    there are two per SM: an SM has about two FP64 lanes, so its tiles'
//    arithmetic sets the time, and 14 qubits on 2^11 tiles keep 8 of 152 SMs
//    busy (the 840-gate layered circuit: 1.11 ms; on 2^8 tiles 0.49 ms).
//  * A complex64 state of 14 to 18 qubits is cut into smaller tiles while
//    there is no more than one per SM, of 2^3 amplitudes per thread up to 17
//    qubits: 15 layers, k = 10, in us on 2^12 / 2^11 / 2^10 tiles with 2^4 and
//    on 2^10 with 2^3 amplitudes: 14 qubits 79 / 65 / 66 / 56, 17 qubits 102 /
//    83 / 91 / 80 (parameterised 153 / 122 / 124 / 114); 18 qubits 111 / 93 /
//    138 / 129, 19 qubits 117 / 149 / 170 / 168.
// whole: false for the plan's own parts where they would become one.
static int interp_mode(const sv_plan *p, bool fp64, uint32_t flags, int t_user, int &t, bool whole = true) {
    const int tc = dense_mode(flags, fp64) & 3;
    const bool ml = !p->inner.empty();
    int R = ml ? part_R(fp64) : interp_R(fp64);
    t = t_user ? t_user : default_tile(fp64, p->max_part);
    if (t_user || ml) return tc | (R << 4);
    const bool cut = p->n >= 12 && p->max_part <= 10 && p->gates.size() >= (p->n == 12 ? 40 : 20) * (size_t)p->n_parts;
    if (whole && !fp64 && p->n <= part_tmax(false) && !cut && !(tc && p->n >= DENSE_K + DENSE_COLS)) {
        t = p->n;
        if (t == 10) R = 3;
        return kModeWhole | (R << 4);
    }
    if (fp64) {
        t = small_tiles(p, t);
    } else if (p->n <= 17 && p->max_part <= 10) {
        t = 10;
        R = 3;
    } else if (t == 12 && p->max_part < 12 && p->n <= 18) {
        t = 11;
    }
    return tc | (R << 4);
}

// Tile and variant of the program that sv_plan_stats and sv_plan_flops
// describe: the one that an apply with these flags runs, so that a caller who
// asks for the statistics first (on a thread that plans) has compiled it for
// the apply; but the plan's own parts where the apply makes them one, and the
// default shape for register bits that the interpreter does not take and for
// double-float states (without SV_FLAG_SPECIALISE).
static int stats_mode(const sv_plan *p, sv_precision prec, uint32_t flags, int t_user, int &t) {
    const bool fp64 = prec != SV_C64;
    if (flags & SV_FLAG_SPECIALISE) return spec_mode(p, prec, flags, t_user, t);
    if (!((flags >> 8) & 0xFu) && prec != SV_C128DF) return interp_mode(p, fp64, flags, t_user, t, false);
    t = t_user ? t_user : default_tile(fp64, p->max_part);
    return dense_mode(flags, fp64) & ~kModeJit;
}

sv_status sv_plan_stats(sv_plan *p, sv_precision prec, int t, uint32_t flags, uint32_t *passes, uint32_t *phases,
                        uint32_t *ops, uint32_t *dense) {
    if (!p) return fail(SV_ERR_ARG, "plan is NULL");
    const bool fp64 = prec != SV_C64;
    if (t != 0 && (t < part_tmin() || t > part_tmax(fp64))) return fail(SV_ERR_ARG, "tile_qubits out of range");
    const int mode = stats_mode(p, prec, flags, t, t);
    if (p->method == SV_PART_NONE || p->n < part_tmin() || (flags & SV_FLAG_GATEWISE)) {
        if (passes) *passes = (uint32_t)p->gates.size();
        if (phases) *phases = 0;
        if (ops) *ops = 0;
        if (dense) *dense = 0;
        return SV_OK;
    }
    const Program *prog = nullptr;
    sv_status st = get_host_program(p, fp64, t, mode, &prog);
    if (st != SV_OK) return st;
    if (passes) *passes = (uint32_t)prog->kind.size();
    if (phases) *phases = (uint32_t)prog->phases.size();
    if (ops) *ops = (uint32_t)prog->ops.size();
    if (dense) *dense = (uint32_t)(prog->dense.size() + prog->pairs.size());
    return SV_OK;
}

// The plan's specialised part kernels for (precision, tile, dense mode),
// compiled and loaded on first use.
static sv_status get_jit_program(sv_plan *p, sv_precision prec, int t, int mode, const Program *hp,
                                 JitProgram **out) {
    std::lock_guard<std::recursive_mutex> lk(p->mu);
    auto key = std::make_tuple((int)prec, t, mode);
    auto it = p->jit_progs.find(key);
    if (it == p->jit_progs.end()) {
        std::unique_ptr<JitProgram> jp(new JitProgram());
        std::string err;
        if (!jit_compile(*hp, *jp, err, true, prec == SV_C128DF))
            return fail(SV_ERR_CUDA, "specialised part kernels: " + err);
        it = p->jit_progs.emplace(key, std::move(jp)).first;
    }
    *out = it->second.get();
    return SV_OK;
}

sv_status sv_plan_specialise(sv_plan *p, sv_precision prec, int t, uint32_t flags, int load, double *compile_s) {
    if (!p) return fail(SV_ERR_ARG, "plan is NULL");
    const bool fp64 = prec != SV_C64;
    if (t != 0 && (t < part_tmin() || t > part_tmax(fp64))) return fail(SV_ERR_ARG, "tile_qubits out of range");
    const int mode = spec_mode(p, prec, flags, t, t);
    const Program *hp = nullptr;
    sv_status st = get_host_program(p, fp64, t, mode, &hp);
    if (st != SV_OK) return st;
    if (load) {
        JitProgram *jp = nullptr;
        st = get_jit_program(p, prec, t, mode, hp, &jp);
        if (st != SV_OK) return st;
        if (compile_s) *compile_s = jp->compile_s;
        return SV_OK;
    }
    JitProgram jp;
    std::string err;
    if (!jit_compile(*hp, jp, err, false, prec == SV_C128DF))
        return fail(SV_ERR_CUDA, "specialised part kernels: " + err);
    if (compile_s) *compile_s = jp.compile_s;
    return SV_OK;
}

sv_status sv_plan_source(sv_plan *p, sv_precision prec, int t, uint32_t flags, uint32_t part, char *buf, size_t cap,
                         size_t *len) {
    if (!p) return fail(SV_ERR_ARG, "plan is NULL");
    const bool fp64 = prec != SV_C64;
    if (t != 0 && (t < part_tmin() || t > part_tmax(fp64))) return fail(SV_ERR_ARG, "tile_qubits out of range");
    int mode = dense_mode(flags, fp64);
    if (flags & SV_FLAG_SPECIALISE) mode = spec_mode(p, prec, flags, t, t);
    else if (t == 0) t = default_tile(fp64, p->max_part);
    const Program *hp = nullptr;
    sv_status st = get_host_program(p, fp64, t, mode, &hp);
    if (st != SV_OK) return st;
    if (part >= hp->parts.size()) return fail(SV_ERR_ARG, "part index out of range");
    const std::string src = jit_part_source(*hp, part, prec == SV_C128DF);
    if (len) *len = src.size();
    if (buf && cap) {
        const size_t m = std::min(cap - 1, src.size());
        std::memcpy(buf, src.data(), m);
        buf[m] = '\0';
    }
    return SV_OK;
}

sv_status sv_plan_flops(sv_plan *p, sv_precision prec, int t, uint32_t flags, double *alu_flops,
                        double *tensor_flops) {
    if (!p) return fail(SV_ERR_ARG, "plan is NULL");
    const bool fp64 = prec != SV_C64;
    if (t != 0 && (t < part_tmin() || t > part_tmax(fp64))) return fail(SV_ERR_ARG, "tile_qubits out of range");
    const int mode = stats_mode(p, prec, flags, t, t);
    double a = 0.0, b = 0.0;
    if (p->method == SV_PART_NONE || p->n < part_tmin() || (flags & SV_FLAG_GATEWISE)) {
        // one general matrix per gate: 14 flops per amplitude for a 2x2, 30 for a 4x4
        for (const GateRef &g : p->gates) a += g.arity == 1 ? 14.0 : 30.0;
    } else {
        const Program *hp = nullptr;
        sv_status st = get_host_program(p, fp64, t, mode, &hp);
        if (st != SV_OK) return st;
        program_flops(*hp, a, b, (mode & kModeJit) != 0);
    }
    const double N = std::ldexp(1.0, p->n);
    if (alu_flops) *alu_flops = a * N;
    if (tensor_flops) *tensor_flops = b * N;
    return SV_OK;
}

sv_status sv_plan_destroy(sv_plan *p) {
    if (!p) return fail(SV_ERR_ARG, "plan is NULL");
    for (auto &kv : p->jit_progs) jit_release(*kv.second);
    int cur = 0;
    cudaGetDevice(&cur);
    for (auto &kv : p->dev_progs) {   // no apply of the plan may be in flight
        cudaSetDevice(kv.second.dev);
        dev_free(kv.second.d_stream, 0);
        dev_free(kv.second.d_windows, 0);
        dev_free(kv.second.d_aimg, 0);
        dev_free(kv.second.d_pimg, 0);
    }
    cudaSetDevice(cur);
    delete p;
    return SV_OK;
}

static void free_dev(DevProgram &d, cudaStream_t st) {
    dev_free(d.d_stream, st);
    dev_free(d.d_windows, st);
    dev_free(d.d_aimg, st);
    dev_free(d.d_pimg, st);
}

static sv_status get_dev_program(sv_state *s, sv_plan *p, int t, int mode, const Program **hp,
                                 const DevProgram **dp) {
    std::lock_guard<std::recursive_mutex> lk(p->mu);
    const bool fp64 = is_fp64(s);
    sv_status st = get_host_program(p, fp64, t, mode, hp);
    if (st != SV_OK) return st;
    auto key = std::make_tuple(s->dev, fp64, t, mode);
    auto it = p->dev_progs.find(key);
    if (it == p->dev_progs.end()) {
        const Program &prog = **hp;
        DevProgram d;
        d.dev = s->dev;
        cudaError_t e = upload_vec(reinterpret_cast<void **>(&d.d_aimg), prog.a_img, s->stream);
        if (e == cudaSuccess) e = upload_vec(reinterpret_cast<void **>(&d.d_pimg), prog.pair_img, s->stream);
        if (e == cudaSuccess && !(mode & kModeJit) && !prog.parts.empty())
            e = upload_lowered(prog, d, s->stream);
        // the program is shared by every state that applies the plan, on any
        // stream: it is complete before it is published
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
        if (e != cudaSuccess) {
            cudaGetLastError();
            free_dev(d, s->stream);
            return fail(e == cudaErrorMemoryAllocation ? SV_ERR_OOM : SV_ERR_CUDA,
                        std::string("program upload: ") + cudaGetErrorString(e));
        }
        it = p->dev_progs.emplace(key, d).first;
    }
    *dp = &it->second;
    return SV_OK;
}

static sv_status apply_gatewise(sv_state *s, sv_plan *p) {
    const bool fp64 = is_fp64(s);
    std::unique_lock<std::recursive_mutex> lk(p->mu);
    if (p->mats.size() != p->gates.size()) {
        p->mats.assign(p->gates.size(), {});
        for (size_t i = 0; i < p->gates.size(); i++) {
            const GateRef &g = p->gates[i];
            if (g.arity == 1) {
                p->mats[i].resize(8);
                gate_matrix_1q(g.kind, g.theta, p->mats[i].data());
            } else {
                p->mats[i].resize(32);
                gate_matrix_2q(g.kind, g.theta, p->mats[i].data());
            }
        }
    }
    lk.unlock();   // the matrices are complete and only read from here
    for (size_t i = 0; i < p->gates.size(); i++) {
        const GateRef &g = p->gates[i];
        cudaError_t e;
        if (g.arity == 1) e = launch_gate1(fp64, s->buf, s->n, g.q[0], p->mats[i].data(), s->stream);
        else e = launch_gate2(fp64, s->buf, s->n, g.q[0], g.q[1], p->mats[i].data(), s->stream);
        if (e != cudaSuccess) return fail(SV_ERR_CUDA, std::string("gate launch: ") + cudaGetErrorString(e));
    }
    return SV_OK;
}

// A circuit on fewer than 10 qubits in one launch (at most 640 ops; 384 in
// complex128). The op records are made at the plan's first apply for the
// precision and kept in the plan; the launch takes a copy.
static sv_status apply_small(sv_state *s, sv_plan *p) {
    if (p->gates.empty()) return SV_OK;
    const bool fp64 = is_fp64(s);
    const void *ops;
    uint32_t n_ops;
    auto made = [&](auto &v, auto list) {
        using Real = decltype(list);
        std::lock_guard<std::recursive_mutex> lk(p->mu);
        if (v.empty()) {
            v = small_ops<Real>(p);
            v.resize(v.size() + small_most(fp64));   // launch_small copies whole records lists
        }
        ops = v.data();
        n_ops = (uint32_t)(v.size() - small_most(fp64));
    };
    if (fp64) made(p->small64, double());
    else made(p->small32, float());
    CUDA_TRY(launch_small(fp64, s->buf, s->n, ops, n_ops, s->stream));
    return SV_OK;
}

sv_status sv_apply_parts(sv_state *s, sv_plan *p, uint32_t flags) {
    if (!s || !p) return fail(SV_ERR_ARG, "NULL argument");
    if (p->n != s->n) return fail(SV_ERR_ARG, "plan and state qubit counts differ");
    sv_status st = SV_OK;
    if (is_df(s)) {
        if ((flags & SV_FLAG_GATEWISE) || p->method == SV_PART_NONE || s->n < part_tmin())
            return fail(SV_ERR_ARG, "a double-float state runs parts of a partitioned plan (n >= 10) only");
        flags = (flags | SV_FLAG_SPECIALISE) & ~SV_FLAG_TC_DENSE;
    }
    if ((flags & SV_FLAG_GATEWISE) || p->method == SV_PART_NONE) {
        st = apply_gatewise(s, p);
    } else if (s->n < part_tmin()) {
        st = apply_small(s, p);
    } else {
        const bool fp64 = is_fp64(s);
        const bool jit = (flags & SV_FLAG_SPECIALISE) != 0;
        int t = 0;
        const int mode = jit ? spec_mode(p, s->prec, flags, s->tile, t) : interp_mode(p, fp64, flags, s->tile, t);
        const Program *hp = nullptr;
        const DevProgram *dp = nullptr;
        st = get_dev_program(s, p, t, mode, &hp, &dp);
        if (st != SV_OK) return st;
        JitProgram *jp = nullptr;
        if (((flags >> 8) & 0xFu) && !jit)
            return fail(SV_ERR_ARG, "register bits other than the default need SV_FLAG_SPECIALISE");
        if (jit && !hp->parts.empty()) {
            st = get_jit_program(p, s->prec, t, mode, hp, &jp);
            if (st != SV_OK) return st;
        }
        if (!hp->dense.empty() || !hp->pairs.empty()) {
            const size_t need = hp->dense.size() + hp->pairs.size() + 1;
            if (s->dnorm_cap < need) {
                dev_free(s->d_dnorm, s->stream);
                s->d_dnorm = nullptr;
                s->dnorm_cap = 0;
                cudaError_t e = dev_alloc(reinterpret_cast<void **>(&s->d_dnorm), sizeof(double) * need, s->stream);
                if (e != cudaSuccess) {
                    cudaGetLastError();
                    return fail(SV_ERR_OOM, std::string("norm accumulators: ") + cudaGetErrorString(e));
                }
                s->dnorm_cap = need;
            }
            CUDA_TRY(cudaMemsetAsync(s->d_dnorm, 0, sizeof(double) * need, s->stream));
        }
        uint32_t didx = 0;   // tensor-core passes of this apply, in order (norm accumulators)
        for (size_t i = 0; i < hp->kind.size(); i++) {
            const uint32_t j = hp->index[i];
            cudaError_t e;
            if (hp->kind[i] == 0 && jp)
                e = jit_launch(*jp, j, s->buf, hp->n_tiles[j], s->stream);
            else if (hp->kind[i] == 0)
                e = (fp64 ? launch_part_f64 : launch_part_f32)(hp->t, hp->R, s->buf, dp->parts[j], dp->d_stream,
                                                               dp->d_windows, hp->n_tiles[j], s->stream);
            else if (hp->kind[i] == 1)
                e = launch_dense6(s->buf, hp->dense[j], dp->d_aimg + (size_t)j * DENSE_A_BYTES, hp->dense_tiles[j],
                                  s->d_err, s->d_dnorm, didx++, s->stream);
            else
                e = launch_dense_pair(s->buf, hp->pairs[j], dp->d_pimg + (size_t)j * 2 * DENSE_A_BYTES,
                                      hp->pair_tiles[j], s->d_err, s->d_dnorm, didx++, s->stream);
            if (e != cudaSuccess) return fail(SV_ERR_CUDA, std::string("part launch: ") + cudaGetErrorString(e));
        }
    }
    if (st != SV_OK) return st;
    if (flags & SV_FLAG_SYNC) {
        CUDA_TRY(cudaStreamSynchronize(s->stream));
        return check_device_error(s);
    }
    return SV_OK;
}

sv_status sv_measure_probs(sv_state *s, void *dev_out, int out_fp64, double *norm_out) {
    if (!s) return fail(SV_ERR_ARG, "state is NULL");
    double *norm = s->d_partials + kProbBlocks;
    if (norm_out) {
        if (!s->h_slot) s->h_slot = result_slots().take();
        if (s->h_slot) norm = s->h_slot;
    }
    CUDA_TRY(launch_probs(is_fp64(s), s->buf, s->n, dev_out, out_fp64, s->d_partials, kProbBlocks, norm, s->stream,
                          is_df(s), reinterpret_cast<uint32_t *>(s->d_err + 1)));
    if (norm_out) {
        if (norm != s->h_slot)
            CUDA_TRY(cudaMemcpyAsync(&s->h_norm, norm, sizeof(double), cudaMemcpyDeviceToHost, s->stream));
        CUDA_TRY(cudaStreamSynchronize(s->stream));
        *norm_out = norm == s->h_slot ? *static_cast<volatile double *>(norm) : s->h_norm;
    }
    return SV_OK;
}

sv_status sv_alu_probe(int fp64, double *flops_per_s) {
    if (!flops_per_s) return fail(SV_ERR_ARG, "flops_per_s is NULL");
    CUDA_TRY(alu_probe(fp64 != 0, flops_per_s, nullptr));
    return SV_OK;
}

sv_status sv_measure_summary(sv_state *s, double *norm_out, double *p0_out, uint64_t *argmax_out,
                             double *pmax_out) {
    if (!s) return fail(SV_ERR_ARG, "state is NULL");
    double *scratch = s->d_partials + kSummaryAt, *d_out = scratch + 3 * kProbBlocks;
    if (!s->h_slot) s->h_slot = result_slots().take();
    CUDA_TRY(launch_summary(is_fp64(s), s->buf, s->n, scratch, kProbBlocks, s->h_slot ? s->h_slot : d_out, s->stream,
                            is_df(s), reinterpret_cast<uint32_t *>(s->d_err + 2)));
    double h[4];
    if (!s->h_slot) CUDA_TRY(cudaMemcpyAsync(h, d_out, sizeof(h), cudaMemcpyDeviceToHost, s->stream));
    CUDA_TRY(cudaStreamSynchronize(s->stream));
    if (s->h_slot)
        for (int i = 0; i < 4; i++) h[i] = static_cast<volatile double *>(s->h_slot)[i];
    if (norm_out) *norm_out = h[0];
    if (p0_out) *p0_out = h[1];
    if (pmax_out) *pmax_out = h[2];
    if (argmax_out) std::memcpy(argmax_out, &h[3], sizeof(uint64_t));
    return SV_OK;
}

}  // extern "C"
