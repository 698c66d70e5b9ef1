// The gate-list interpreter's inner loop (shared by the part kernel and the
// batched kernels): a phase's ops on a thread's 2^R amplitudes.
//
// What bounds it is instruction supply. Every op has its own code per
// register bit (the amplitudes stay in registers, so the bit must be a
// compile-time index), and with 2^5 amplitudes per thread and two dispatch
// levels that code was larger than the SM's instruction cache: on a 21-qubit
// layered circuit (k = 10) 3.4 to 4.3 of 9 stall cycles per instruction were
// "no instruction" and a pass took 36 us. So the code is kept small: 2^4
// complex64 (2^3 complex128) amplitudes per thread, one packed instruction
// for both halves of an amplitude where the arithmetic allows it, one form
// per gate kind where the planner's can be reduced to another (interp.hpp),
// permutations as selects (a permutation of registers, or through shared
// memory, would cost more code or a round trip), one indirect branch per op.
// The next op's record is fetched while an op runs.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "interp.hpp"
#include "ops_core.cuh"
#include "packed.cuh"

namespace hisv {

template <typename Real> struct CT;
template <> struct CT<float> { typedef float2 T; };
template <> struct CT<double> { typedef double2 T; };

// One op record; p may point to shared or global memory.
__device__ __forceinline__ IOp<float> ld_op(const IOp<float> *p) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    IOp<float> o;
    o.code = __float_as_uint(v.x);
    o.arg = __float_as_uint(v.y);
    o.c[0] = v.z;
    o.c[1] = v.w;
    return o;
}
__device__ __forceinline__ IOp<double> ld_op(const IOp<double> *p) {
    const uint2 h = *reinterpret_cast<const uint2 *>(p);
    const double2 c = *reinterpret_cast<const double2 *>(&p->c[0]);
    IOp<double> o;
    o.code = h.x;
    o.arg = h.y;
    o.c[0] = c.x;
    o.c[1] = c.y;
    return o;
}

// H, RY and RX of one register bit; float amplitudes packed where no
// component changes place.
template <int NR, int B> __device__ __forceinline__ void in_h(float2 (&a)[NR]) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if (i & (1 << B)) continue;
        const int j = i | (1 << B);
        const float2 x = a[i], y = a[j];
        a[i] = add2(x, y);
        a[j] = sub2(x, y);
    }
}
template <int NR, int B> __device__ __forceinline__ void in_h(double2 (&a)[NR]) { op_h<NR, B>(a); }

template <int NR, int B, int F> __device__ __forceinline__ void in_ry(float2 (&a)[NR], float t) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if (i & (1 << B)) continue;
        const int j = i | (1 << B);
        const float2 x = a[i], y = a[j];
        if (F == 0) {
            a[i] = fma2(-t, y, x);
            a[j] = fma2(t, x, y);
        } else {
            a[i] = fma2(t, x, make_float2(-y.x, -y.y));
            a[j] = fma2(t, y, x);
        }
    }
}
template <int NR, int B, int F> __device__ __forceinline__ void in_ry(double2 (&a)[NR], double t) {
    op_rys<NR, B, F>(a, t);
}

// Exchange a[i] and a[i | bit B] where the register index has all bits of
// rm set and the thread condition holds: selects, so that no register is
// renamed differently on the paths of the op switch.
template <int NR, int B, typename C>
__device__ __forceinline__ void in_swap(C (&a)[NR], uint32_t rm, bool tc) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if (i & (1 << B)) continue;
        const int j = i | (1 << B);
        const bool p = tc && (i & rm) == rm;
        const C x = a[i], y = a[j];
        a[i].x = p ? y.x : x.x;
        a[i].y = p ? y.y : x.y;
        a[j].x = p ? x.x : y.x;
        a[j].y = p ? x.y : y.y;
    }
}

// v negated where p holds: a sign-bit flip (not FP64 work for doubles).
__device__ __forceinline__ float flip(float v, uint32_t m) { return __uint_as_float(__float_as_uint(v) ^ m); }
__device__ __forceinline__ double flip(double v, uint32_t m) {
    return __hiloint2double(__double2hiint(v) ^ (int)m, __double2loint(v));
}

// The ops of one phase header (hdr: in shared or global memory), at ops_at.
template <typename Real, int R>
__device__ __forceinline__ void run_ops(typename CT<Real>::T (&a)[1 << R], const char *hdr, uint32_t ops_at,
                                        uint32_t count,
                                        uint32_t tid, Real &tpr, Real &tpi, uint32_t &tsg) {
    constexpr int NR = 1 << R;
    if (count == 0) return;
    const IOp<Real> *const ops = reinterpret_cast<const IOp<Real> *>(hdr + ops_at);
    IOp<Real> op = ld_op(ops);
    for (uint32_t o = 1;; o++) {
        const IOp<Real> cur = op;
        if (o < count) op = ld_op(ops + o);
        const Real *const table = reinterpret_cast<const Real *>(hdr + cur.arg);   // IK_U2, IM_DIAG
        const uint32_t tm = cur.arg & 0xFFFFu;
        const bool tc = (tid & tm) == tm;
        switch (cur.code) {
// one case per register bit below R
#define HISV_BIT(K, B, BODY) \
    case (K) * 8 + (B):      \
        if constexpr ((B) < R) BODY; \
        break;
#define HISV_BITS(K, BODY0, BODY1, BODY2, BODY3, BODY4) \
    HISV_BIT(K, 0, BODY0) HISV_BIT(K, 1, BODY1) HISV_BIT(K, 2, BODY2) HISV_BIT(K, 3, BODY3) HISV_BIT(K, 4, BODY4)
#define HISV_EACH(K, CALL) HISV_BITS(K, CALL(0), CALL(1), CALL(2), CALL(3), CALL(4))
#define HISV_H(B) (in_h<NR, B>(a))
#define HISV_RX0(B) (op_rxs<NR, B, 0>(a, cur.c[0]))
#define HISV_RX1(B) (op_rxs<NR, B, 1>(a, cur.c[0]))
#define HISV_RY0(B) (in_ry<NR, B, 0>(a, cur.c[0]))
#define HISV_RY1(B) (in_ry<NR, B, 1>(a, cur.c[0]))
#define HISV_U2(B) \
    (op_u2s<NR, B, 0>(a, table[0], table[1], table[2], table[3], table[4], table[5]))
#define HISV_SWAP(B) (in_swap<NR, B>(a, cur.arg >> 16, tc))
#define HISV_P(B) (op_p<NR, B>(a, tc ? cur.c[0] : Real(1), tc ? cur.c[1] : Real(0)))
            HISV_EACH(IK_H, HISV_H)
            HISV_EACH(IK_RX0, HISV_RX0)
            HISV_EACH(IK_RX1, HISV_RX1)
            HISV_EACH(IK_RY0, HISV_RY0)
            HISV_EACH(IK_RY1, HISV_RY1)
            HISV_EACH(IK_U2, HISV_U2)
            HISV_EACH(IK_SWAP, HISV_SWAP)
            HISV_EACH(IK_P, HISV_P)
// one case per pair A < B of register bits below R
#define HISV_CP(A, B)                             \
    case IK_CP * 8 + (B) * ((B) - 1) / 2 + (A):   \
        if constexpr ((B) < R) op_cp<NR, A, B>(a, cur.c[0], cur.c[1]); \
        break;
            HISV_CP(0, 1)
            HISV_CP(0, 2) HISV_CP(1, 2)
            HISV_CP(0, 3) HISV_CP(1, 3) HISV_CP(2, 3)
            HISV_CP(0, 4) HISV_CP(1, 4) HISV_CP(2, 4) HISV_CP(3, 4)
#undef HISV_BIT
#undef HISV_BITS
#undef HISV_EACH
#undef HISV_H
#undef HISV_RX0
#undef HISV_RX1
#undef HISV_RY0
#undef HISV_RY1
#undef HISV_U2
#undef HISV_SWAP
#undef HISV_P
#undef HISV_CP
        case IM_TPH:
            if (tc) {
                const Real x = tpr, y = tpi;
                tpr = x * cur.c[0] - y * cur.c[1];
                tpi = x * cur.c[1] + y * cur.c[0];
            }
            break;
        case IM_DIAG:
#pragma unroll
            for (int i = 0; i < NR; i++) {
                if constexpr (sizeof(Real) == 4) {
                    if (i & 1) continue;
                    const float4 v = reinterpret_cast<const float4 *>(table)[i / 2];
                    cmul_in(a[i], v.x, v.y);
                    cmul_in(a[i + 1], v.z, v.w);
                } else {
                    const double2 v = reinterpret_cast<const double2 *>(table)[i];
                    cmul_in(a[i], v.x, v.y);
                }
            }
            break;
        case IM_TAPPLY:
#pragma unroll
            for (int i = 0; i < NR; i++) cmul_in(a[i], tpr, tpi);
            tpr = Real(1);
            tpi = Real(0);
            break;
        case IM_TSG:
            tsg ^= tc ? 0x80000000u : 0u;
            break;
        case IM_TSAPPLY:
#pragma unroll
            for (int i = 0; i < NR; i++) {
                a[i].x = flip(a[i].x, tsg);
                a[i].y = flip(a[i].y, tsg);
            }
            tsg = 0u;
            break;
        case IM_SIGN: {
            const uint32_t rm = cur.arg >> 16;
#pragma unroll
            for (int i = 0; i < NR; i++) {
                const uint32_t m = tc && (i & rm) == rm ? 0x80000000u : 0u;
                a[i].x = flip(a[i].x, m);
                a[i].y = flip(a[i].y, m);
            }
        } break;
        default:
            break;
        }
        if (o >= count) break;
    }
}

// XOR of the offsets off[j] over the set bits j of v (TB bits).
template <int TB>
__device__ __forceinline__ uint32_t xor_bits(uint32_t v, const uint16_t *off) {
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < TB; j++) s ^= (v >> j) & 1 ? off[j] : 0u;
    return s;
}

// A phase's layout for this thread: offset of its amplitude 0 and of each
// register bit.
template <int R, int TB> struct Slots {
    uint32_t thr, reg[R];
    __device__ __forceinline__ void load(const char *hdr, uint32_t tid) {
        union { uint4 q[3]; uint16_t h[24]; } u;
#pragma unroll
        for (int i = 0; i < 3; i++) u.q[i] = reinterpret_cast<const uint4 *>(hdr)[i];
#pragma unroll
        for (int b = 0; b < R; b++) reg[b] = u.h[b];
        thr = xor_bits<TB>(tid, u.h + 8);
    }
    __device__ __forceinline__ uint32_t at(int i) const {
        uint32_t o = thr;
#pragma unroll
        for (int b = 0; b < R; b++)
            if (i & (1 << b)) o ^= reg[b];
        return o;
    }
};

// The phases of one window (w: in shared or global memory) on the tile in
// buf. first: the tile's first phase, which loads without a transpose. sync()
// orders the tile's threads.
template <typename Real, int R, int TB, typename Sync>
__device__ __forceinline__ void run_window(typename CT<Real>::T (&a)[1 << R], typename CT<Real>::T *buf,
                                           Slots<R, TB> &S, const char *w, uint32_t n_phases, bool first,
                                           uint32_t tid, Real &tpr, Real &tpi, uint32_t &tsg, Sync &&sync) {
    constexpr int NR = 1 << R;
    for (uint32_t p = 0; p < n_phases; p++) {
        const uint4 h = *reinterpret_cast<const uint4 *>(w + 48);   // n_ops, bytes, flags, ops_at
        if (!(h.z & IPH_CONT)) {
            if (!first) {   // transpose through shared memory: write with the previous layout
                sync();
#pragma unroll
                for (int i = 0; i < NR; i++) buf[S.at(i)] = a[i];
                sync();
            }
            first = false;
            S.load(w, tid);
#pragma unroll
            for (int i = 0; i < NR; i++) a[i] = buf[S.at(i)];
            if (h.z & IPH_WRITE) S.load(w + sizeof(IPhase), tid);
        }
        run_ops<Real, R>(a, w, h.w, h.x, tid, tpr, tpi, tsg);
        w += h.y;
    }
}

// Copy a window into shared memory (all threads of the CTA; the caller
// synchronises).
__device__ __forceinline__ void copy_window(char *dst, const uint4 *__restrict__ stream, const IWindow &W, uint32_t tid,
                                            uint32_t nt) {
    for (uint32_t i = tid; i < W.bytes / 16; i += nt) reinterpret_cast<uint4 *>(dst)[i] = __ldg(stream + W.at + i);
}

}  // namespace hisv
