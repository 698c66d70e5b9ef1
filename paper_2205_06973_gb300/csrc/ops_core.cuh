// Register-level gate arithmetic on a thread's 2^R amplitudes, with
// compile-time register bits. Self-contained (no standard or CUDA headers),
// so that both the library's kernels and the part kernels compiled for a
// plan at run time (NVRTC) use the same definitions.
//
// A thread holds 2^R amplitudes a[0..2^R) of its tile; register bit b of the
// index i is one tile slot (qubit).
#pragma once

namespace hisv {

// -v without arithmetic: for doubles a sign-bit flip (FP64 work otherwise).
template <typename Real>
__device__ __forceinline__ Real neg_of(Real v) { return -v; }
#if defined(__CUDA_ARCH__)
__device__ __forceinline__ double neg_of(double v) {
    return __hiloint2double(__double2hiint(v) ^ (int)0x80000000, __double2loint(v));
}
#endif

// (x + i y) times e^{i phi} by three shears (Paeth, Graphics Interface 1986),
// t = tan(phi / 2), s = sin(phi): three multiply-adds instead of two products
// and two multiply-adds. Used for complex128, whose kernels are bound by FP64
// work (24 qubits, 20 layers, k = 10: 29.9 -> 28.6 ms; largest error against
// exact arithmetic 1.87e-15 with products, 1.90e-15 with shears).
template <typename C, typename Real>
__device__ __forceinline__ void rot_in(C &v, Real t, Real s) {
    v.x = v.x - t * v.y;
    v.y = v.y + s * v.x;
    v.x = v.x - t * v.y;
}
// The same times i^Q first (exchange and sign of the parts).
template <int Q, typename C, typename Real>
__device__ __forceinline__ void rotq_in(C &v, Real t, Real s) {
    const Real x = v.x, y = v.y;
    if (Q == 1) { v.x = neg_of(y); v.y = x; }
    if (Q == 2) { v.x = neg_of(x); v.y = neg_of(y); }
    if (Q == 3) { v.x = y; v.y = neg_of(x); }
    rot_in(v, t, s);
}
template <int NR, int B, int Q, typename C, typename Real>
__device__ __forceinline__ void op_prot(C (&a)[NR], Real t, Real s) {
#pragma unroll
    for (int i = 0; i < NR; i++)
        if (i & (1 << B)) rotq_in<Q>(a[i], t, s);
}

// ------------------------------------------------------------------------
// register-bit operations; B, A are compile-time register bits
// ------------------------------------------------------------------------
// Hadamard without its 1/sqrt2: the planner folds the factor into the part's
// store factor, so each H costs one add and one subtract per amplitude pair.
template <int NR, int B, typename C>
__device__ __forceinline__ void op_h(C (&a)[NR]) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if (i & (1 << B)) continue;
        const int j = i | (1 << B);
        const C x = a[i], y = a[j];
        a[i].x = x.x + y.x; a[i].y = x.y + y.y;
        a[j].x = x.x - y.x; a[j].y = x.y - y.y;
    }
}

// Scaled rotations: the gate divided by its largest entry (the factor is
// applied once, with the part's store factor), so every output component is
// one multiply-add. F = form (see OP_RXS / OP_RYS / OP_U2S in program.hpp).
template <int NR, int B, int F, typename C, typename Real>
__device__ __forceinline__ void op_rxs(C (&a)[NR], Real t) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if (i & (1 << B)) continue;
        const int j = i | (1 << B);
        const C x = a[i], y = a[j];
        if (F == 0) {            // (x + (-it) y, y + (-it) x)
            a[i].x = x.x + t * y.y; a[i].y = x.y - t * y.x;
            a[j].x = y.x + t * x.y; a[j].y = y.y - t * x.x;
        } else {                 // (y + (it) x, x + (it) y)
            a[i].x = y.x - t * x.y; a[i].y = y.y + t * x.x;
            a[j].x = x.x - t * y.y; a[j].y = x.y + t * y.x;
        }
    }
}

template <int NR, int B, int F, typename C, typename Real>
__device__ __forceinline__ void op_rys(C (&a)[NR], Real t) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if (i & (1 << B)) continue;
        const int j = i | (1 << B);
        const C x = a[i], y = a[j];
        if (F == 0) {            // (x - t y, y + t x)
            a[i].x = x.x - t * y.x; a[i].y = x.y - t * y.y;
            a[j].x = y.x + t * x.x; a[j].y = y.y + t * x.y;
        } else {                 // (t x - y, x + t y)
            a[i].x = t * x.x - y.x; a[i].y = t * x.y - y.y;
            a[j].x = x.x + t * y.x; a[j].y = x.y + t * y.y;
        }
    }
}

template <int NR, int B, int F, typename C, typename Real>
__device__ __forceinline__ void op_u2s(C (&a)[NR], Real ur, Real ui, Real vr, Real vi, Real wr, Real wi) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if (i & (1 << B)) continue;
        const int j = i | (1 << B);
        const C x = a[i], y = a[j];
        if (F == 0) {            // (x + u y, v x + w y)
            a[i].x = x.x + ur * y.x - ui * y.y; a[i].y = x.y + ur * y.y + ui * y.x;
        } else {                 // (u x + y, v x + w y)
            a[i].x = y.x + ur * x.x - ui * x.y; a[i].y = y.y + ur * x.y + ui * x.x;
        }
        a[j].x = vr * x.x - vi * x.y + wr * y.x - wi * y.y;
        a[j].y = vr * x.y + vi * x.x + wr * y.y + wi * y.x;
    }
}

template <typename C, typename Real>
__device__ __forceinline__ void cmul_in(C &v, Real dr, Real di) {
    const Real x = v.x, y = v.y;
    v.x = x * dr - y * di;
    v.y = x * di + y * dr;
}

template <int NR, int B, typename C, typename Real>
__device__ __forceinline__ void op_p(C (&a)[NR], Real dr, Real di) {
#pragma unroll
    for (int i = 0; i < NR; i++)
        if (i & (1 << B)) cmul_in(a[i], dr, di);
}

template <int NR, int B, typename C>
__device__ __forceinline__ void op_z(C (&a)[NR]) {
#pragma unroll
    for (int i = 0; i < NR; i++)
        if (i & (1 << B)) { a[i].x = neg_of(a[i].x); a[i].y = neg_of(a[i].y); }
}

template <int NR, int A, int B, typename C, typename Real>
__device__ __forceinline__ void op_cp(C (&a)[NR], Real dr, Real di) {
#pragma unroll
    for (int i = 0; i < NR; i++)
        if ((i & (1 << A)) && (i & (1 << B))) cmul_in(a[i], dr, di);
}

template <int NR, int A, int B, typename C>
__device__ __forceinline__ void op_cz(C (&a)[NR]) {
#pragma unroll
    for (int i = 0; i < NR; i++)
        if ((i & (1 << A)) && (i & (1 << B))) { a[i].x = neg_of(a[i].x); a[i].y = neg_of(a[i].y); }
}

// Programmatic dependent launch: wait until the previous kernel on the stream
// has completed and its writes are visible; let the next one launch.
__device__ __forceinline__ void pdl_wait() {
#if defined(__CUDA_ARCH__)
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
#endif
}
__device__ __forceinline__ void pdl_launch() {
#if defined(__CUDA_ARCH__)
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
#endif
}

// Every amplitude negated where neg holds (a controlled Z of two thread bits):
// a product for single floats, selects (no FP64 work) for the wider forms.
template <int NR, typename C>
__device__ __forceinline__ void op_flip(C (&a)[NR], bool neg) {
#pragma unroll
    for (int i = 0; i < NR; i++) {
        if constexpr (sizeof(C) == 8) {
            const auto s = neg ? -1.0f : 1.0f;
            a[i].x = a[i].x * s;
            a[i].y = a[i].y * s;
        } else {
            a[i].x = neg ? neg_of(a[i].x) : a[i].x;
            a[i].y = neg ? neg_of(a[i].y) : a[i].y;
        }
    }
}

// Swizzled shared-memory index contribution of tile slot p. The swizzle XORs
// the slot bits above the bank group into the low bits (linear over GF(2)),
// so a warp whose lane bits sit on slots of distinct residues touches
// distinct banks: 8-byte elements use 4-bit groups, 16-byte elements 3-bit.
template <typename Real>
__device__ __forceinline__ unsigned int swz(int p) {
    if constexpr (sizeof(Real) == 4) return p < 4 ? (1u << p) : ((1u << p) | (1u << (p & 3)));
    else return p < 3 ? (1u << p) : ((1u << p) | (1u << (p % 3)));
}


}  // namespace hisv
