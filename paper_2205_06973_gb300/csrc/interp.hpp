// The op stream that the gate-list interpreter runs: the planner's program
// (program.hpp) lowered for a number format and register-bit count.
//
// An op is one record (16 bytes for float) with its opcode, thread condition
// and coefficients together, so that a warp fetches an op with one load; the
// opcode holds the register bit, so that the kernel reaches the op's code
// with one indirect branch.
#pragma once
#include <cstdint>
#include <vector>

#include "program.hpp"

namespace hisv {

// Opcode = kind * 8 + register bit; IK_CP = kind * 8 + index of the register
// bit pair (a < b): b (b - 1) / 2 + a (up to 15 pairs, two opcode rows).
enum InterpKind : uint32_t {
    IK_H = 0,
    IK_RX0, IK_RX1,   // OP_RXS forms; c[0] = t
    IK_RY0, IK_RY1,   // OP_RYS forms; c[0] = t
    IK_U2,            // [[1, u], [v, w]]; table[arg..]: u, v, w (re, im)
    IK_SWAP,          // exchange the halves where the conditions hold: X, CX, CXT
    IK_P,             // phase c on the set half where the thread condition holds
    IK_CP, IK_CP2,    // phase c where both register bits are set
    IK_MISC,          // IM_*
};
enum InterpMisc : uint32_t {
    IM_TPH = IK_MISC * 8,   // per-thread phase *= c where the thread condition holds
    IM_DIAG,                // register amplitude i *= table[arg + 2 i] (re, im)
    IM_TAPPLY,              // multiply by the per-thread phase, reset it
    IM_TSG,                 // per-thread sign flips where the thread condition holds
    IM_TSAPPLY,             // negate where the per-thread sign is set, reset it
    IM_SIGN,                // negate where the register mask and the thread condition hold: Z, CZ
};

// arg: low half = thread-bit mask (all set: the condition holds; 0 = always),
// high half = register mask of IK_SWAP and IM_SIGN; for IK_U2 and IM_DIAG the
// table index (in reals).
template <typename Real> struct alignas(16) IOp {
    uint32_t code;
    uint32_t arg;
    Real c[2];
};
static_assert(sizeof(IOp<float>) == 16 && sizeof(IOp<double>) == 32, "IOp layout");

// A register phase with its shared-memory layout: swizzled offsets of the
// register and thread bits.
struct alignas(16) IPhase {
    uint16_t sreg[8];
    uint16_t sthr[MAX_TB];
    uint32_t op_begin;
    uint32_t op_count;
    uint32_t pad[2];
};
static_assert(sizeof(IPhase) == 64, "IPhase layout");

struct Program;
template <typename Real> struct Lowered {
    std::vector<IPhase> phases;
    std::vector<IOp<Real>> ops;
    std::vector<Real> table;   // 16-byte aligned entries (IM_DIAG, IK_U2)
};
// Lower every phase of the program (its parts keep their phase indices).
template <typename Real> void lower_program(const Program &prog, Lowered<Real> &out);

}  // namespace hisv
