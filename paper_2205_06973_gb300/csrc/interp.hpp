// The instruction stream that the gate-list interpreter runs: the planner's
// program (program.hpp) lowered for a number format and register-bit count.
//
// A part's phases follow one another in the stream, each as a header with its
// shared-memory layout, its op records and the tables these refer to. An op
// is one record (16 bytes for float) with its opcode, thread condition and
// coefficients together, so that a warp fetches an op with one load; the
// opcode holds the register bit, so that the kernel reaches the op's code
// with one indirect branch. The stream is cut into windows that a CTA copies
// into shared memory as a whole: read from global memory op by op, a circuit
// that is run once waits for L2 at every eighth op and at every table (16
// parameterised 10-qubit circuits of up to 50 layers, a CTA each: 0.38 ms).
#pragma once
#include <cstdint>
#include <vector>

#include "program.hpp"

namespace hisv {

// Opcode = kind * 8 + register bit; IK_CP = kind * 8 + index of the register
// bit pair (a < b): b (b - 1) / 2 + a (up to 10 pairs, two opcode rows).
enum InterpKind : uint32_t {
    IK_H = 0,
    IK_RX0, IK_RX1,   // OP_RXS forms; c[0] = t
    IK_RY0, IK_RY1,   // OP_RYS forms; c[0] = t
    IK_U2,            // [[1, u], [v, w]]; table: u, v, w (re, im)
    IK_SWAP,          // exchange the halves where the conditions hold: X, CX, CXT
    IK_P,             // phase c on the set half where the thread condition holds
    IK_CP, IK_CP2,    // phase c where both register bits are set
    IK_MISC,          // IM_*
};
enum InterpMisc : uint32_t {
    IM_TPH = IK_MISC * 8,   // per-thread phase *= c where the thread condition holds
    IM_DIAG,                // register amplitude i *= table[2 i], table[2 i + 1] (re, im)
    IM_TAPPLY,              // multiply by the per-thread phase, reset it
    IM_TSG,                 // per-thread sign flips where the thread condition holds
    IM_TSAPPLY,             // negate where the per-thread sign is set, reset it
    IM_SIGN,                // negate where the register mask and the thread condition hold: Z, CZ
};

// arg: low half = thread-bit mask (all set: the condition holds; 0 = always),
// high half = register mask of IK_SWAP and IM_SIGN; for IK_U2 and IM_DIAG
// the table's distance in bytes from the phase's header.
template <typename Real> struct alignas(16) IOp {
    uint32_t code;
    uint32_t arg;
    alignas(2 * sizeof(Real) < 16 ? 8 : 16) Real c[2];
};
static_assert(sizeof(IOp<float>) == 16 && sizeof(IOp<double>) == 32, "IOp layout");

// Header of a register phase: swizzled offsets of the register and thread
// bits in the tile's buffer, then n_ops op records and the tables. A phase
// that is written with another layout than it is read (IPH_WRITE) has that
// one, in the form of the first 64 bytes, before its ops. A phase whose ops
// do not fit a window is continued (IPH_CONT) under a second header with the
// same layout and no transpose in between.
struct alignas(16) IPhase {
    uint16_t sreg[8];
    uint16_t sthr[MAX_TB];
    uint32_t n_ops;
    uint32_t bytes;      // all of it: the next header follows
    uint32_t flags;
    uint32_t ops_at;     // bytes from the header to the op records
};
static_assert(sizeof(IPhase) == 64, "IPhase layout");
constexpr uint32_t IPH_CONT = 1u, IPH_WRITE = 2u;

struct IWindow {
    uint32_t at;         // in 16-byte units from the stream's start
    uint32_t bytes;      // at most INTERP_WINDOW, a multiple of 16
    uint32_t phases;     // headers
    uint32_t pad;
};
constexpr uint32_t INTERP_WINDOW = 8192;

struct Program;
struct Lowered {
    std::vector<uint32_t> stream;
    std::vector<IWindow> windows;
    // the program's parts with phase_begin / n_phases = first window / windows
    std::vector<PartLaunch> parts;
};
void lower_program(const Program &prog, Lowered &out);

}  // namespace hisv
