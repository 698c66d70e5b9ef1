// Lowering of a part program to the interpreter's stream (see interp.hpp).
#include "interp.hpp"

#include <cstring>
#include <utility>

#include "planner.hpp"

namespace hisv {
namespace {

// The shared-memory swizzle of ops_core.cuh.
uint16_t swz_of(int p, bool wide) {
    if (!wide) return (uint16_t)(p < 4 ? (1u << p) : ((1u << p) | (1u << (p & 3))));
    return (uint16_t)(p < 3 ? (1u << p) : ((1u << p) | (1u << (p % 3))));
}

uint16_t swz_mask(uint16_t v, bool wide) {
    uint16_t o = 0;
    for (int p = 0; p < 16; p++)
        if ((v >> p) & 1) o = (uint16_t)(o ^ swz_of(p, wide));
    return o;
}

// A phase under construction: its op records and the tables (their place in
// the stream is known once the op count is).
template <typename Real> struct PhaseOut {
    std::vector<IOp<Real>> ops;
    std::vector<uint32_t> table_at;   // per op: index into table + 1, or 0
    std::vector<Real> table;

    // two headers: a phase may have a write layout
    size_t bytes() const { return 2 * sizeof(IPhase) + ops.size() * sizeof(IOp<Real>) + table.size() * sizeof(Real); }
    void emit(uint32_t code, uint32_t arg, double c0 = 0.0, double c1 = 0.0) {
        IOp<Real> o{};
        o.code = code;
        o.arg = arg;
        o.c[0] = (Real)c0;
        o.c[1] = (Real)c1;
        ops.push_back(o);
        table_at.push_back(0);
    }
    void emit_table(uint32_t code, const double *v, int count) {
        emit(code, 0);
        table_at.back() = (uint32_t)table.size() + 1;
        for (int i = 0; i < count; i++) table.push_back((Real)v[i]);
        while ((table.size() * sizeof(Real)) % 16) table.push_back((Real)0);
    }
};

template <typename Real> void lower(const Program &prog, Lowered &out) {
    const bool wide = sizeof(Real) == 8;
    const int R = prog.R, NR = 1 << R, TB = prog.t - R;
    // room a single op may need: its record and a full table
    const size_t most = sizeof(IOp<Real>) + 2 * NR * sizeof(Real);
    out = Lowered();
    for (PartLaunch L : prog.parts) {
        const uint32_t w0 = (uint32_t)out.windows.size();
        for (uint32_t p = 0; p < L.n_phases; p++) {
            const Phase &ph = prog.phases[L.phase_begin + p];
            PhaseOut<Real> q;
            bool cont = false;
            auto close = [&]() {   // append q to the stream
                IPhase h{};
                auto layout = [&](const Layout &l, IPhase &d) {
                    for (int b = 0; b < R; b++) d.sreg[b] = swz_mask(l.reg[b], wide);
                    for (int j = 0; j < TB; j++) d.sthr[j] = swz_mask(l.thr[j], wide);
                };
                layout(ph.rd, h);
                // the last phase's write layout is the part's store layout
                const bool write = !cont && p + 1 < L.n_phases && std::memcmp(&ph.rd, &ph.wr, sizeof(Layout)) != 0;
                h.n_ops = (uint32_t)q.ops.size();
                h.ops_at = (uint32_t)(write ? 2 * sizeof(IPhase) : sizeof(IPhase));
                const uint32_t t0 = h.ops_at + (uint32_t)(q.ops.size() * sizeof(IOp<Real>));
                h.bytes = t0 + (uint32_t)(q.table.size() * sizeof(Real));
                h.flags = (cont ? IPH_CONT : 0u) | (write ? IPH_WRITE : 0u);
                for (size_t i = 0; i < q.ops.size(); i++)
                    if (q.table_at[i]) q.ops[i].arg = t0 + (q.table_at[i] - 1) * (uint32_t)sizeof(Real);
                if (out.windows.size() == w0 || out.windows.back().bytes + h.bytes > INTERP_WINDOW)
                    out.windows.push_back({(uint32_t)(out.stream.size() / 4), 0, 0, 0});
                out.windows.back().bytes += h.bytes;
                out.windows.back().phases++;
                const size_t at = out.stream.size();
                out.stream.resize(at + h.bytes / 4);
                char *d = reinterpret_cast<char *>(out.stream.data() + at);
                std::memcpy(d, &h, sizeof(h));
                if (write) {
                    IPhase wr{};
                    layout(ph.wr, wr);
                    std::memcpy(d + sizeof(h), &wr, sizeof(wr));
                }
                if (!q.ops.empty()) std::memcpy(d + h.ops_at, q.ops.data(), q.ops.size() * sizeof(IOp<Real>));
                if (!q.table.empty()) std::memcpy(d + t0, q.table.data(), q.table.size() * sizeof(Real));
                q = PhaseOut<Real>();
                cont = true;
            };
            auto kind = [](uint32_t k, int bit) { return k * 8 + (uint32_t)bit; };
            for (uint32_t k = 0; k < ph.op_count; k++) {
                if (q.bytes() + 2 * most > INTERP_WINDOW) close();
                const Op &op = prog.ops[ph.op_begin + k];
                const double *c = prog.coefs.data() + op.coef;
                const uint32_t tm = 1u << op.tb;
                switch (op.kind) {
                case OP_H: q.emit(kind(IK_H, op.a), 0); break;
                case OP_RXS: q.emit(kind(op.b ? IK_RX1 : IK_RX0, op.a), 0, c[0]); break;
                case OP_RYS: q.emit(kind(op.b ? IK_RY1 : IK_RY0, op.a), 0, c[0]); break;
                case OP_U2S:
                    if (op.b) {   // [[u, 1], [v, w]] (x, y) = [[1, u], [w, v]] (y, x)
                        const double m[6] = {c[0], c[1], c[4], c[5], c[2], c[3]};
                        q.emit(kind(IK_SWAP, op.a), 0);
                        q.emit_table(kind(IK_U2, op.a), m, 6);
                    } else {
                        q.emit_table(kind(IK_U2, op.a), c, 6);
                    }
                    break;
                case OP_X: q.emit(kind(IK_SWAP, op.a), 0); break;
                case OP_CX: q.emit(kind(IK_SWAP, op.b), (1u << op.a) << 16); break;
                case OP_CXT: q.emit(kind(IK_SWAP, op.b), tm); break;
                case OP_Y: {   // X, then -i on the clear half and i on the set half
                    std::vector<double> d(2 * NR, 0.0);
                    for (int i = 0; i < NR; i++) d[2 * i + 1] = (i >> op.a) & 1 ? 1.0 : -1.0;
                    q.emit(kind(IK_SWAP, op.a), 0);
                    q.emit_table(IM_DIAG, d.data(), 2 * NR);
                } break;
                case OP_P: q.emit(kind(IK_P, op.a), 0, c[0], c[1]); break;
                case OP_Z: q.emit(IM_SIGN, (1u << op.a) << 16); break;
                case OP_CPT: q.emit(kind(IK_P, op.a), tm, c[0], c[1]); break;
                case OP_CZT: q.emit(IM_SIGN, ((1u << op.a) << 16) | tm); break;
                case OP_CP: {
                    const int lo = op.a < op.b ? op.a : op.b, hi = op.a < op.b ? op.b : op.a;
                    q.emit(IK_CP * 8 + (uint32_t)(hi * (hi - 1) / 2 + lo), 0, c[0], c[1]);
                } break;
                case OP_CZ: q.emit(IM_SIGN, ((1u << op.a) | (1u << op.b)) << 16); break;
                case OP_TD: q.emit(IM_TPH, tm, c[2], c[3]); break;   // the planner's d0 is 1
                case OP_TP2: q.emit(IM_TPH, tm | (1u << op.b), c[0], c[1]); break;
                case OP_DIAG: q.emit_table(IM_DIAG, c, 2 * NR); break;
                case OP_TAPPLY: q.emit(IM_TAPPLY, 0); break;
                case OP_TSG: q.emit(IM_TSG, tm | (1u << op.b)); break;
                case OP_TSAPPLY: q.emit(IM_TSAPPLY, 0); break;
                default: break;
                }
            }
            close();
        }
        L.phase_begin = w0;
        L.n_phases = (uint32_t)out.windows.size() - w0;
        out.parts.push_back(L);
    }
}

}  // namespace

void lower_program(const Program &prog, Lowered &out) {
    if (prog.fp64) lower<double>(prog, out);
    else lower<float>(prog, out);
}

}  // namespace hisv
