// Lowering of a part program to the interpreter's op stream (see interp.hpp).
#include "interp.hpp"

#include "planner.hpp"

namespace hisv {

// The shared-memory swizzle of ops_core.cuh.
static uint16_t swz_of(int p, bool wide) {
    if (!wide) return (uint16_t)(p < 4 ? (1u << p) : ((1u << p) | (1u << (p & 3))));
    return (uint16_t)(p < 3 ? (1u << p) : ((1u << p) | (1u << (p % 3))));
}

template <typename Real> void lower_program(const Program &prog, Lowered<Real> &out) {
    const bool wide = sizeof(Real) == 8;
    const int R = prog.R, NR = 1 << R, TB = prog.t - R;
    out = Lowered<Real>();
    out.phases.reserve(prog.phases.size());
    for (const Phase &ph : prog.phases) {
        IPhase ip{};
        for (int b = 0; b < R; b++) ip.sreg[b] = swz_of(ph.reg[b], wide);
        for (int j = 0; j < TB; j++) ip.sthr[j] = swz_of(ph.thr[j], wide);
        ip.op_begin = (uint32_t)out.ops.size();
        auto emit = [&](uint32_t code, uint32_t arg, double c0 = 0.0, double c1 = 0.0) {
            IOp<Real> o{};
            o.code = code;
            o.arg = arg;
            o.c[0] = (Real)c0;
            o.c[1] = (Real)c1;
            out.ops.push_back(o);
        };
        auto table = [&](const double *v, int count) {
            const uint32_t at = (uint32_t)out.table.size();
            for (int i = 0; i < count; i++) out.table.push_back((Real)v[i]);
            while (out.table.size() % 4) out.table.push_back((Real)0);
            return at;
        };
        auto kind = [](uint32_t k, int bit) { return k * 8 + (uint32_t)bit; };
        auto pair = [](int a, int b) {
            if (a > b) std::swap(a, b);
            return IK_CP * 8 + (uint32_t)(b * (b - 1) / 2 + a);
        };
        for (uint32_t k = 0; k < ph.op_count; k++) {
            const Op &op = prog.ops[ph.op_begin + k];
            const double *c = prog.coefs.data() + op.coef;
            const uint32_t tm = 1u << op.tb;
            switch (op.kind) {
            case OP_H: emit(kind(IK_H, op.a), 0); break;
            case OP_RXS: emit(kind(op.b ? IK_RX1 : IK_RX0, op.a), 0, c[0]); break;
            case OP_RYS: emit(kind(op.b ? IK_RY1 : IK_RY0, op.a), 0, c[0]); break;
            case OP_U2S:
                if (op.b) {   // [[u, 1], [v, w]] (x, y) = [[1, u], [w, v]] (y, x)
                    const double m[6] = {c[0], c[1], c[4], c[5], c[2], c[3]};
                    emit(kind(IK_SWAP, op.a), 0);
                    emit(kind(IK_U2, op.a), table(m, 6));
                } else {
                    emit(kind(IK_U2, op.a), table(c, 6));
                }
                break;
            case OP_X: emit(kind(IK_SWAP, op.a), 0); break;
            case OP_CX: emit(kind(IK_SWAP, op.b), (1u << op.a) << 16); break;
            case OP_CXT: emit(kind(IK_SWAP, op.b), tm); break;
            case OP_Y: {   // X, then -i on the clear half and i on the set half
                std::vector<double> d(2 * NR, 0.0);
                for (int i = 0; i < NR; i++) d[2 * i + 1] = (i >> op.a) & 1 ? 1.0 : -1.0;
                emit(kind(IK_SWAP, op.a), 0);
                emit(IM_DIAG, table(d.data(), 2 * NR));
            } break;
            case OP_P: emit(kind(IK_P, op.a), 0, c[0], c[1]); break;
            case OP_Z: emit(IM_SIGN, (1u << op.a) << 16); break;
            case OP_CPT: emit(kind(IK_P, op.a), tm, c[0], c[1]); break;
            case OP_CZT: emit(IM_SIGN, ((1u << op.a) << 16) | tm); break;
            case OP_CP: emit(pair(op.a, op.b), 0, c[0], c[1]); break;
            case OP_CZ: emit(IM_SIGN, ((1u << op.a) | (1u << op.b)) << 16); break;
            case OP_TD: emit(IM_TPH, tm, c[2], c[3]); break;   // the planner's d0 is 1
            case OP_TP2: emit(IM_TPH, tm | (1u << op.b), c[0], c[1]); break;
            case OP_DIAG: emit(IM_DIAG, table(c, 2 * NR)); break;
            case OP_TAPPLY: emit(IM_TAPPLY, 0); break;
            case OP_TSG: emit(IM_TSG, tm | (1u << op.b)); break;
            case OP_TSAPPLY: emit(IM_TSAPPLY, 0); break;
            default: break;
            }
        }
        ip.op_count = (uint32_t)out.ops.size() - ip.op_begin;
        out.phases.push_back(ip);
    }
}

template void lower_program<float>(const Program &, Lowered<float> &);
template void lower_program<double>(const Program &, Lowered<double> &);

}  // namespace hisv
