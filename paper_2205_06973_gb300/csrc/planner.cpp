// Part planner (host): for each part of the partition, fix its tile, split
// its gates into register phases and emit the kernel's op stream.
//
//  * Tile: the part's qubits S (|S| <= k) padded with the lowest qubits not
//    in S up to t (Sec. IV-B, multi-level partitioning: a part smaller than
//    the limit takes extra qubits for spatial locality). Slot p of the tile
//    holds the p-th smallest tile qubit; the n - t others are the outer
//    qubits of Algorithm 1, one CTA per binary assignment of them.
//  * Phases: a second partitioning level inside the part, with limit R on
//    the qubits that need register residency (targets of non-diagonal
//    gates). Gates are taken greedily along the part's gate order; a gate
//    that does not fit blocks its qubits for the rest of the phase, so every
//    qubit keeps its gate order (the schedule rule of Sec. IV-A).
//    Diagonal gates and CX controls need no residency: on a thread bit they
//    become per-thread conditions or a per-thread phase (and in programs for
//    the specialised kernels the same on a qubit outside the tile, whose bit
//    is the tile index's: outer_diag).
//  * SWAP gates cost nothing: they exchange the slots of their two qubits
//    for the rest of the part, and the store uses the final slot map.
#include "planner.hpp"

#include <algorithm>
#include <array>
#include <cstdint>
#include <cmath>
#include <cstring>

#include "../../include/hisvsim.h"

namespace hisv {

static inline int popc(uint64_t x) { return __builtin_popcountll(x); }

bool gate_is_two_qubit(int kind) {
    return kind == SV_GATE_CX || kind == SV_GATE_CZ || kind == SV_GATE_CP || kind == SV_GATE_SWAP;
}

void gate_matrix_1q(int kind, double th, double m[8]) {
    for (int i = 0; i < 8; i++) m[i] = 0.0;
    const double c = std::cos(th / 2), s = std::sin(th / 2), r = std::sqrt(0.5);
    switch (kind) {
    case SV_GATE_H: m[0] = r; m[2] = r; m[4] = r; m[6] = -r; break;
    case SV_GATE_X: m[2] = 1; m[4] = 1; break;
    case SV_GATE_Y: m[3] = -1; m[5] = 1; break;          // [[0,-i],[i,0]]
    case SV_GATE_Z: m[0] = 1; m[6] = -1; break;
    case SV_GATE_S: m[0] = 1; m[7] = 1; break;
    case SV_GATE_T: m[0] = 1; m[6] = r; m[7] = r; break;
    case SV_GATE_RX: m[0] = c; m[3] = -s; m[5] = -s; m[6] = c; break;
    case SV_GATE_RY: m[0] = c; m[2] = -s; m[4] = s; m[6] = c; break;
    case SV_GATE_RZ: m[0] = c; m[1] = -s; m[6] = c; m[7] = s; break;
    case SV_GATE_P: m[0] = 1; m[6] = std::cos(th); m[7] = std::sin(th); break;
    default: break;
    }
}

void gate_matrix_2q(int kind, double th, double m[32]) {
    for (int i = 0; i < 32; i++) m[i] = 0.0;
    auto set = [&](int r, int c, double re, double im) { m[2 * (4 * r + c)] = re; m[2 * (4 * r + c) + 1] = im; };
    switch (kind) {
    case SV_GATE_CX:   // l = b_c + 2 b_t: l=1 <-> l=3
        set(0, 0, 1, 0); set(2, 2, 1, 0); set(1, 3, 1, 0); set(3, 1, 1, 0); break;
    case SV_GATE_CZ:
        set(0, 0, 1, 0); set(1, 1, 1, 0); set(2, 2, 1, 0); set(3, 3, -1, 0); break;
    case SV_GATE_CP:
        set(0, 0, 1, 0); set(1, 1, 1, 0); set(2, 2, 1, 0); set(3, 3, std::cos(th), std::sin(th)); break;
    case SV_GATE_SWAP:
        set(0, 0, 1, 0); set(1, 2, 1, 0); set(2, 1, 1, 0); set(3, 3, 1, 0); break;
    default: break;
    }
}

// slots that must be register bits for this gate
static uint32_t needed_slots(const GateRef &g, const int *slot_of) {
    switch (g.kind) {
    case SV_GATE_H: case SV_GATE_X: case SV_GATE_Y: case SV_GATE_RX: case SV_GATE_RY:
        return 1u << slot_of[g.q[0]];
    case SV_GATE_CX:
        return 1u << slot_of[g.q[1]];
    default:
        return 0u;
    }
}

static bool is_diagonal(int kind) {
    switch (kind) {
    case SV_GATE_Z: case SV_GATE_S: case SV_GATE_T: case SV_GATE_RZ: case SV_GATE_P: case SV_GATE_CZ: case SV_GATE_CP:
        return true;
    default:
        return false;
    }
}

// qubits that the gate acts on non-diagonally (not as a phase or a control)
static uint64_t acts_nondiag(const GateRef &g) {
    if (is_diagonal(g.kind)) return 0;
    if (g.kind == SV_GATE_SWAP) return (1ull << g.q[0]) | (1ull << g.q[1]);
    return 1ull << (g.kind == SV_GATE_CX ? g.q[1] : g.q[0]);
}

// A one-qubit phase on a qubit outside the tile would multiply every
// amplitude; inside, it joins a merged diagonal.
uint64_t tile_need(const GateRef &g) {
    return is_diagonal(g.kind) && g.arity == 1 ? 1ull << g.q[0] : acts_nondiag(g);
}

// QFT, beam k = 12: the part with the 12 highest targets moved runs of 16
// bytes (28 qubits: 3.3 ms against 0.64), as the last part of SWAPs did, and
// their halves move whole lines; the parts of phases alone cost a pass each
// (the 30-qubit circuit's 12 passes took 55.5 ms, at 2.6 a pass of whole
// lines 31). us with the plan's
// parts / with these: 20 qubits 26 / 19, 24 qubits 435 / 288, 26 qubits 1910
// / 1208, 28 qubits 11268 / 6870, 30 qubits 55532 / 25103; k = 9 at 28 qubits
// 14271 / 7571. Layered circuits, k = 12 at 28 qubits 17659 / 17333.
uint32_t refine_parts(const std::vector<GateRef> &gates, int n, const std::vector<uint32_t> &pog, uint32_t n_parts,
                      bool fp64, int t, std::vector<uint32_t> &out) {
    struct Group {
        std::vector<int> gates;
        uint64_t need = 0, all = 0;   // qubits of the tile, qubits
    };
    auto add = [&](Group &g, int i) {
        g.gates.push_back(i);
        g.need |= tile_need(gates[i]);
        for (int j = 0; j < gates[i].arity; j++) g.all |= 1ull << gates[i].q[j];
    };
    // time of a pass, in passes at full rate, by the bytes of its tile's runs
    // (the lowest qubits in the tile): 8 and 16 (3.3 against 0.64 ms at 28
    // qubits), 32 (0.54 of HBM), 64 (0.91), 128 and more
    auto cost = [&](uint64_t need) {
        int spare = std::min(n, t) - popc(need), run = fp64 ? 1 : 0;
        for (int q = 0; q < n && (((need >> q) & 1) || spare-- > 0); q++) run++;
        return run >= 4 ? 1.0 : run == 3 ? 1.1 : run == 2 ? 1.8 : 5.0;
    };
    std::vector<Group> parts(n_parts), cut;
    for (size_t i = 0; i < gates.size(); i++) add(parts[pog[i]], (int)i);
    for (Group &p : parts) {
        if (p.gates.empty()) continue;
        const double whole = cost(p.need);
        double best = whole;
        size_t at = 0;
        std::vector<uint64_t> tail(p.gates.size() + 1, 0);
        for (size_t i = p.gates.size(); i-- > 0;) tail[i] = tail[i + 1] | tile_need(gates[p.gates[i]]);
        uint64_t head = 0;
        for (size_t i = 1; whole > 2.0 && i < p.gates.size(); i++) {   // of equal cuts the most even
            head |= tile_need(gates[p.gates[i - 1]]);
            const double c = cost(head) + cost(tail[i]);
            const size_t half = p.gates.size() / 2;
            auto far = [&](size_t x) { return x > half ? x - half : half - x; };
            if (c < best || (at && c == best && far(i) < far(at))) {
                best = c;
                at = i;
            }
        }
        if (at == 0) {
            cut.push_back(std::move(p));
            continue;
        }
        Group a, b;
        for (size_t i = 0; i < p.gates.size(); i++) add(i < at ? a : b, p.gates[i]);
        cut.push_back(std::move(a));
        cut.push_back(std::move(b));
    }
    // joined parts stay within 192 gates (30-qubit QFT: 9 passes, 25.1 ms;
    // with 128 gates 11 passes, 4 ms more; with 320 still 9), for the size of their
    // code, and within 32 slots
    std::vector<Group> done;
    auto fits = [&](const Group &a, const Group &b) {
        return a.gates.size() + b.gates.size() <= 192 && popc(a.need | b.need) <= t &&
               (n <= 32 || t + popc(a.all | b.all) <= 32) &&
               cost(a.need | b.need) <= std::max(cost(a.need), cost(b.need));
    };
    auto phases_only = [&](const Group &g) {
        for (int i : g.gates)
            if (!is_diagonal(gates[i].kind) || gates[i].arity == 1) return false;
        return true;
    };
    auto join = [&](Group &a, const Group &b) {
        for (int i : b.gates) add(a, i);
    };
    for (size_t i = 0; i < cut.size(); i++) {
        Group &g = cut[i];
        const bool prev = !done.empty() && fits(done.back(), g), next = i + 1 < cut.size() && fits(g, cut[i + 1]);
        if (phases_only(g) && prev && (!next || done.back().gates.size() <= cut[i + 1].gates.size()))
            join(done.back(), g);
        else if (phases_only(g) && next) {
            join(g, cut[i + 1]);
            cut[i + 1] = std::move(g);
        } else {
            done.push_back(std::move(g));
        }
    }
    out.assign(gates.size(), 0);
    for (size_t p = 0; p < done.size(); p++)
        for (int i : done[p].gates) out[i] = (uint32_t)p;
    return (uint32_t)done.size();
}

// Thread-bit order of a phase: lane bits first. The first lanes cover
// distinct slot residues (mod 4 for 8-byte, mod 3 for 16-byte amplitudes) so
// the swizzled shared-memory accesses are conflict free; otherwise slots
// follow the preference key (lowest global qubit first for the phases that
// load or store, for coalescing).
static std::vector<int> order_thread_slots(std::vector<int> cand, const std::vector<int> &key, bool fp64) {
    std::stable_sort(cand.begin(), cand.end(), [&](int a, int b) { return key[a] < key[b]; });
    const int mod = fp64 ? 3 : 4;
    std::vector<int> lanes, rest;
    std::vector<char> used(cand.size(), 0);
    uint32_t covered = 0;
    for (size_t i = 0; i < cand.size() && (int)lanes.size() < mod; i++) {
        int r = cand[i] % mod;
        if (!((covered >> r) & 1)) {
            covered |= 1u << r;
            lanes.push_back(cand[i]);
            used[i] = 1;
        }
    }
    for (size_t i = 0; i < cand.size(); i++)
        if (!used[i]) rest.push_back(cand[i]);
    // fill to a full warp of lanes, then warp bits, in key order
    std::vector<int> out = lanes;
    for (int s : rest) out.push_back(s);
    return out;
}

void fused_unitary(const std::vector<GateRef> &gates, const std::vector<int> &ids, const int *qs, int k,
                   std::vector<double> &U) {
    // U <- G U for each gate G in order, on the rows of the row-major 2^k x 2^k
    // matrix (the same update on every column): pairs of rows for a one-qubit
    // gate, quads for a two-qubit one
    const int D = 1 << k;
    U.assign((size_t)2 * D * D, 0.0);
    for (int i = 0; i < D; i++) U[2 * (D * i + i)] = 1.0;
    double *u = U.data();
    auto row = [&](int r) { return u + (size_t)2 * D * r; };
    for (int g : ids) {
        const GateRef &gr = gates[g];
        int loc[2] = {0, 0};
        for (int a = 0; a < gr.arity; a++)
            for (int j = 0; j < k; j++)
                if (qs[j] == gr.q[a]) loc[a] = j;
        if (gr.arity == 1) {
            double m[8];
            gate_matrix_1q(gr.kind, gr.theta, m);
            const int s = 1 << loc[0];
            for (int x = 0; x < D; x++) {
                if (x & s) continue;
                double *a = row(x), *b = row(x + s);
                for (int c = 0; c < D; c++) {
                    const double ar = a[2 * c], ai = a[2 * c + 1], br = b[2 * c], bi = b[2 * c + 1];
                    a[2 * c] = m[0] * ar - m[1] * ai + m[2] * br - m[3] * bi;
                    a[2 * c + 1] = m[0] * ai + m[1] * ar + m[2] * bi + m[3] * br;
                    b[2 * c] = m[4] * ar - m[5] * ai + m[6] * br - m[7] * bi;
                    b[2 * c + 1] = m[4] * ai + m[5] * ar + m[6] * bi + m[7] * br;
                }
            }
            continue;
        }
        const int s0 = 1 << loc[0], s1 = 1 << loc[1];   // control, target
        switch (gr.kind) {
        case SV_GATE_CX:    // rows with the control set swap their target halves
            for (int x = 0; x < D; x++)
                if ((x & s0) && !(x & s1)) std::swap_ranges(row(x), row(x) + 2 * D, row(x + s1));
            break;
        case SV_GATE_SWAP:
            for (int x = 0; x < D; x++)
                if ((x & s0) && !(x & s1)) std::swap_ranges(row(x), row(x) + 2 * D, row(x - s0 + s1));
            break;
        case SV_GATE_CZ: case SV_GATE_CP: {
            const double dr = gr.kind == SV_GATE_CZ ? -1.0 : std::cos(gr.theta);
            const double di = gr.kind == SV_GATE_CZ ? 0.0 : std::sin(gr.theta);
            for (int x = 0; x < D; x++)
                if ((x & s0) && (x & s1)) {
                    double *a = row(x);
                    for (int c = 0; c < D; c++) {
                        const double ar = a[2 * c], ai = a[2 * c + 1];
                        a[2 * c] = ar * dr - ai * di;
                        a[2 * c + 1] = ar * di + ai * dr;
                    }
                }
        } break;
        default: {   // any other two-qubit gate: its 4x4 matrix on quads of rows
            double m[32];
            gate_matrix_2q(gr.kind, gr.theta, m);
            std::vector<double> t(8);
            for (int x = 0; x < D; x++) {
                if ((x & s0) || (x & s1)) continue;
                double *rw[4] = {row(x), row(x + s0), row(x + s1), row(x + s0 + s1)};
                for (int c = 0; c < D; c++) {
                    for (int r = 0; r < 4; r++) {
                        double re = 0, im = 0;
                        for (int cc = 0; cc < 4; cc++) {
                            const double mr = m[2 * (4 * r + cc)], mi = m[2 * (4 * r + cc) + 1];
                            re += mr * rw[cc][2 * c] - mi * rw[cc][2 * c + 1];
                            im += mr * rw[cc][2 * c + 1] + mi * rw[cc][2 * c];
                        }
                        t[2 * r] = re;
                        t[2 * r + 1] = im;
                    }
                    for (int r = 0; r < 4; r++) {
                        rw[r][2 * c] = t[2 * r];
                        rw[r][2 * c + 1] = t[2 * r + 1];
                    }
                }
            }
        }
        }
    }
}

// Bank bits of the pair kernel's shared buffer: slot p < 4 keeps its bit;
// slot p >= 4 also flips the 4-bit bank-pair value v_p. A half-warp's 16
// lanes run over the slots of the lowest 4 column qubits of layout 1 (when
// writing) or layout 2 (when reading); the v_p are picked (fixed-seed search)
// so that both sets of 4 slots map to independent bank vectors, i.e. 16
// distinct bank pairs. Falls back to v_p = bit (p mod 4) if none is found.
static void pair_swizzle(DensePairLaunch &D) {
    const int NS = DENSE_K + DENSE_COLS;
    auto indep = [](const uint32_t *w) {
        uint32_t span = 1u;   // bit mask over the 16 bank values reachable
        for (int i = 0; i < 4; i++) {
            if ((span >> w[i]) & 1u) return false;
            uint32_t ns = span;
            for (uint32_t x = 0; x < 16; x++)
                if ((span >> x) & 1u) ns |= 1u << (x ^ w[i]);
            span = ns;
        }
        return true;
    };
    uint32_t v[DENSE_K + DENSE_COLS];
    uint64_t st = 0x9E3779B97F4A7C15ull;
    bool found = false;
    for (int trial = 0; trial < 4096 && !found; trial++) {
        for (int p = 0; p < NS; p++) {
            if (p < 4) v[p] = 1u << p;
            else if (trial == 0) v[p] = 1u << (p & 3);
            else {
                st = st * 6364136223846793005ull + 1442695040888963407ull;
                v[p] = 1u + (uint32_t)((st >> 33) % 15u);
            }
        }
        uint32_t w1[4], w2[4];
        for (int i = 0; i < 4; i++) {
            w1[i] = v[D.s_c1[i]];
            w2[i] = v[D.s_c2[i]];
        }
        found = indep(w1) && indep(w2);
    }
    if (!found)
        for (int p = 4; p < NS; p++) v[p] = 1u << (p & 3);
    for (int p = 0; p < NS; p++) D.xsw[p] = (uint16_t)(p < 4 ? (1u << p) : ((1u << p) | v[p]));
}

// Modulus of the factor that the planner gathered for an op (the op alone
// grows a state by up to its inverse): the first row of a scaled matrix has
// the norm of 1 and its smaller entry.
static double factor_of(const Op &op, const std::vector<double> &coefs) {
    const double *c = coefs.data() + op.coef;
    switch (op.kind) {
    case OP_H: return std::sqrt(0.5);
    case OP_RXS: case OP_RYS: return 1.0 / std::hypot(1.0, c[0]);
    case OP_U2S: return 1.0 / std::sqrt(1.0 + c[0] * c[0] + c[1] * c[1]);
    default: return 1.0;
    }
}

// Rank of a warp's 32 lanes in the shared-memory banks (bank groups of one
// amplitude: 4 index bits for 8-byte amplitudes, 3 for 16-byte ones).
static int bank_rank(const Layout &l, bool wide) {
    const int m = wide ? 3 : 4;
    uint32_t rows[5];
    for (int j = 0; j < 5; j++) {
        uint32_t v = 0;
        for (int p = 0; p < 16; p++)
            if ((l.thr[j] >> p) & 1) v ^= p < m ? (1u << p) : (1u << (p % m));   // the swizzle's low bits
        rows[j] = v;
    }
    int rank = 0;
    for (int bit = 0; bit < m; bit++) {
        int piv = -1;
        for (int j = rank; j < 5 && piv < 0; j++)
            if ((rows[j] >> bit) & 1) piv = j;
        if (piv < 0) continue;
        std::swap(rows[rank], rows[piv]);
        for (int j = 0; j < 5; j++)
            if (j != rank && ((rows[j] >> bit) & 1)) rows[j] ^= rows[rank];
        rank++;
    }
    return rank;
}

bool compile_program(const std::vector<GateRef> &gates, int n, const std::vector<uint32_t> &pog,
                     uint32_t n_parts, bool fp64, int t_cfg, int R, int dense_mode, Program &prog,
                     std::string &err, const std::vector<uint32_t> *inner, bool outer_diag, bool refined) {
    prog = Program();
    prog.fp64 = fp64;
    prog.R = R;
    const int t = std::min(n, t_cfg);
    prog.t = t;
    if (t - R > MAX_TB || R < 1 || R > MAX_R || t < R + 5) {
        err = "tile configuration out of range";
        return false;
    }
    std::vector<std::vector<int>> members(n_parts);
    for (size_t g = 0; g < gates.size(); g++) {
        if (pog[g] >= n_parts) {
            err = "part id out of range";
            return false;
        }
        members[pog[g]].push_back((int)g);
    }
    std::vector<uint64_t> gmask(gates.size());
    for (size_t g = 0; g < gates.size(); g++) {
        uint64_t m = 0;
        for (int j = 0; j < gates[g].arity; j++) m |= 1ull << gates[g].q[j];
        gmask[g] = m;
    }
    const uint64_t all = (n >= 64) ? ~0ull : ((1ull << n) - 1);
    for (uint32_t pi = 0; pi < n_parts; pi++) {
        const std::vector<int> &gl = members[pi];
        if (gl.empty()) continue;
        uint64_t S = 0;
        for (int g : gl) S |= gmask[g];
        if ((dense_mode & 2) && !fp64 && popc(S) <= DENSE_K && n >= DENSE_K + DENSE_COLS && pi + 1 < n_parts &&
            !members[pi + 1].empty()) {
            // two consecutive dense parts in one pass (multi-level
            // partitioning, Sec. IV-B: a 13-qubit tile as the first level,
            // two 6-qubit products as the second); each part is padded to 6
            // with the other's qubits first, and the tile adds the lowest
            // remaining qubits; paired only if the tile holds qubits 0 and 1
            // (runs of 4 consecutive amplitudes: whole 32-byte sectors)
            uint64_t S2 = 0;
            for (int g : members[pi + 1]) S2 |= gmask[g];
            if (popc(S2) <= DENSE_K) {
                auto pad = [&](uint64_t P, uint64_t pref) {
                    for (int q = n - 1; q >= 0 && popc(P) < DENSE_K; q--)
                        if ((pref >> q) & 1) P |= 1ull << q;
                    for (int q = n - 1; q >= 0 && popc(P) < DENSE_K; q--) P |= 1ull << q;
                    return P;
                };
                const uint64_t P1 = pad(S, S2 & ~S), P2 = pad(S2, S & ~S2);
                uint64_t T = P1 | P2;
                for (int q = 0; q < n && popc(T) < DENSE_K + DENSE_COLS; q++) T |= 1ull << q;
                if ((T & 3ull) == 3ull && popc(T) == DENSE_K + DENSE_COLS) {
                    DensePairLaunch D;
                    std::memset(&D, 0, sizeof(D));
                    D.n = n;
                    D.outer_mask = all & ~T;
                    int f = 0;
                    while (f < 4 && ((T >> f) & 1)) f++;
                    D.prefetch = (uint8_t)f;
                    int slot = 0, j1 = 0, c1 = 0, j2 = 0, c2 = 0, qs1[DENSE_K], qs2[DENSE_K];
                    for (int q = 0; q < n; q++) {
                        if (!((T >> q) & 1)) continue;
                        if ((P1 >> q) & 1) { qs1[j1] = q; D.s_q1[j1] = (uint8_t)slot; D.q1[j1++] = (uint8_t)q; }
                        else { D.s_c1[c1] = (uint8_t)slot; D.c1[c1++] = (uint8_t)q; }
                        if ((P2 >> q) & 1) { qs2[j2] = q; D.s_q2[j2] = (uint8_t)slot; D.q2[j2++] = (uint8_t)q; }
                        else { D.s_c2[c2] = (uint8_t)slot; D.c2[c2++] = (uint8_t)q; }
                        slot++;
                    }
                    pair_swizzle(D);
                    std::vector<double> U;
                    std::vector<uint8_t> img;
                    fused_unitary(gates, gl, qs1, DENSE_K, U);
                    dense_a_image(U.data(), img);
                    prog.pair_img.insert(prog.pair_img.end(), img.begin(), img.end());
                    fused_unitary(gates, members[pi + 1], qs2, DENSE_K, U);
                    dense_a_image(U.data(), img);
                    prog.pair_img.insert(prog.pair_img.end(), img.begin(), img.end());
                    prog.kind.push_back(2);
                    prog.index.push_back((uint32_t)prog.pairs.size());
                    prog.pairs.push_back(D);
                    prog.pair_tiles.push_back(1ull << (n - DENSE_K - DENSE_COLS));
                    pi++;   // the second part is done
                    continue;
                }
            }
        }
        if ((dense_mode & 1) && !fp64 && popc(S) <= DENSE_K && n >= DENSE_K + DENSE_COLS) {
            // dense part: the part's qubits padded to 6 with the highest others
            // (the unitary is the identity on them), columns on the lowest 7
            // remaining qubits, so that the 32 lanes of a warp (columns) stay
            // consecutive amplitudes unless the part itself holds low qubits
            uint64_t P = S, C = 0;
            for (int q = n - 1; q >= 0 && popc(P) < DENSE_K; q--) P |= 1ull << q;
            for (int q = 0; q < n && popc(C) < DENSE_COLS; q++)
                if (!((P >> q) & 1)) C |= 1ull << q;
            DenseLaunch D;
            std::memset(&D, 0, sizeof(D));
            D.n = n;
            D.outer_mask = all & ~(P | C);
            int qs[DENSE_K], jp = 0, jc = 0, js = 0;
            for (int q = 0; q < n; q++) {
                if ((P >> q) & 1) {
                    qs[jp] = q;
                    D.part_q[jp++] = (uint8_t)q;
                    D.slot_part |= (uint16_t)(1u << js);
                    D.slot_q[js++] = (uint8_t)q;
                } else if ((C >> q) & 1) {
                    D.col_q[jc++] = (uint8_t)q;
                    D.slot_q[js++] = (uint8_t)q;
                }
            }
            std::vector<double> U;
            fused_unitary(gates, gl, qs, DENSE_K, U);
            std::vector<uint8_t> img;
            dense_a_image(U.data(), img);
            D.reverse = prog.kind.size() & 1;
            prog.kind.push_back(1);
            prog.index.push_back((uint32_t)prog.dense.size());
            prog.dense.push_back(D);
            prog.dense_tiles.push_back(1ull << (n - DENSE_K - DENSE_COLS));
            prog.a_img.insert(prog.a_img.end(), img.begin(), img.end());
            continue;
        }
        if (popc(S) > t && !refined) {
            err = "part " + std::to_string(pi) + " has " + std::to_string(popc(S)) + " qubits > tile " + std::to_string(t);
            return false;
        }
        // the tile: with outer_diag only the qubits of tile_need must be in it,
        // and more low qubits (longer contiguous runs) take the places of the
        // others
        uint64_t Tm = S;
        if (outer_diag) {
            Tm = 0;
            for (int g : gl) Tm |= tile_need(gates[g]);
        }
        for (int q = 0; q < n && popc(Tm) < t; q++) Tm |= 1ull << q;
        int slot_of[64], q_at[64];
        for (int q = 0, p = 0, o = t; q < n; q++) {
            if ((Tm >> q) & 1) {
                slot_of[q] = p;
                q_at[p] = q;
                p++;
            } else if ((S >> q) & 1) {
                slot_of[q] = o++;   // a part qubit outside the tile: a slot past its slots
            }
        }
        int rank[64];   // place of a tile qubit among the tile's qubits
        std::memcpy(rank, slot_of, sizeof(rank));
        PartLaunch L;
        std::memset(&L, 0, sizeof(L));
        L.outer_mask = all & ~Tm;
        L.n = n;
        L.t = t;
        L.phase_begin = (uint32_t)prog.phases.size();
        L.op_begin = (uint32_t)prog.ops.size();
        L.coef_begin = (uint32_t)prog.coefs.size();
        for (int p = 0; p < t; p++) L.tile_q[p] = (uint8_t)q_at[p];
        // part factor: 1/sqrt2 per (unnormalised) H and e^{-i theta/2} per RZ
        double fr = 1.0, fi = 0.0;
        bool modulus = false;   // it holds more than phases
        auto fmul = [&](double dr, double di) {
            const double x = fr, y = fi;
            fr = x * dr - y * di;
            fi = x * di + y * dr;
        };
        // a factor goes into a merged diagonal's coefficients
        auto scale_by = [&](const Op &op, double dr, double di) {
            double *c = prog.coefs.data() + op.coef;
            for (int i = 0; i < (1 << R); i++) {
                const double x = c[2 * i], y = c[2 * i + 1];
                c[2 * i] = x * dr - y * di;
                c[2 * i + 1] = x * di + y * dr;
            }
        };
        auto scale_diag = [&](Op &op) {   // the part factor
            scale_by(op, fr, fi);
            if (modulus) op.a = 1;
            fr = 1.0;
            fi = 0.0;
            modulus = false;
        };
        auto unit_diag = [&]() {   // coefficients of a diagonal of ones
            const uint32_t at = (uint32_t)prog.coefs.size();
            for (int i = 0; i < (1 << R); i++) prog.coefs.insert(prog.coefs.end(), {1.0, 0.0});
            return at;
        };
        bool last_tphase = false;
        std::vector<int> remaining = gl;
        bool first = true;
        while (!remaining.empty()) {
            // pass 1: choose the register slots and the gates of this phase
            int sim_slot[64];
            std::memcpy(sim_slot, slot_of, sizeof(slot_of));
            uint32_t Rset = 0;
            uint64_t blocked = 0, blocked_nd = 0;   // for every gate; for gates non-diagonal on the qubit
            std::vector<int> sched, rest;
            std::vector<std::array<int, 2>> slot_before;   // tile slots of a scheduled gate's qubits
            if (inner && !inner->empty()) {
                // multi-level partitioning: the phase is the next second-level
                // part (the smallest inner id left; its gates in order)
                uint32_t next = UINT32_MAX;
                for (int g : remaining) next = std::min(next, (*inner)[g]);
                for (int g : remaining) {
                    if ((*inner)[g] != next) {
                        rest.push_back(g);
                        continue;
                    }
                    const GateRef &gr = gates[g];
                    Rset |= needed_slots(gr, sim_slot);
                    sched.push_back(g);
                    if (gr.kind == SV_GATE_SWAP) std::swap(sim_slot[gr.q[0]], sim_slot[gr.q[1]]);
                }
                if (popc(Rset) > R) {
                    err = "a second-level part needs " + std::to_string(popc(Rset)) + " register qubits > " +
                          std::to_string(R);
                    return false;
                }
            } else
            for (int g : remaining) {
                // gates that are diagonal on every qubit they share (phases,
                // controls) commute: a gate that stays behind blocks its
                // non-diagonal qubits for all others, its diagonal ones only
                // for gates that are not diagonal there
                const GateRef &gr = gates[g];
                const uint64_t nd = acts_nondiag(gr), dg = gmask[g] & ~nd;
                const uint32_t need = needed_slots(gr, sim_slot);
                if ((nd & (blocked | blocked_nd)) || (dg & blocked) ||
                    ((need & ~Rset) && popc(Rset | need) > R)) {
                    blocked |= nd;
                    blocked_nd |= dg;
                    rest.push_back(g);
                    continue;
                }
                Rset |= need;
                sched.push_back(g);
                slot_before.push_back({sim_slot[gr.q[0]], sim_slot[gr.q[1]]});
                if (gr.kind == SV_GATE_SWAP) std::swap(sim_slot[gr.q[0]], sim_slot[gr.q[1]]);
            }
            if (!(inner && !inner->empty())) {
                // A diagonal gate on thread bits alone costs a complex product
                // of every amplitude at the phase's end, while on a register
                // bit it joins the phase's merged diagonal. So it is left to a
                // later phase if one of its qubits must be resident in one
                // anyway and the gates of this phase that follow it on its
                // qubits are diagonal there too.
                uint64_t later = 0, need = 0;   // qubits that must be resident after this phase
                for (int g : rest)
                    if (gates[g].kind != SV_GATE_SWAP) need |= acts_nondiag(gates[g]);
                std::vector<int> keep;
                bool moved = false;
                for (size_t i = sched.size(); i-- > 0;) {
                    const int g = sched[i];
                    bool thread = Rset != 0 && is_diagonal(gates[g].kind) && (gmask[g] & need) && !(gmask[g] & later);
                    for (int j = 0; thread && j < gates[g].arity; j++) thread = !((Rset >> slot_before[i][j]) & 1);
                    if (thread) {
                        rest.push_back(g);
                        moved = true;
                        continue;
                    }
                    later |= acts_nondiag(gates[g]);
                    keep.push_back(g);
                }
                if (moved) {
                    std::sort(rest.begin(), rest.end());
                    std::reverse(keep.begin(), keep.end());
                    sched.swap(keep);
                }
                std::memcpy(sim_slot, slot_of, sizeof(slot_of));
                for (int g : sched)
                    if (gates[g].kind == SV_GATE_SWAP) std::swap(sim_slot[gates[g].q[0]], sim_slot[gates[g].q[1]]);
            }
            const bool last = rest.empty();
            if (sched.empty()) {
                err = "no gate of part " + std::to_string(pi) + " fits the register bits";
                return false;
            }
            // slot -> qubit at the end of this phase
            int q_end[64];
            for (int q = 0; q < n; q++)
                if ((Tm >> q) & 1) q_end[sim_slot[q]] = q;
            // Spare register bits go to the thread bits of diagonal gates, then
            // to the highest slots; in the last phase, which stores the tile,
            // to the slots that end on the highest qubits, since the lowest
            // five are the lanes of the store (with a register bit on one of
            // them 28-qubit passes lost 1 to 3 %; the QFT's swap passes, whose
            // high slots end on low qubits, ran at 0.34 to 0.46 of HBM).
            auto key_of = [&](int p) { return last ? rank[q_end[p]] : p; };
            if (!(inner && !inner->empty())) {
                int at[64];
                std::memcpy(at, slot_of, sizeof(slot_of));
                for (int g : sched) {
                    if (is_diagonal(gates[g].kind))
                        for (int j = 0; j < gates[g].arity; j++) {
                            const int sl = at[gates[g].q[j]];
                            if (popc(Rset) < R && sl < t && (!last || key_of(sl) >= 5)) Rset |= 1u << sl;
                        }
                    if (gates[g].kind == SV_GATE_SWAP) std::swap(at[gates[g].q[0]], at[gates[g].q[1]]);
                }
            }
            for (int v = t - 1; v >= 0 && popc(Rset) < R; v--)
                for (int p = 0; p < t; p++)
                    if (key_of(p) == v) Rset |= 1u << p;
            Phase ph;
            std::memset(&ph, 0, sizeof(ph));
            int rb[64], tbit[64], reg_slot[MAX_R], thr_slot[MAX_TB];
            for (int p = 0, b = 0; p < t; p++)
                if ((Rset >> p) & 1) {
                    reg_slot[b] = p;
                    rb[p] = b++;
                }
            std::vector<int> cand;
            std::vector<int> key(t, 0);
            for (int p = 0; p < t; p++) {
                if (!((Rset >> p) & 1)) cand.push_back(p);
                key[p] = key_of(p);   // the last phase stores: lanes on the lowest qubits
            }
            std::vector<int> thr = order_thread_slots(cand, key, fp64);
            for (size_t j = 0; j < thr.size(); j++) {
                thr_slot[j] = thr[j];
                tbit[thr[j]] = (int)j;
            }
            for (int q = 0; q < n; q++)
                if (((S & ~Tm) >> q) & 1) tbit[slot_of[q]] = OP_OUTER + q;
            // pass 2: emit ops
            ph.op_begin = (uint32_t)prog.ops.size();
            const double grown_before = std::hypot(fr, fi);   // not yet applied, of earlier phases
            bool tphase = false, tsign = false;
            auto coef = [&](std::initializer_list<double> v) {
                uint32_t at = (uint32_t)prog.coefs.size();
                prog.coefs.insert(prog.coefs.end(), v.begin(), v.end());
                return at;
            };
            auto emit = [&](uint8_t kind, int a, int b, int tb, uint32_t c) {
                Op op;
                op.kind = kind;
                op.a = (uint8_t)a;
                op.b = (uint8_t)b;
                op.tb = (uint8_t)tb;
                op.coef = c;
                prog.ops.push_back(op);
            };
            // one gate's ops (the gate alone)
            auto emit_one = [&](int g) -> bool {
                const GateRef &gr = gates[g];
                const double th = gr.theta;
                const int s0 = slot_of[gr.q[0]];
                const bool r0 = (Rset >> s0) & 1;
                switch (gr.kind) {
                case SV_GATE_H:
                    emit(OP_H, rb[s0], 0, 0, 0);
                    fmul(std::sqrt(0.5), 0.0);
                    modulus = true;
                    break;
                case SV_GATE_X: emit(OP_X, rb[s0], 0, 0, 0); break;
                case SV_GATE_Y: emit(OP_Y, rb[s0], 0, 0, 0); break;
                case SV_GATE_RX: case SV_GATE_RY: {
                    // the largest entry joins the part factor: RX = c [[1, -it], [-it, 1]]
                    // (t = s/c) or -is [[it, 1], [1, it]] (t = c/s); RY = c [[1, -t], [t, 1]]
                    // or s [[t, -1], [1, t]], whichever keeps |t| <= 1
                    const double c = std::cos(th / 2), sn = std::sin(th / 2);
                    const bool rx = gr.kind == SV_GATE_RX;
                    modulus = true;
                    if (std::fabs(c) >= std::fabs(sn)) {
                        fmul(c, 0.0);
                        emit(rx ? OP_RXS : OP_RYS, rb[s0], 0, 0, coef({sn / c}));
                    } else {
                        if (rx) fmul(0.0, -sn);
                        else fmul(sn, 0.0);
                        emit(rx ? OP_RXS : OP_RYS, rb[s0], 1, 0, coef({c / sn}));
                    }
                } break;
                case SV_GATE_Z: case SV_GATE_S: case SV_GATE_T: case SV_GATE_P: {
                    double ang = gr.kind == SV_GATE_Z ? M_PI : gr.kind == SV_GATE_S ? M_PI / 2 : gr.kind == SV_GATE_T ? M_PI / 4 : th;
                    double dr = gr.kind == SV_GATE_Z ? -1.0 : std::cos(ang), di = gr.kind == SV_GATE_Z ? 0.0 : std::sin(ang);
                    if (gr.kind == SV_GATE_S) { dr = 0.0; di = 1.0; }
                    if (r0) {
                        if (gr.kind == SV_GATE_Z) emit(OP_Z, rb[s0], 0, 0, 0);
                        else emit(OP_P, rb[s0], 0, 0, coef({dr, di}));
                    } else if (gr.kind == SV_GATE_Z) {
                        emit(OP_TSG, 0, tbit[s0], tbit[s0], 0);
                        tsign = true;
                    } else {
                        emit(OP_TD, 0, 0, tbit[s0], coef({1.0, 0.0, dr, di}));
                        tphase = true;
                    }
                } break;
                case SV_GATE_RZ: {
                    // RZ(t) = e^{-it/2} diag(1, e^{it}): the global phase joins the part factor
                    fmul(std::cos(th / 2), -std::sin(th / 2));
                    if (r0) emit(OP_P, rb[s0], 0, 0, coef({std::cos(th), std::sin(th)}));
                    else {
                        emit(OP_TD, 0, 0, tbit[s0], coef({1.0, 0.0, std::cos(th), std::sin(th)}));
                        tphase = true;
                    }
                } break;
                case SV_GATE_CX: {
                    const int s1 = slot_of[gr.q[1]];
                    if (r0) emit(OP_CX, rb[s0], rb[s1], 0, 0);
                    else emit(OP_CXT, 0, rb[s1], tbit[s0], 0);
                } break;
                case SV_GATE_CZ: case SV_GATE_CP: {
                    const int s1 = slot_of[gr.q[1]];
                    const bool r1 = (Rset >> s1) & 1;
                    const bool cz = gr.kind == SV_GATE_CZ;
                    const double dr = cz ? -1.0 : std::cos(th), di = cz ? 0.0 : std::sin(th);
                    if (r0 && r1) {
                        if (cz) emit(OP_CZ, rb[s0], rb[s1], 0, 0);
                        else emit(OP_CP, rb[s0], rb[s1], 0, coef({dr, di}));
                    } else if (r0 || r1) {
                        const int rs = r0 ? s0 : s1, ts = r0 ? s1 : s0;
                        if (cz) emit(OP_CZT, rb[rs], 0, tbit[ts], 0);
                        else emit(OP_CPT, rb[rs], 0, tbit[ts], coef({dr, di}));
                    } else if (cz) {
                        emit(OP_TSG, 0, tbit[s1], tbit[s0], 0);
                        tsign = true;
                    } else {
                        emit(OP_TP2, 0, tbit[s1], tbit[s0], coef({dr, di}));
                        tphase = true;
                    }
                } break;
                case SV_GATE_SWAP:
                    std::swap(slot_of[gr.q[0]], slot_of[gr.q[1]]);
                    break;
                default:
                    err = "unknown gate kind";
                    return false;
                }
                return true;
            };
            // the product of a run of one-qubit gates on qubit q as one op
            auto emit_product = [&](int q, const std::vector<int> &run) -> bool {
                if (run.size() == 1) return emit_one(run[0]);
                double M[8] = {1, 0, 0, 0, 0, 0, 1, 0};
                for (int g : run) {
                    double U[8], T[8];
                    gate_matrix_1q(gates[g].kind, gates[g].theta, U);
                    for (int r = 0; r < 2; r++)
                        for (int c = 0; c < 2; c++) {
                            double re = 0, im = 0;
                            for (int k = 0; k < 2; k++) {
                                const double ar = U[2 * (2 * r + k)], ai = U[2 * (2 * r + k) + 1];
                                const double br = M[2 * (2 * k + c)], bi = M[2 * (2 * k + c) + 1];
                                re += ar * br - ai * bi;
                                im += ar * bi + ai * br;
                            }
                            T[2 * (2 * r + c)] = re;
                            T[2 * (2 * r + c) + 1] = im;
                        }
                    std::memcpy(M, T, sizeof(M));
                }
                const int sq = slot_of[q];
                const double off = std::hypot(M[2], M[3]) + std::hypot(M[4], M[5]);
                if (off < 1e-14) {
                    // diag(m00, m11) = m00 diag(1, m11 / m00), |m00| = 1
                    const double d0r = M[0], d0i = M[1], d1r = M[6], d1i = M[7];
                    fmul(d0r, d0i);
                    const double pr = d1r * d0r + d1i * d0i, pi = d1i * d0r - d1r * d0i;
                    if (std::fabs(pr - 1.0) < 1e-15 && std::fabs(pi) < 1e-15) return true;   // identity
                    if ((Rset >> sq) & 1) emit(OP_P, rb[sq], 0, 0, coef({pr, pi}));
                    else {
                        emit(OP_TD, 0, 0, tbit[sq], coef({1.0, 0.0, pr, pi}));
                        tphase = true;
                    }
                    return true;
                }
                if (!((Rset >> sq) & 1)) {
                    err = "fused non-diagonal gate on a thread slot";
                    return false;
                }
                // divide by the larger of m00 and m01 (the part factor takes it):
                // [[1, u], [v, w]] or [[u, 1], [v, w]], entries of modulus <= 1
                {
                    const bool f1 = std::hypot(M[2], M[3]) > std::hypot(M[0], M[1]);
                    const double pr = f1 ? M[2] : M[0], pi = f1 ? M[3] : M[1];
                    const double den = pr * pr + pi * pi;
                    auto div = [&](double xr, double xi, double &qr, double &qi) {
                        qr = (xr * pr + xi * pi) / den;
                        qi = (xi * pr - xr * pi) / den;
                    };
                    double ur, ui, vr, vi, wr, wi;
                    div(f1 ? M[0] : M[2], f1 ? M[1] : M[3], ur, ui);
                    div(M[4], M[5], vr, vi);
                    div(M[6], M[7], wr, wi);
                    fmul(pr, pi);
                    modulus = true;
                    emit(OP_U2S, rb[sq], f1 ? 1 : 0, 0, coef({ur, ui, vr, vi, wr, wi}));
                }
                return true;
            };
            // Runs of one-qubit gates on one qubit with no multi-qubit gate on it
            // in between (gates on other qubits commute with them) become one
            // op: their product, as a phase (diagonal; the entry of |0> joins
            // the part factor) or a general 2x2 matrix. With fewer than three
            // non-diagonal gates the run stays those gates and one phase
            // between them: 2 or 4 flops per amplitude and gate, and the
            // phases mostly join a merged diagonal, against 11 for the matrix.
            auto emit_fused = [&](int q, const std::vector<int> &whole) -> bool {
                int nondiag = 0;
                for (int g : whole) nondiag += !is_diagonal(gates[g].kind);
                if (nondiag == 0 || nondiag > 2) return emit_product(q, whole);
                std::vector<int> diag;
                for (int g : whole) {
                    if (is_diagonal(gates[g].kind)) {
                        diag.push_back(g);
                        continue;
                    }
                    if (!diag.empty() && !emit_product(q, diag)) return false;
                    diag.clear();
                    if (!emit_one(g)) return false;
                }
                return diag.empty() || emit_product(q, diag);
            };
            std::vector<std::vector<int>> pend(n);
            std::vector<int> pend_order;
            auto flush = [&](int q) -> bool {
                if (pend[q].empty()) return true;
                const bool ok = emit_fused(q, pend[q]);
                pend[q].clear();
                return ok;
            };
            for (int g : sched) {
                const GateRef &gr = gates[g];
                if (gr.arity == 1) {
                    if (pend[gr.q[0]].empty()) pend_order.push_back(gr.q[0]);
                    pend[gr.q[0]].push_back(g);
                    continue;
                }
                for (int j = 0; j < gr.arity; j++)
                    if (!flush(gr.q[j])) return false;
                if (!emit_one(g)) return false;
            }
            for (int q : pend_order)
                if (!flush(q)) return false;
            // the last phase's per-thread phase is applied with the part factor at the store
            // Diagonal gates on register bits commute with each other and with
            // every op on other register bits: a run of them (interleaved with
            // such ops) merges into one OP_DIAG holding the product's phase for
            // each of the 2^R register indices. The run ends where an op acts
            // non-diagonally on a register bit the product depends on.
            {
                const int NR = 1 << R;
                std::vector<Op> in(prog.ops.begin() + ph.op_begin, prog.ops.end());
                prog.ops.resize(ph.op_begin);
                std::vector<double> D(2 * NR);
                uint32_t dep = 0;
                int merged = 0;
                Op single{};
                auto reset = [&]() {
                    for (int i = 0; i < NR; i++) { D[2 * i] = 1.0; D[2 * i + 1] = 0.0; }
                    dep = 0;
                    merged = 0;
                };
                auto mulphase = [&](int i, double pr, double pi) {
                    const double x = D[2 * i], y = D[2 * i + 1];
                    D[2 * i] = x * pr - y * pi;
                    D[2 * i + 1] = x * pi + y * pr;
                };
                auto flush = [&]() {
                    if (merged == 1) prog.ops.push_back(single);
                    else if (merged > 1) {
                        Op op{};
                        op.kind = OP_DIAG;
                        op.coef = (uint32_t)prog.coefs.size();
                        prog.coefs.insert(prog.coefs.end(), D.begin(), D.end());
                        prog.ops.push_back(op);
                    }
                    reset();
                };
                reset();
                for (const Op &op : in) {
                    const double *c = prog.coefs.data() + op.coef;
                    bool diag = true;
                    switch (op.kind) {
                    case OP_P: for (int i = 0; i < NR; i++) if ((i >> op.a) & 1) mulphase(i, c[0], c[1]); break;
                    case OP_Z: for (int i = 0; i < NR; i++) if ((i >> op.a) & 1) mulphase(i, -1.0, 0.0); break;
                    case OP_CZ:
                        for (int i = 0; i < NR; i++) if (((i >> op.a) & 1) && ((i >> op.b) & 1)) mulphase(i, -1.0, 0.0);
                        break;
                    case OP_CP:
                        for (int i = 0; i < NR; i++) if (((i >> op.a) & 1) && ((i >> op.b) & 1)) mulphase(i, c[0], c[1]);
                        break;
                    default: diag = false; break;
                    }
                    if (diag) {
                        dep |= 1u << op.a;
                        if (op.kind == OP_CZ || op.kind == OP_CP) dep |= 1u << op.b;
                        merged++;
                        single = op;
                        continue;
                    }
                    // register bits the op acts on non-diagonally
                    uint32_t touch = 0;
                    switch (op.kind) {
                    case OP_H: case OP_X: case OP_Y: case OP_RXS: case OP_RYS: case OP_U2S: touch = 1u << op.a; break;
                    case OP_CX: touch = (1u << op.a) | (1u << op.b); break;
                    case OP_CXT: touch = 1u << op.b; break;
                    default: touch = 0; break;   // thread-bit phases: diagonal, they commute
                    }
                    if (touch & dep) flush();
                    prog.ops.push_back(op);
                }
                flush();
            }
            // A phase may hold any number of gates on its register bits, each
            // growing the unnormalised amplitudes by up to sqrt2: where their
            // factors reach 2^-40 the modulus gathered so far is applied in
            // the middle of the phase, long before a float's range ends (the
            // part factor below may join the same diagonal: 2^-80).
            {
                const std::vector<Op> in(prog.ops.begin() + ph.op_begin, prog.ops.end());
                prog.ops.resize(ph.op_begin);
                double grown = grown_before;
                for (const Op &op : in) {
                    prog.ops.push_back(op);
                    grown *= factor_of(op, prog.coefs);
                    if (grown >= 0x1p-40) continue;
                    emit(OP_DIAG, 1, 0, 0, unit_diag());
                    scale_by(prog.ops.back(), grown, 0.0);
                    fr /= grown;
                    fi /= grown;
                    grown = 1.0;
                }
            }
            if (tphase && !last) emit(OP_TAPPLY, 0, 0, 0, 0);
            if (tsign) emit(OP_TSAPPLY, 0, 0, 0, 0);
            // a part of many phases (a whole circuit) applies the part factor
            // before the unnormalised amplitudes grow out of range: into a
            // merged diagonal of the phase, else as one of its own
            if (!last && std::hypot(fr, fi) < 0x1p-24) {
                uint32_t o = ph.op_begin;
                while (o < (uint32_t)prog.ops.size() && prog.ops[o].kind != OP_DIAG) o++;
                if (o == (uint32_t)prog.ops.size()) emit(OP_DIAG, 0, 0, 0, unit_diag());
                scale_diag(prog.ops[o]);
            }
            if (last) last_tphase = tphase;
            // CX gates at either end of the phase go into its layouts: param
            // circuits of 15 layers at 21 qubits 628 -> 535 us, at 18 qubits
            // 193 -> 164; layered 21q 346 -> 331. Only in the interpreter's
            // programs: a specialised kernel renames registers, which costs
            // nothing either, and selects for a control on a thread bit. A CX
            // of the last phase whose control is one of the lowest five
            // qubits stays a gate: its lanes would store to different lines.
            {
                std::vector<Op> ops(prog.ops.begin() + ph.op_begin, prog.ops.end());
                const size_t N = ops.size();
                std::vector<char> fold(N, 0);   // 1: into the write layout, 2: into the read layout
                auto touch = [&](const Op &op, uint32_t &any, uint32_t &nd) {
                    switch (op.kind) {
                    case OP_H: case OP_RXS: case OP_RYS: case OP_U2S: case OP_Y: case OP_X:
                        any |= 1u << op.a; nd |= 1u << op.a; break;
                    case OP_CX: any |= (1u << op.a) | (1u << op.b); nd |= 1u << op.b; break;
                    case OP_CXT: any |= 1u << op.b; nd |= 1u << op.b; break;
                    case OP_P: case OP_Z: case OP_CPT: case OP_CZT: any |= 1u << op.a; break;
                    case OP_CP: case OP_CZ: any |= (1u << op.a) | (1u << op.b); break;
                    case OP_DIAG: {
                        const double *c = prog.coefs.data() + op.coef;
                        for (int b = 0; b < R; b++)
                            for (int i = 0; i < (1 << R); i++) {
                                const int j = i ^ (1 << b);
                                if (c[2 * i] != c[2 * j] || c[2 * i + 1] != c[2 * j + 1]) any |= 1u << b;
                            }
                    } break;
                    default: break;   // conditions on thread bits, which no gate of the phase moves
                    }
                };
                auto foldable = [&](const Op &op, uint32_t any, uint32_t nd, bool write, bool lanes) {
                    if (outer_diag || (op.kind != OP_CX && op.kind != OP_CXT)) return false;
                    if ((any >> op.b) & 1) return false;
                    if (op.kind == OP_CX && ((nd >> op.a) & 1)) return false;
                    if (op.kind != OP_CXT) return true;
                    if (op.tb < 5 && !lanes) return false;
                    return !(write && last && key_of(thr_slot[op.tb]) < 5);
                };
                // G of an op on an index given as a set of slots
                auto act = [&](const Op &op, uint16_t v) -> uint16_t {
                    const int c = op.kind == OP_CX ? reg_slot[op.a] : thr_slot[op.tb];
                    return (v >> c) & 1 ? (uint16_t)(v ^ (1u << reg_slot[op.b])) : v;
                };
                auto apply = [&](Layout &l, const Op &op) {
                    for (int b = 0; b < R; b++) l.reg[b] = act(op, l.reg[b]);
                    for (int j = 0; j < t - R; j++) l.thr[j] = act(op, l.thr[j]);
                };
                Layout plain;
                std::memset(&plain, 0, sizeof(plain));
                for (int b = 0; b < R; b++) plain.reg[b] = (uint16_t)(1u << reg_slot[b]);
                for (int j = 0; j < t - R; j++) plain.thr[j] = (uint16_t)(1u << thr_slot[j]);
                // a CX under a lane bit moves lanes: only where the warp's
                // accesses stay on as many shared-memory banks
                for (int lanes = 1; lanes >= 0; lanes--) {
                    std::fill(fold.begin(), fold.end(), 0);
                    uint32_t any = 0, nd = 0;
                    for (size_t k = N; k-- > 0;) {
                        if (foldable(ops[k], any, nd, true, lanes)) fold[k] = 1;
                        else touch(ops[k], any, nd);
                    }
                    any = nd = 0;
                    for (size_t k = 0; k < N; k++) {
                        if (!fold[k] && foldable(ops[k], any, nd, false, lanes)) fold[k] = 2;
                        else touch(ops[k], any, nd);
                    }
                    ph.rd = ph.wr = plain;
                    // write: the amplitude at index v goes to G_k .. G_1 v; read: the
                    // state after the leading gates at v is the one before at G_1 .. G_k v
                    for (size_t k = 0; k < N; k++)
                        if (fold[k] == 1) apply(ph.wr, ops[k]);
                    for (size_t k = N; k-- > 0;)
                        if (fold[k] == 2) apply(ph.rd, ops[k]);
                    const int banks = bank_rank(plain, fp64);
                    if (bank_rank(ph.rd, fp64) == banks && (last || bank_rank(ph.wr, fp64) == banks)) break;
                }
                prog.ops.resize(ph.op_begin);
                for (size_t k = 0; k < N; k++)
                    if (!fold[k]) prog.ops.push_back(ops[k]);
            }
            ph.op_count = (uint32_t)prog.ops.size() - ph.op_begin;
            prog.phases.push_back(ph);
            if (last) {
                auto qubits = [&](uint16_t v) {
                    uint64_t m = 0;
                    for (int p = 0; p < t; p++)
                        if ((v >> p) & 1) m |= 1ull << q_end[p];
                    return m;
                };
                for (int b = 0; b < R; b++) L.store_reg[b] = qubits(ph.wr.reg[b]);
                for (int j = 0; j < t - R; j++) L.store_thr[j] = qubits(ph.wr.thr[j]);
            }
            remaining.swap(rest);
            first = false;
        }
        L.n_phases = (uint32_t)prog.phases.size() - L.phase_begin;
        L.op_end = (uint32_t)prog.ops.size();
        L.coef_end = (uint32_t)prog.coefs.size();
        // the part factor is one complex scalar: any op that multiplies every
        // amplitude by a per-index phase (a merged diagonal) takes it into its
        // coefficients, which saves the multiply at the store unless the last
        // phase also left a per-thread phase to apply there
        if (!last_tphase && (fr != 1.0 || fi != 0.0)) {
            for (uint32_t o = L.op_begin; o < (uint32_t)prog.ops.size(); o++) {
                if (prog.ops[o].kind != OP_DIAG) continue;
                scale_diag(prog.ops[o]);
                break;
            }
        }
        L.gr = fr;
        L.gi = fi;
        L.flags = (last_tphase || fr != 1.0 || fi != 0.0) ? PL_STORE_FACTOR : 0u;
        // every other pass takes the tiles backwards: it begins with what the
        // pass before wrote last, which L2 still holds (layered circuits, k =
        // 7 to 9 specialised: 24 qubits 699 -> 610 and 1156 -> 1072 us, 26 qubits
        // 4.60 -> 4.51 ms, 28 qubits 21.29 -> 21.24; tensor-core passes at 24
        // qubits 1.64 -> 1.52 ms; up to 23 qubits the state stays in L2 anyway)
        if (prog.kind.size() & 1) L.flags |= PL_REVERSE;
        prog.kind.push_back(0);
        prog.index.push_back((uint32_t)prog.parts.size());
        prog.parts.push_back(L);
        prog.n_tiles.push_back(1ull << (n - t));
    }
    return true;
}

// Real floating-point operations per amplitude of the whole state that the
// program's kernels execute (an FMA counts two; sign changes, permutations
// and shared-memory moves count none): per op of a gate-list part, the
// arithmetic of its template in ops_core.cuh over the amplitudes it touches,
// plus the store factor (gather: a run of OP_CPT on a register bit is one
// product, as the specialised kernels apply it); per dense part, the split-BF16 products (3 x 128
// real MACs per real output, 1536 per complex amplitude, tensor cores).
void program_flops(const Program &prog, double &alu_per_amp, double &tensor_per_amp, bool gather) {
    alu_per_amp = 0.0;
    tensor_per_amp = 0.0;
    const int NR = 1 << prog.R;
    for (size_t i = 0; i < prog.kind.size(); i++) {
        if (prog.kind[i] == 1 || prog.kind[i] == 2) {
            tensor_per_amp += (prog.kind[i] == 2 ? 2.0 : 1.0) * 2.0 * 3.0 * 2.0 * 128.0;
            continue;
        }
        const PartLaunch &L = prog.parts[prog.index[i]];
        for (uint32_t p = 0; p < L.n_phases; p++) {
            const Phase &ph = prog.phases[L.phase_begin + p];
            uint32_t gathered = 0;   // register bits whose OP_CPT run is one product (specialised kernels)
            for (uint32_t k = 0; k < ph.op_count; k++) {
                const Op &op = prog.ops[ph.op_begin + k];
                switch (op.kind) {
                case OP_H: case OP_RXS: case OP_RYS: case OP_U2S: case OP_X: case OP_Y: gathered &= ~(1u << op.a); break;
                case OP_CX: case OP_CXT: gathered &= ~(1u << op.b); break;
                default: break;
                }
                switch (op.kind) {
                case OP_H: alu_per_amp += 2.0; break;                 // a + b, a - b per component pair
                case OP_RXS: case OP_RYS: alu_per_amp += 4.0; break;  // one multiply-add per component
                case OP_U2S: alu_per_amp += 11.0; break;              // x + u y (8), v x + w y (14) per pair
                case OP_DIAG: case OP_TAPPLY: alu_per_amp += 6.0; break;   // complex product, all
                case OP_P: alu_per_amp += 3.0; break;                 // complex product on half
                case OP_CPT:
                    if (!gather || !((gathered >> op.a) & 1)) alu_per_amp += 3.0;
                    gathered |= 1u << op.a;
                    break;
                case OP_CP: alu_per_amp += 1.5; break;                // complex product on a quarter
                default: break;                                       // X, Y, Z, CX, CZ, SWAP, thread phases
                }
            }
        }
        if (L.flags & PL_STORE_FACTOR) alu_per_amp += 6.0;
        (void)NR;
    }
}

}  // namespace hisv
