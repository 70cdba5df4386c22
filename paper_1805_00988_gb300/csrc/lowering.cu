// lowering.cu -- circuit gates to the planners' gate form.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>
#include <vector>

#include "internal.cuh"

namespace qsim {

bool commute(const SGate &a, const SGate &b)
{
    const uint64_t shared = (a.xq() | a.dq()) & (b.xq() | b.dq());
    return (shared & (a.xq() | b.xq())) == 0;
}

// Columns orthogonal and of length 1, so both singular values are 1.  (The norm bound
// alone would let contractions and projectors pass.)
bool unitary_2x2(const double m[8])
{
    const std::complex<double> a(m[0], m[1]), b(m[2], m[3]), c(m[4], m[5]), d(m[6], m[7]);
    constexpr double tol = 1e-6;
    return std::abs(std::norm(a) + std::norm(c) - 1.0) < tol && std::abs(std::norm(b) + std::norm(d) - 1.0) < tol &&
           std::abs(std::conj(a) * b + std::conj(c) * d) < tol;
}

// SWAP(a, b) with controls c = CNOT(b -> a) . X(target b; controls c + a) . CNOT(b -> a)
static void lower_one(const sim_gate &gate, size_t k, const int *at, std::vector<SGate> *out)
{
    static const double X[8] = {0, 0, 1, 0, 1, 0, 0, 0};
    const PairGate p = make_pair_gate(gate);
    uint64_t cm = 0;
    for (int c = 0; c < p.nctrl; ++c) cm |= 1ull << at[p.ctrl[c]];
    if (p.op == OP_IDENTITY) return;
    if (p.op == OP_SWAP) {
        const int a = at[p.target], b = at[p.target2];
        SGate g1{OP_XPERM, a, 1ull << b, {}, (int)k};
        SGate g2{OP_XPERM, b, cm | (1ull << a), {}, (int)k};
        memcpy(g1.m, X, sizeof X);
        memcpy(g2.m, X, sizeof X);
        out->push_back(g1);
        out->push_back(g2);
        out->push_back(g1);
        return;
    }
    SGate g{p.op, at[p.target], cm, {}, (int)k};
    memcpy(g.m, p.m, sizeof g.m);
    out->push_back(g);
}

void lower_gates(const sim_gate *gates, size_t n_gates, std::vector<SGate> *out)
{
    int same[64];
    for (int q = 0; q < 64; ++q) same[q] = q;
    for (size_t k = 0; k < n_gates; ++k) lower_one(gates[k], k, same, out);
}

void lower_renamed(const sim_gate *gates, size_t n_gates, int n, std::vector<SGate> *out)
{
    int at[64];                    // where the circuit's qubit q lives
    for (int q = 0; q < 64; ++q) at[q] = q;
    for (size_t k = 0; k < n_gates; ++k) {
        if (gates[k].kind == SIM_GATE_SWAP && gates[k].n_controls == 0) std::swap(at[gates[k].target], at[gates[k].target2]);
        else lower_one(gates[k], k, at, out);
    }
    // bring qubit q back to place q, one exchange of places after the other
    // (around the lowest place of each cycle, which most tiles hold)
    for (int q = 0; q < n; ++q)
        while (at[q] != q) {
            const int p = at[q];              // place q holds another qubit; swap places q and p
            SGate g{OP_SWAP, std::min(p, q), 0, {}, -1};
            g.target2 = std::max(p, q);
            out->push_back(g);
            for (int r = 0; r < n; ++r)
                if (at[r] == q && r != q) {
                    at[r] = p;
                    break;
                }
            at[q] = q;
        }
}

double sgate_flops(const SGate &g, int n)
{
    const double amps = std::ldexp(1.0, n - __builtin_popcountll(g.ctrl));
    switch (g.op) {
    case OP_DENSE: return 16.0 * amps;                 // two complex MACs per amplitude
    case OP_ANTIDIAG: return 6.0 * amps;               // one complex multiply per amplitude
    case OP_DIAG: return 6.0 * amps;
    case OP_DIAG_HI:                                   // only the |1> half; a sign flip is a move
        return (g.m[6] == -1.0 && g.m[7] == 0.0) ? 0.0 : 3.0 * amps;
    case OP_SUPER: return 32.0 * amps;                 // four complex MACs per amplitude
    default: return 0.0;                               // exchanges
    }
}

}  // namespace qsim
