// tile.cuh -- register layouts of a tile, the host pass planner, and the
// record schedule of a pass (for 256 threads a tile).  No kernel runs the records: the cost
// model's features count them, and sim_plan_describe (all but its passes) and
// sim_plan_staged_ops report them.  What the kernels run is compiled from the
// passes by tileprog.cuh.  See staged.cu for the design.
#pragma once

#include <complex>
#include <cstring>
#include <vector>

#include "internal.cuh"

namespace qsim {
namespace {


constexpr int kLow = 5;          // qubits 0..4 are local bits 0..4 of every tile
constexpr int kThrBits = 8;      // thread bits of the record schedule

enum StKind { SK_LAYOUT = 0, SK_DENSE, SK_ANTI, SK_XPERM, SK_DIAG, SK_PHASE, SK_NEG, SK_RAMP, SK_NOP };

// SK_RAMP: a run of controlled phases that share one qubit q, each pairing q
// with a tile-local qubit m (phase f_m when both bits are 1), applied at
// once: amplitudes whose q bit is 1 are multiplied by the product of f_m over
// the local bits m that are 1 -- the product over the thread's thread bits
// times the product over the register's register bits.  The host tabulates
// both: entry k < RA is register k's product, entries RA + x and RA + 16 + y
// the products over thread bits 0..3 set in x and 4..7 set in y, so a thread
// forms its factor from two entries and each register needs one more.  Entry
// e sits in record e / 4 of the op, coefficient slots 2 (e % 4) and
// 2 (e % 4) + 1; the first record also carries q as a diagonal op's target
// (km_t / thr_t / out_t).  The other records, and the padding that keeps a
// ramp inside one staged chunk of kOpChunk ops, are SK_NOP records.
__host__ __device__ constexpr int ramp_records(int RA) { return (RA + 32 + 3) / 4; }
constexpr int kOpChunk = 64;      // a ramp's records stay inside one run of this many
static_assert(kThrBits == 8, "ramp tables cover thread bits as two groups of four");

template <typename R>
struct __align__(16) StOp {
    int32_t kind;      // StKind
    int32_t arg;       // exchange ops: register bit of the target; SK_LAYOUT: new layout
    uint32_t thr_c;    // thread bits that must be 1
    int32_t plain;     // exchange ops: no condition of any kind
    uint64_t out_c;    // global bits (outside the tile) that must be 1
    uint64_t km_c;     // bit k: register k satisfies the register-bit conditions
    uint64_t km_t;     // diagonal ops, bit k: the target bit of register k is 1
    uint32_t thr_t;    // diagonal ops: thread bit of the target (0 if not a thread bit)
    uint32_t pad;
    uint64_t out_t;    // diagonal ops: global bit of the target (0 if inside the tile)
    R m[8];            // A, B, C, D
};

// ---------------------------------------------------------------- layouts
// VEC = 2 for complex64 (the I/O layout keeps local bit 0 in registers so a
// thread loads two neighbouring amplitudes as one 16-byte vector), 1 for
// complex128.  Layout 0 is the I/O layout; layouts 1.. put windows of RB
// consecutive local bits into registers.
__host__ __device__ constexpr int n_layouts(int M, int RB) { return 1 + (M - RB + RB - 1) / RB; }

__host__ __device__ constexpr int reg_local(int M, int RB, int VEC, int l, int j)
{
    if (l == 0) return (VEC == 2) ? (j == 0 ? 0 : M - RB + j) : (M - RB + j);
    int s = (VEC == 2 ? 1 : 0) + RB * (l - 1);
    if (s > M - RB) s = M - RB;
    return s + j;
}

__host__ __device__ constexpr bool is_reg(int M, int RB, int VEC, int l, int b)
{
    for (int j = 0; j < RB; ++j)
        if (reg_local(M, RB, VEC, l, j) == b) return true;
    return false;
}

__host__ __device__ constexpr int thr_local(int M, int RB, int VEC, int l, int i)
{
    int c = 0;
    for (int b = 0; b < M; ++b)
        if (!is_reg(M, RB, VEC, l, b)) {
            if (c == i) return b;
            ++c;
        }
    return -1;
}

__host__ __device__ constexpr int reg_part(int M, int RB, int VEC, int l, int k)
{
    int x = 0;
    for (int j = 0; j < RB; ++j)
        if ((k >> j) & 1) x |= 1 << reg_local(M, RB, VEC, l, j);
    return x;
}

struct TileGeom {
    int n_outer;
    int outer_pos[40];   // global qubit of outer bit i (ascending)
    int hpos[16];        // global qubit of local bit kLow + i
};

// ---------------------------------------------------------------- host planner
struct Pass {
    std::vector<int> high;      // global qubits of local bits kLow .. M-1
    std::vector<int> members;   // gate indices (a valid order)
};

// Greedy passes: scan the remaining gates in order; a gate joins the pass if
// it commutes with every gate skipped before it and its non-diagonal qubits
// fit in Q (adding up to M - kLow high qubits).
class PassFormer {
public:
    PassFormer(const std::vector<SGate> &g, int n, int M) : g_(g), n_(n), cap_(M - kLow), done_(g.size(), 0) {}

    // false when every gate has been given to a pass
    bool next(Pass *out)
    {
        while (first_ < g_.size() && done_[first_]) ++first_;
        if (first_ >= g_.size()) return false;
        Pass ps;
        uint64_t qmask = (1ull << kLow) - 1ull;
        uint64_t bx = 0, bd = 0;      // qubits where skipped gates act non-diagonally / diagonally
        for (size_t i = first_; i < g_.size(); ++i) {
            if (done_[i]) continue;
            const uint64_t x = g_[i].xq(), d = g_[i].dq();
            const bool free_of_skipped = ((x & (bx | bd)) == 0) && ((d & bx) == 0);
            const uint64_t add = x & ~qmask;
            if (free_of_skipped && (int)ps.high.size() + __builtin_popcountll(add) <= cap_) {
                for (uint64_t m = add; m; m &= m - 1) ps.high.push_back(__builtin_ctzll(m));
                qmask |= add;
                ps.members.push_back((int)i);
                done_[i] = 1;
            } else {
                bx |= x;
                bd |= d;
            }
        }
        // fill the tile with unused qubits (lowest first)
        for (int q = kLow; q < n_ && (int)ps.high.size() < cap_; ++q)
            if (!((qmask >> q) & 1)) { ps.high.push_back(q); qmask |= 1ull << q; }
        *out = ps;
        return true;
    }
    // the gates no pass has yet, if none of them is an exchange
    bool only_diagonal_left(std::vector<int> *left) const
    {
        left->clear();
        for (size_t i = first_; i < g_.size(); ++i) {
            if (done_[i]) continue;
            if (g_[i].xq()) return false;
            left->push_back((int)i);
        }
        return true;
    }
    void finish() { first_ = g_.size(); }

private:
    const std::vector<SGate> &g_;
    int n_, cap_;
    std::vector<char> done_;
    size_t first_ = 0;
};

inline std::vector<Pass> form_passes(const std::vector<SGate> &g, int n, int M)
{
    std::vector<Pass> passes;
    PassFormer f(g, n, M);
    Pass p;
    while (f.next(&p)) passes.push_back(p);
    return passes;
}

// a controlled phase on two qubits (phase on |11>, not a sign flip, which
// the lazy sign mask handles for free): a candidate for a ramp
inline bool ramp_candidate(const SGate &g)
{
    return g.op == OP_DIAG_HI && __builtin_popcountll(g.ctrl) == 1 && !(g.m[6] == -1.0 && g.m[7] == 0.0);
}

template <typename R>
struct PlanBuilder {
    int n, M, RB, VEC;
    std::vector<StOp<R>> ops;
    std::vector<int> order;       // circuit index of each emitted gate op
    int layout_changes = 0;
    size_t pass_start = 0;        // first op of the pass being scheduled (chunks count from it)
    bool allow_ramps = true;      // merge runs of controlled phases into SK_RAMP ops
    size_t filler = 0;            // SK_NOP records (a ramp's table records and padding)

    int local_of(const Pass &ps, int q) const
    {
        if (q < kLow) return q;
        for (size_t i = 0; i < ps.high.size(); ++i)
            if (ps.high[i] == q) return kLow + (int)i;
        return -1;
    }
    int reg_of(int l, int b) const
    {
        for (int j = 0; j < RB; ++j)
            if (reg_local(M, RB, VEC, l, j) == b) return j;
        return -1;
    }
    int thr_of(int l, int b) const
    {
        for (int i = 0; i < kThrBits; ++i)
            if (thr_local(M, RB, VEC, l, i) == b) return i;
        return -1;
    }

    void emit_gate(const Pass &ps, const SGate &g, int layout)
    {
        StOp<R> o;
        memset(&o, 0, sizeof o);
        uint32_t reg_c = 0, reg_t = 0;
        for (int q = 0; q < n; ++q) {
            if (!((g.ctrl >> q) & 1)) continue;
            const int b = local_of(ps, q);
            if (b < 0) o.out_c |= 1ull << q;
            else if (reg_of(layout, b) >= 0) reg_c |= 1u << reg_of(layout, b);
            else o.thr_c |= 1u << thr_of(layout, b);
        }
        for (int k = 0; k < 8; ++k) o.m[k] = (R)g.m[k];
        const int bt = local_of(ps, g.target);
        if (g.op == OP_DIAG || g.op == OP_DIAG_HI) {
            if (bt < 0) o.out_t = 1ull << g.target;
            else if (reg_of(layout, bt) >= 0) reg_t = 1u << reg_of(layout, bt);
            else o.thr_t = 1u << thr_of(layout, bt);
            const bool neg = g.m[6] == -1.0 && g.m[7] == 0.0;
            o.kind = (g.op == OP_DIAG) ? SK_DIAG : (neg ? SK_NEG : SK_PHASE);
        } else {
            o.kind = (g.op == OP_DENSE) ? SK_DENSE : (g.op == OP_ANTIDIAG) ? SK_ANTI : SK_XPERM;
            o.arg = reg_of(layout, bt);
        }
        const int RA = 1 << RB;
        for (int k = 0; k < RA; ++k) {
            if (((uint32_t)k & reg_c) == reg_c) o.km_c |= 1ull << k;
            if ((uint32_t)k & reg_t) o.km_t |= 1ull << k;
        }
        o.plain = (reg_c == 0 && o.thr_c == 0 && o.out_c == 0) ? 1 : 0;
        ops.push_back(o);
    }

    // one SK_RAMP: amplitudes with qubit q at 1 times the product of the phases
    // of the pairs (q, m) whose local qubit m is 1 (see SK_RAMP)
    void emit_ramp(const Pass &ps, int q, const std::vector<std::pair<int, const SGate *>> &pairs, int layout)
    {
        // the records stay inside one chunk of kOpChunk ops
        const int RA = 1 << RB, nrec = ramp_records(RA);
        while ((ops.size() - pass_start) % kOpChunk > (size_t)(kOpChunk - nrec)) {
            StOp<R> nop;
            memset(&nop, 0, sizeof nop);
            nop.kind = SK_NOP;
            ops.push_back(nop);
            ++filler;
        }
        // per-bit factors: register bit j, thread bit i (products of repeated pairs)
        std::complex<double> freg[8], fthr[kThrBits];
        for (auto &f : freg) f = 1.0;
        for (auto &f : fthr) f = 1.0;
        for (const auto &pm : pairs) {
            const int b = local_of(ps, pm.first);
            const int j = reg_of(layout, b);
            const std::complex<double> ph(pm.second->m[6], pm.second->m[7]);
            if (j >= 0) freg[j] *= ph;
            else fthr[thr_of(layout, b)] *= ph;
        }
        // the tables (see SK_RAMP), each entry one FP64 product rounded once
        std::vector<std::complex<double>> tab(4 * nrec, 1.0);
        for (int k = 0; k < RA; ++k)
            for (int j = 0; j < RB; ++j)
                if ((k >> j) & 1) tab[k] *= freg[j];
        for (int x = 0; x < 16; ++x)
            for (int i = 0; i < 4; ++i)
                if ((x >> i) & 1) {
                    tab[RA + x] *= fthr[i];
                    tab[RA + 16 + x] *= fthr[4 + i];
                }
        std::vector<StOp<R>> rec(nrec);
        memset(rec.data(), 0, sizeof(StOp<R>) * nrec);
        rec[0].kind = SK_RAMP;
        const int bq = local_of(ps, q);
        uint32_t reg_t = 0;
        if (bq < 0) rec[0].out_t = 1ull << q;
        else if (reg_of(layout, bq) >= 0) reg_t = 1u << reg_of(layout, bq);
        else rec[0].thr_t = 1u << thr_of(layout, bq);
        for (int k = 0; k < RA; ++k)
            if ((uint32_t)k & reg_t) rec[0].km_t |= 1ull << k;
        for (int e = 0; e < 4 * nrec; ++e) {
            rec[e >> 2].m[2 * (e & 3)] = (R)tab[e].real();
            rec[e >> 2].m[2 * (e & 3) + 1] = (R)tab[e].imag();
        }
        for (int r = 1; r < nrec; ++r) rec[r].kind = SK_NOP;
        filler += (size_t)(nrec - 1);
        for (int r = 0; r < nrec; ++r) ops.push_back(rec[r]);
    }

    void emit_layout(int l)
    {
        ++layout_changes;
        StOp<R> o;
        memset(&o, 0, sizeof o);
        o.kind = SK_LAYOUT;
        o.arg = l;
        ops.push_back(o);
    }

    // order the pass's gates (respecting non-commuting pairs) so that
    // consecutive exchange gates share a layout; returns the op count
    int schedule(const Pass &ps, const std::vector<SGate> &g)
    {
        const size_t P = ps.members.size();
        const size_t start = ops.size();
        pass_start = start;
        std::vector<int> indeg(P, 0);
        std::vector<std::vector<int>> succ(P);
        for (size_t a = 0; a < P; ++a)
            for (size_t b = a + 1; b < P; ++b)
                if (!commute(g[ps.members[a]], g[ps.members[b]])) {
                    succ[a].push_back((int)b);
                    indeg[b]++;
                }
        std::vector<char> emitted(P, 0);
        const int NL = n_layouts(M, RB);
        int layout = 0;
        size_t left = P;
        auto fits = [&](int i, int l) {
            const SGate &s = g[ps.members[i]];
            if (!s.xq()) return true;
            return reg_of(l, local_of(ps, s.target)) >= 0;
        };
        while (left) {
            // controlled phases wait while any other gate can run: the gates
            // that run first free more phases to join one ramp
            int pick = -1;
            for (size_t i = 0; i < P && pick < 0 && allow_ramps; ++i)
                if (!emitted[i] && indeg[i] == 0 && !ramp_candidate(g[ps.members[i]]) && fits((int)i, layout))
                    pick = (int)i;
            for (size_t i = 0; i < P && pick < 0; ++i)
                if (!emitted[i] && indeg[i] == 0 && fits((int)i, layout)) pick = (int)i;
            if (pick < 0) {
                int best = -1, bestc = -1;
                for (int l = 0; l < NL; ++l) {
                    if (l == layout) continue;
                    int c = 0;
                    for (size_t i = 0; i < P; ++i)
                        if (!emitted[i] && indeg[i] == 0 && fits((int)i, l)) ++c;
                    if (c > bestc) { bestc = c; best = l; }
                }
                emit_layout(best);
                layout = best;
                continue;
            }
            auto mark = [&](int i) {
                order.push_back(g[ps.members[i]].orig);
                emitted[i] = 1;
                --left;
                for (int s2 : succ[i]) indeg[s2]--;
            };
            if (allow_ramps && ramp_candidate(g[ps.members[pick]])) {
                // every controlled phase that could run now and shares a qubit
                // with this one goes into one ramp over the qubit they share
                // most (the partner qubit must be inside the tile)
                const SGate &a = g[ps.members[pick]];
                const int qa = a.target, qb = __builtin_ctzll(a.ctrl);
                auto partner = [&](const SGate &c, int q) {
                    const int t = c.target, u = __builtin_ctzll(c.ctrl);
                    return t == q ? u : (u == q ? t : -1);
                };
                std::vector<int> cand;
                for (size_t i = 0; i < P; ++i)
                    if (!emitted[i] && indeg[i] == 0 && ramp_candidate(g[ps.members[i]])) cand.push_back((int)i);
                int best_q = -1;
                size_t best = 0;
                for (int q : {qa, qb}) {
                    size_t c = 0;
                    for (int i : cand) {
                        const int m = partner(g[ps.members[i]], q);
                        if (m >= 0 && local_of(ps, m) >= 0) ++c;
                    }
                    if (c > best) { best = c; best_q = q; }
                }
                if (best >= 3) {
                    std::vector<std::pair<int, const SGate *>> pairs;
                    std::vector<int> used;
                    for (int i : cand) {
                        const int m = partner(g[ps.members[i]], best_q);
                        if (m >= 0 && local_of(ps, m) >= 0) {
                            pairs.push_back({m, &g[ps.members[i]]});
                            used.push_back(i);
                        }
                    }
                    emit_ramp(ps, best_q, pairs, layout);
                    for (int i : used) mark(i);
                    continue;
                }
            }
            emit_gate(ps, g[ps.members[pick]], layout);
            mark(pick);
        }
        if (layout != 0) emit_layout(0);
        return (int)(ops.size() - start);
    }
};

}  // namespace
}  // namespace qsim
