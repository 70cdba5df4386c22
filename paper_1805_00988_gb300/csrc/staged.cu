// staged.cu -- multi-gate tile passes: one HBM read + write of the state
// applies a whole run of gates.
//
// Algorithm 1 (§2.3) touches the full state once per gate.  Consecutive gates
// whose non-diagonal qubits all lie in one qubit set Q can instead be applied
// tile by tile: a tile is the 2^M amplitudes that share the bits of every
// qubit outside Q, so a gate on a qubit of Q only pairs amplitudes inside one
// tile.  Q always holds the low qubits 0..4 (so a tile is made of contiguous
// 32-amplitude chunks) plus M - 5 further qubits chosen per pass.  Diagonal
// gates (Z, S, T, P, RZ, CZ, CP, ...) and controls never need their qubit in
// Q: outside Q the bit is constant over the tile.
//
// Inside a CTA the tile lives in registers: with 128 threads each thread holds
// 2^(M-7) amplitudes.  A register layout assigns the tile's local bits to
// register bits and thread bits; a gate whose target is a register bit is
// applied by each thread alone.  Layouts change through shared memory (one
// store + one load of the tile, padded so the layouts are free of bank
// conflicts).  The host planner forms the passes (tile.cuh); the gates of a
// pass are ordered and compiled into a tile program (tileprog.cuh), which the
// kernel below runs.
#include <algorithm>
#include <cstring>
#include <vector>

#include "tileprog.cuh"

namespace qsim {

namespace {

template <typename R, int M, bool kFull>
__global__ void __launch_bounds__(kTpThr, (tile_ctas<R, M>()))
    k_staged(R *__restrict__ st, const uint4 *__restrict__ prog, int nunits, TileGeom geo, int start_layout,
             int end_layout, uint64_t flip)
{
    constexpr int VEC = (sizeof(R) == 4) ? 2 : 1;
    constexpr int RB = M - kTpThrBits;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *sm = reinterpret_cast<R *>(smem_raw);
    uint4 *sp = reinterpret_cast<uint4 *>(smem_raw + (size_t)tile_slots<M, RB, VEC>() * 2 * sizeof(R));
    const int tid = threadIdx.x;
    const uint32_t tile = blockIdx.x;

    prog_stage(prog, nunits, tid, sp);
    uint64_t base = tile_base(geo, tile);
    Amps<R, (1 << RB)> v;
    tile_load<M, RB, VEC, false>(start_layout, v, st, geo, tid, base);
    __syncthreads();
    run_program<R, M, kFull>(v, prog, nunits, tile, tid, sm, sp);
    // addresses are formed again from inputs the compiler cannot prove equal,
    // instead of being held live across the program
    int t2 = tid;
    asm volatile("" : "+r"(t2), "+l"(base));
    tile_store<M, RB, VEC, false>(end_layout, v, st, geo, t2, base, flip);
}

template <typename R, int M, bool kFull>
int launch_staged_v(qsim_state *s, const uint4 *prog, int nunits, const TileGeom &geo, const TilePass &tp, double flops)
{
    const size_t smem = tile_smem_bytes<R, M>();
    // set on every launch: the attribute belongs to the current device's
    // context, and the call costs a microsecond against a multi-ms pass
    QSIM_CUDA(cudaFuncSetAttribute(k_staged<R, M, kFull>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const uint64_t tiles = 1ull << (s->n - M);
    launch_begin(s, KC_STAGED, 2.0 * (double)s->bytes, flops);
    k_staged<R, M, kFull><<<(unsigned)tiles, kTpThr, smem, s->stream>>>((R *)s->amps, prog, nunits, geo,
                                                                        tp.start_layout, tp.end_layout, tp.flip);
    return launch_end(s, "staged pass");
}

template <typename R, int M>
int launch_staged(qsim_state *s, const uint4 *prog, int nunits, const TileGeom &geo, const TilePass &tp, double flops)
{
    // complex128 passes are bound by the FP64 pipe: one variant is enough
    if (sizeof(R) == 4 && tp.groups_only()) {
        if constexpr (sizeof(R) == 4) return launch_staged_v<R, M, false>(s, prog, nunits, geo, tp, flops);
    }
    return launch_staged_v<R, M, true>(s, prog, nunits, geo, tp, flops);
}

// Programs are planned, copied and launched one pass at a time, so the host
// plans the next pass while the GPU runs this one (a 20-qubit random circuit
// spent 0.45 ms planning before 0.27 ms of kernels).  They go through one
// pinned buffer, each at its own place; when it is full the stream is waited
// for and the buffer starts again.
constexpr size_t kProgBuffer = (size_t)1 << 18;

template <typename R, int M>
int run_staged(qsim_state *s, const std::vector<SGate> &g)
{
    const int VEC = sizeof(R) == 4 ? 2 : 1;
    TilePlanner<R> plan(g, s->n, M, VEC);
    Program p;
    size_t off = 0;
    int rc = SIM_OK;
    while (rc == SIM_OK && plan.next(&p)) {
        const size_t bytes = p.words.size() * 4;
        if (off + bytes > s->host_ops_bytes || off + bytes > s->dev_ops_bytes) {
            if (off) QSIM_CUDA(cudaStreamSynchronize(s->stream));
            off = 0;
            const size_t need = std::max(kProgBuffer, 2 * bytes);
            if ((rc = ensure_host_pinned(&s->host_ops, &s->host_ops_bytes, need))) break;
            if ((rc = ensure_device(s, &s->dev_ops, &s->dev_ops_bytes, need))) break;
        }
        memcpy((char *)s->host_ops + off, p.words.data(), bytes);
        uint4 *prog = (uint4 *)((char *)s->dev_ops + off);
        if (cudaMemcpyAsync(prog, (char *)s->host_ops + off, bytes, cudaMemcpyHostToDevice, s->stream) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "tile program upload");
            break;
        }
        double f = 0.0;
        for (int m : p.members) f += sgate_flops(g[(size_t)m], s->n);
        rc = launch_staged<R, M>(s, prog, (int)(p.words.size() / 4), tile_geom(p.pass, s->n), p.tp, f);
        off += (bytes + 255) & ~(size_t)255;
    }
    // the pinned buffer is reused by the next call: wait for the copies
    const cudaError_t e = cudaStreamSynchronize(s->stream);
    if (rc == SIM_OK && e != cudaSuccess) rc = cuda_fail(e, "staged plan");
    return rc;
}

template <typename R>
int run_staged(qsim_state *s, const std::vector<SGate> &g, int M)
{
    if (M == 11) return run_staged<R, 11>(s, g);
    if (M == 12) return run_staged<R, 12>(s, g);
    if constexpr (sizeof(R) == 4) return run_staged<R, 13>(s, g);
    return fail(SIM_EINVAL, "staged: complex128 tiles are at most 12 qubits");
}

}  // namespace

double tile_cost(const std::vector<SGate> &g, int n, int dtype)
{
    double t = 0.0;
    Program p;
    if (dtype == SIM_C128) {
        TilePlanner<double> plan(g, n, 12, 1, false, false);
        while (plan.next(&p)) t += pass_cost<double>(p.tp);
    } else {
        TilePlanner<float> plan(g, n, 13, 2, false, false);
        while (plan.next(&p)) t += pass_cost<float>(p.tp);
    }
    return t;
}

// The tile size when the caller leaves it open.  Small tiles give small
// registers more CTAs and shorter programs: 14 qubits, depth-20 random circuit
// 274 / 307 / 338 us with 11- / 12- / 13-qubit tiles, 18 qubits 385 / 418 / 456, 20
// qubits 440 / 458 / 500; 22 qubits 839 / 798 / 858.  From 23 on 13: it saves passes that HBM bounds
// (28 qubits, Haar layers 13.1 / 12.4 ms with 12 / 13, reversible 6.8 / 6.0), which
// at 23 to 25 is worth nothing yet (the two are within 6 % on Haar layers, QFTs, ladders and reversible
// circuits there, phases take 223 / 300 us at 24; the learned plan takes 12 up to 25).
// 12 where controlled gates other than moves, or doubly controlled phases, are more than an eighth:
// each costs every amplitude a masked multiply, dearer with 64 amplitudes a thread (random gates, 24
// qubits 0.81 / 1.13 ms, 27 7.1 / 9.4, 28 14.0 / 18.2; 1.06, 8.2 and 16.5 before tile programs).
// complex128: 12 qubits wherever they fit (26-qubit QFT 24.3 against 25.3 ms).
static int open_tile(const std::vector<SGate> &g, int n, bool c128)
{
    if (c128) return n >= 20 ? 12 : 11;
    if (n <= 22) return n <= 18 ? 11 : 12;
    size_t masked = 0;
    for (const SGate &x : g)
        masked += x.xq() ? x.ctrl && x.op != OP_XPERM && x.op != OP_SWAP : __builtin_popcountll(x.ctrl) >= 2;
    return 8 * masked > g.size() ? 12 : 13;
}

int run_tiles(qsim_state *s, const std::vector<SGate> &g)
{
    const int M = open_tile(g, s->n, s->dtype == SIM_C128);
    return s->dtype == SIM_C128 ? run_staged<double>(s, g, M) : run_staged<float>(s, g, M);
}

int64_t tile_passes(const std::vector<SGate> &g, int n, int dtype, int tile_qubits)
{
    const bool c128 = dtype == SIM_C128;
    const int M = tile_qubits ? tile_qubits : open_tile(g, n, c128);
    int64_t count = 0;
    Program p;
    if (c128) {
        TilePlanner<double> plan(g, n, M, 1, false, false);
        while (plan.next(&p)) ++count;
    } else {
        TilePlanner<float> plan(g, n, M, 2, false, false);
        while (plan.next(&p)) ++count;
    }
    return count;
}

int describe_staged(int n, int dtype, const sim_gate *gates, size_t n_gates, int tile_qubits, int64_t *passes,
                    int64_t *ops, int64_t *layout_changes, int32_t *order, size_t order_cap, size_t *order_len)
{
    const bool c128 = dtype == SIM_C128;
    std::vector<SGate> g;
    int M = tile_qubits;
    if (!M) {
        lower_renamed(gates, n_gates, n, &g);     // as a run has them
        M = open_tile(g, n, c128);
        g.clear();
    }
    if (M > n || M < 11 || M > (c128 ? 12 : 13)) return fail(SIM_EINVAL, "describe: no staged tile fits");
    lower_gates(gates, n_gates, &g);
    std::vector<Pass> ps = form_passes(g, n, M);
    PlanBuilder<double> pb{n, M, M - kThrBits, c128 ? 1 : 2, {}, {}, 0};
    for (const Pass &p : ps) pb.schedule(p, g);
    if (passes) *passes = (int64_t)ps.size();
    if (ops) *ops = (int64_t)(pb.ops.size() - pb.filler);   // a phase ramp counts once
    if (layout_changes) *layout_changes = pb.layout_changes;
    if (order_len) *order_len = pb.order.size();
    if (order)
        for (size_t i = 0; i < pb.order.size() && i < order_cap; ++i) order[i] = pb.order[i];
    return SIM_OK;
}

int encode_staged(int n, int dtype, const sim_gate *gates, size_t n_gates, int tile_qubits, sim_tile_op *ops,
                  size_t ops_cap, int32_t *info, size_t info_cap, size_t *n_ops, size_t *n_passes)
{
    const bool c128 = dtype == SIM_C128;
    std::vector<SGate> g;
    int M = tile_qubits;
    if (!M) {
        lower_renamed(gates, n_gates, n, &g);     // as a run has them
        M = open_tile(g, n, c128);
        g.clear();
    }
    if (M > n || M < 11 || M > (c128 ? 12 : 13)) return fail(SIM_EINVAL, "encode: no staged tile fits");
    lower_gates(gates, n_gates, &g);
    std::vector<Pass> ps = form_passes(g, n, M);
    PlanBuilder<double> pb{n, M, M - kThrBits, c128 ? 1 : 2, {}, {}, 0};
    std::vector<size_t> first;
    for (const Pass &p : ps) {
        first.push_back(pb.ops.size());
        pb.schedule(p, g);
    }
    if (n_ops) *n_ops = pb.ops.size();
    if (n_passes) *n_passes = ps.size();
    for (size_t k = 0; k < pb.ops.size() && k < ops_cap && ops; ++k) {
        const StOp<double> &o = pb.ops[k];
        sim_tile_op &t = ops[k];
        t.kind = o.kind;
        t.arg = o.arg;
        t.thr_c = o.thr_c;
        t.plain = o.plain;
        t.out_c = o.out_c;
        t.km_c = o.km_c;
        t.km_t = o.km_t;
        t.thr_t = o.thr_t;
        t.pad = 0;
        t.out_t = o.out_t;
        for (int j = 0; j < 8; ++j) t.m[j] = o.m[j];
    }
    for (size_t p = 0; p < ps.size() && info && (p + 1) * SIM_TILE_PASS_INFO <= info_cap; ++p) {
        int32_t *r = info + p * SIM_TILE_PASS_INFO;
        for (int j = 0; j < SIM_TILE_PASS_INFO; ++j) r[j] = 0;
        r[0] = (int32_t)first[p];
        r[1] = (int32_t)((p + 1 < ps.size() ? first[p + 1] : pb.ops.size()) - first[p]);
        r[2] = M;
        r[3] = M - kThrBits;
        r[4] = c128 ? 1 : 2;
        r[5] = (int32_t)ps[p].high.size();
        for (size_t i = 0; i < ps[p].high.size() && i < 16; ++i) r[6 + i] = ps[p].high[i];
    }
    return SIM_OK;
}

int export_tile_programs(int n, int dtype, const sim_gate *gates, size_t n_gates, int tile_qubits, uint32_t *words,
                         size_t words_cap, int32_t *info, size_t info_cap, size_t *n_words, size_t *n_passes)
{
    const bool c128 = dtype == SIM_C128;
    std::vector<SGate> g;
    lower_renamed(gates, n_gates, n, &g);
    int M = tile_qubits ? tile_qubits : open_tile(g, n, c128);
    if (M > n || M < 11 || M > (c128 ? 12 : 13)) return fail(SIM_EINVAL, "tile programs: no staged tile fits");
    const std::vector<Program> ps = compile_passes<double>(g, n, M, c128 ? 1 : 2);
    size_t at = 0;
    for (size_t p = 0; p < ps.size(); ++p) {
        for (size_t k = 0; words && k < ps[p].words.size() && at + k < words_cap; ++k) words[at + k] = ps[p].words[k];
        if (info && (p + 1) * SIM_TILE_PASS_INFO <= info_cap) {
            int32_t *r = info + p * SIM_TILE_PASS_INFO;
            for (int j = 0; j < SIM_TILE_PASS_INFO; ++j) r[j] = 0;
            const uint64_t flip = ps[p].tp.flip;
            const std::vector<int> &high = ps[p].pass.high;
            const int32_t v[10] = {(int32_t)at, (int32_t)ps[p].words.size(), M, M - kTpThrBits, c128 ? 1 : 2,
                                   ps[p].tp.start_layout, ps[p].tp.end_layout, (int32_t)(uint32_t)flip,
                                   (int32_t)(uint32_t)(flip >> 32), (int32_t)high.size()};
            for (int j = 0; j < 10; ++j) r[j] = v[j];
            for (size_t i = 0; i < high.size() && i < 14; ++i) r[10 + i] = high[i];
        }
        at += ps[p].words.size();
    }
    if (n_words) *n_words = at;
    if (n_passes) *n_passes = ps.size();
    return SIM_OK;
}

int apply_circuit_staged(qsim_state *s, const sim_gate *gates, size_t n_gates, const sim_plan_opts &o)
{
    const bool c128 = s->dtype == SIM_C128;
    std::vector<SGate> g;
    if (s->n >= 11) lower_renamed(gates, n_gates, s->n, &g);
    int M = o.tile_qubits ? o.tile_qubits : open_tile(g, s->n, c128);
    if (M > s->n) M = (s->n >= 11) ? 11 : 0;
    if (c128 && M > 12) M = 12;
    if (M != 0 && (M < 11 || M > 13)) return fail(SIM_EINVAL, "staged: tile_qubits must be 11, 12 or 13");
    if (M == 0) {
        // the state is smaller than a tile: one launch per gate
        for (size_t k = 0; k < n_gates; ++k)
            if (int rc = launch_pair_gate(s, make_pair_gate(gates[k]))) return rc;
        return SIM_OK;
    }
    if (g.empty()) return SIM_OK;
    return c128 ? run_staged<double>(s, g, M) : run_staged<float>(s, g, M);
}

}  // namespace qsim
