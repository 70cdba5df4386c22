// tileprog.cuh -- tile programs: what a register-tile pass executes.
//
// The planner (tile.cuh) decides which gates a pass holds, in which order and
// under which register layouts.  Before the launch the host compiles that
// order into a short program of the operations below; the kernels
// (k_staged, k_batch) run the program on the 2^M amplitudes of each tile.
//
// What the compilation buys.  A dense 2 x 2 gate costs 8 fused multiply-adds
// per amplitude.  Every unitary 2 x 2 is diag * R * diag with a real rotation
// R = [[1, -t], [t, 1]] / sqrt(1 + t^2), |t| <= 1 (rows swapped if needed),
// and R is diag(1, 1 + t^2) times two real shears
//     lo += a * hi;   hi += b * lo;        a = -t, b = t / (1 + t^2),
// which run in place: 2 multiply-adds per amplitude, no temporary, no move.
// The diagonal factors (phases, the scale, CZ, CP, RZ, ...) commute with
// everything that does not touch their qubits non-diagonally, so the host
// keeps them in a pool (DiagPool) across gates, layouts and passes, and only
// when a rotation needs them they are applied -- all at once, as one table
// multiply of the thread's registers (TP_CDIAG / TP_RDIAG), as sign bits
// carried by the thread (TP_Z) or as a phase ramp (TP_RAMP).  Row swaps and X
// gates only relabel a qubit (flip); the final store applies the labels
// through its addresses.
//
// Precision: two roundings per gate and amplitude instead of four, plus one
// complex multiply per merged diagonal; tables and shears are formed in FP64
// on the host and rounded once.
//
// Range.  The amplitudes in memory are the state without the pending factors,
// so those must stay where FP32 tables and FP32 amplitudes hold them: the
// common factor is applied when it leaves 2^-8..2^8; a rotation leaves a factor
// of modulus 1/4..4 on its qubit, which the next one takes; pairs have modulus
// one; and a gate whose own factors are not of modulus one (a contraction, say) is
// kept aside only while all moduli pending stay within kPoolBits bits together,
// otherwise applied where it stands.
#pragma once

#include <cmath>
#include <complex>
#include <cstring>
#include <vector>

#include "f32x2.cuh"
#include "tile.cuh"

namespace qsim {
namespace {

// A program is a stream of 16-byte units.  Word x of an operation's header:
// bits 0..3 the operation, 4..11 its length in units, 12.. its arguments.
enum TileOp {
    TP_END = 0,     // program done
    TP_CHUNK,       // continue in the next staged chunk
    TP_GROUP,       // in this order, each optional: sign entries, one diagonal, shears, FLUSH of the signs, a
                    // change of layout.  x: 12..14 diagonal (GroupDiag), 15..17 its register bit, 18..23 register
                    // bits of the shears, 24..28 number of sign entries, 29 shears under pending signs, 30 flush;
                    // 31 change of
                    // layout (y: from | to << 2).  Then the sign entries (two a unit: x =
                    // thread condition | sign bits << 16 (bit j: Z on register bit j, bit 6: the whole thread), y =
                    // tile condition), the factors, the shears' (a, b) per register bit.
    TP_RAMP,        // x: 12..14 centre register bit (7: registers in unit 1), 15 register table, 16 thread tables,
                    // 17..22 outer tables; y: thread condition, z: tile condition; unit 2..: the tables
    TP_XCH,         // x: 12..14 register bit, 15..16 kind; y, z: conditions; unit 1: registers; unit 2..: matrix
    TP_PH,          // y, z: conditions, w: the target's place (0: a register bit); unit 1: registers, target
                    // registers; unit 2: thread and tile condition of the target; unit 3..: factors for 0 and 1
    TP_CSHEARS,     // x: 12..14 register bit; unit 1..: complex a, b
    TP_PERM         // a change of layout that also permutes the tile's bits.  x: 12..15 from | to << 2; unit 1..: the
                    // slot weight of the source bit of each thread bit, then of each register bit
};
enum GroupDiag {
    GD_NONE = 0,
    GD_REAL,        // real factor per register
    GD_CPLX,        // complex factor per register
    GD_HALF         // one phase e^{i phi}, |phi| <= pi / 2, for the registers with the bit set: a = -tan(phi / 2), b = sin phi
};

// A tile program runs on 128 threads, each holding 2^(M - 7) amplitudes (64
// of a 13-qubit tile).  With 256 threads of half as many, every operation's
// decoding was paid for half the arithmetic and windows of five instead of
// six register bits took more groups and changes of layout: 203 against 189 ms
// for the 30-qubit depth-20 circuit.
constexpr int kTpThr = 128;
constexpr int kTpThrBits = 7;
constexpr double kCostLayout = 7.0, kCostGroup = 1.5;   // see schedule_pass
constexpr int kChunkUnits = 512;      // 16-byte units of a staged chunk (8 KB of shared memory)
constexpr int kThrTab = 24;           // thread table of a ramp: 16 entries for thread bits 0..3, 8 for bits 4..6
constexpr int kOutGroup = 4;          // outer qubits per table of a ramp
constexpr int kOutGroups = 6;         // 4 x 6 >= 34 - 11 outer qubits

// A thread condition packs a mask and a value: (tid & mask) == value.
__host__ __device__ constexpr uint32_t thr_cond(uint32_t mask, uint32_t val) { return mask | (val << 8); }

// ---------------------------------------------------------------- device
template <typename R> struct V2;
template <> struct V2<float> { using T = float2; };
template <> struct V2<double> { using T = double2; };

// A thread's amplitudes.  complex64 keeps real and imaginary parts in packs
// along register bit 0, so that one packed FP32x2 instruction (fma.rn.f32x2)
// works on two amplitudes and a complex multiply needs neither swaps nor
// moves.  A pack is one 64-bit value for the compiler: as float2 its halves
// were carried separately from one operation to the next, and the moves that
// paired them up again were a third of all instructions.  complex128 keeps
// plain doubles.
template <typename R, int RA> struct Amps;
template <int RA> struct Amps<float, RA> {
    pack2 r[RA / 2], i[RA / 2];
    __device__ __forceinline__ float re(int k) const
    {
        const float2 t = unpk(r[k >> 1]);
        return (k & 1) ? t.y : t.x;
    }
    __device__ __forceinline__ float im(int k) const
    {
        const float2 t = unpk(i[k >> 1]);
        return (k & 1) ? t.y : t.x;
    }
    __device__ __forceinline__ void set(int k, float a, float b)
    {
        const float2 t = unpk(r[k >> 1]), u = unpk(i[k >> 1]);
        r[k >> 1] = (k & 1) ? pk(t.x, a) : pk(a, t.y);
        i[k >> 1] = (k & 1) ? pk(u.x, b) : pk(b, u.y);
    }
};
template <int RA> struct Amps<double, RA> {
    double r[RA], i[RA];
    __device__ __forceinline__ double re(int k) const { return r[k]; }
    __device__ __forceinline__ double im(int k) const { return i[k]; }
    __device__ __forceinline__ void set(int k, double a, double b)
    {
        r[k] = a;
        i[k] = b;
    }
};

template <typename T, typename R>
__device__ __forceinline__ void cmul(T &v, R gr, R gi)
{
    const R t = gi * v.y, u = gi * v.x;
    v.x = gr * v.x - t;
    v.y = gr * v.y + u;
}
template <typename R, int RA>
__device__ __forceinline__ void cmul_at(Amps<R, RA> &v, int k, R gr, R gi)
{
    const R x = v.re(k), y = v.im(k);
    v.set(k, gr * x - gi * y, gr * y + gi * x);
}
// x negated when bit 31 of s is set (other bits of s are 0)
__device__ __forceinline__ float flip_sign(float x, uint32_t s) { return __uint_as_float(__float_as_uint(x) ^ s); }
__device__ __forceinline__ double flip_sign(double x, uint32_t s)
{
    return __hiloint2double((int)((uint32_t)__double2hiint(x) ^ s), __double2loint(x));
}

// shared-memory slot of local index x.  The padding is additive over disjoint
// bits, so a register's slot is the thread's slot plus a constant (an
// immediate offset), and the layouts are free of bank conflicts (checked on
// the CPU for every tile size and layout; only the top window of 11-qubit
// complex64 tiles has two-way ones).  complex64: a plane of real and a plane
// of imaginary parts, 4-byte accesses, 8-byte ones (a whole pack) in layout
// 0; complex128: 16-byte amplitudes.
template <int RB, int VEC>
__host__ __device__ constexpr int slot_of(int x)
{
    return (VEC == 2) ? x + ((x >> (RB + 1)) << 1) : x + (x >> RB);
}
template <int M, int RB, int VEC>
__host__ __device__ constexpr int tile_slots() { return slot_of<RB, VEC>((1 << M) - 1) + 1; }

// thread bit i starts a run of thread bits whose slots double from bit to bit;
// its length
template <int M, int RB, int VEC, int L>
__host__ __device__ constexpr int slot_run(int i)
{
    auto w = [](int j) { return slot_of<RB, VEC>(1 << thr_local(M, RB, VEC, L, j)); };
    if (i > 0 && w(i) == 2 * w(i - 1)) return 0;
    int n = 1;
    while (i + n < kTpThrBits && w(i + n) == 2 * w(i + n - 1)) ++n;
    return n;
}
template <int M, int RB, int VEC, int L, int I = 0>
__device__ __forceinline__ int thr_slot(int tid)
{
    if constexpr (I < kTpThrBits) {
        constexpr int n = slot_run<M, RB, VEC, L>(I);
        constexpr int w = slot_of<RB, VEC>(1 << thr_local(M, RB, VEC, L, I));
        const int rest = thr_slot<M, RB, VEC, L, I + 1>(tid);
        if constexpr (n > 0) return rest + ((tid >> I) & ((1 << n) - 1)) * w;
        else return rest;
    } else {
        return 0;
    }
}

template <int M, int RB, int VEC, int L, int RA>
__device__ __forceinline__ void store_layout(const Amps<float, RA> &v, float *sm, int tid)
{
    if constexpr (L < n_layouts(M, RB)) {
        float *p = sm + thr_slot<M, RB, VEC, L>(tid);
        constexpr int PLANE = tile_slots<M, RB, VEC>();
        if constexpr (L == 0) {
#pragma unroll
            for (int k = 0; k < RA; k += 2) {
                float *q = p + slot_of<RB, VEC>(reg_part(M, RB, VEC, L, k));
                *reinterpret_cast<pack2 *>(q) = v.r[k >> 1];
                *reinterpret_cast<pack2 *>(q + PLANE) = v.i[k >> 1];
            }
        } else {
#pragma unroll
            for (int k = 0; k < RA; ++k) {
                float *q = p + slot_of<RB, VEC>(reg_part(M, RB, VEC, L, k));
                q[0] = v.re(k);
                q[PLANE] = v.im(k);
            }
        }
    }
}
template <int M, int RB, int VEC, int L, int RA>
__device__ __forceinline__ void load_layout(Amps<float, RA> &v, const float *sm, int tid)
{
    if constexpr (L < n_layouts(M, RB)) {
        const float *p = sm + thr_slot<M, RB, VEC, L>(tid);
        constexpr int PLANE = tile_slots<M, RB, VEC>();
        if constexpr (L == 0) {
#pragma unroll
            for (int k = 0; k < RA; k += 2) {
                const float *q = p + slot_of<RB, VEC>(reg_part(M, RB, VEC, L, k));
                v.r[k >> 1] = *reinterpret_cast<const pack2 *>(q);
                v.i[k >> 1] = *reinterpret_cast<const pack2 *>(q + PLANE);
            }
        } else {
#pragma unroll
            for (int k = 0; k < RA; k += 2) {
                const float *q0 = p + slot_of<RB, VEC>(reg_part(M, RB, VEC, L, k));
                const float *q1 = p + slot_of<RB, VEC>(reg_part(M, RB, VEC, L, k + 1));
                v.r[k >> 1] = pk(q0[0], q1[0]);
                v.i[k >> 1] = pk(q0[PLANE], q1[PLANE]);
            }
        }
    }
}
template <int M, int RB, int VEC, int L, int RA>
__device__ __forceinline__ void store_layout(const Amps<double, RA> &v, double *sm, int tid)
{
    if constexpr (L < n_layouts(M, RB)) {
        double *p = sm + 2 * thr_slot<M, RB, VEC, L>(tid);
#pragma unroll
        for (int k = 0; k < RA; ++k)
            *reinterpret_cast<double2 *>(p + 2 * slot_of<RB, VEC>(reg_part(M, RB, VEC, L, k))) =
                make_double2(v.r[k], v.i[k]);
    }
}
template <int M, int RB, int VEC, int L, int RA>
__device__ __forceinline__ void load_layout(Amps<double, RA> &v, const double *sm, int tid)
{
    if constexpr (L < n_layouts(M, RB)) {
        const double *p = sm + 2 * thr_slot<M, RB, VEC, L>(tid);
#pragma unroll
        for (int k = 0; k < RA; ++k) {
            const double2 t = *reinterpret_cast<const double2 *>(p + 2 * slot_of<RB, VEC>(reg_part(M, RB, VEC, L, k)));
            v.set(k, t.x, t.y);
        }
    }
}

template <int M, int RB, int VEC, typename R, int RA>
__device__ __forceinline__ void relayout(int from, int to, Amps<R, RA> &v, R *sm, int tid)
{
    __syncthreads();
    switch (from) {
    case 0: store_layout<M, RB, VEC, 0>(v, sm, tid); break;
    case 1: store_layout<M, RB, VEC, 1>(v, sm, tid); break;
    case 2: store_layout<M, RB, VEC, 2>(v, sm, tid); break;
    default: store_layout<M, RB, VEC, 3>(v, sm, tid); break;
    }
    __syncthreads();
    switch (to) {
    case 0: load_layout<M, RB, VEC, 0>(v, sm, tid); break;
    case 1: load_layout<M, RB, VEC, 1>(v, sm, tid); break;
    case 2: load_layout<M, RB, VEC, 2>(v, sm, tid); break;
    default: load_layout<M, RB, VEC, 3>(v, sm, tid); break;
    }
}

// a change of layout by slot weights: thread bits, then register bits
template <int M, int RB, int VEC, typename R, int RA>
__device__ __forceinline__ void permute(int from, Amps<R, RA> &v, R *sm, int tid, const int *w)
{
    __syncthreads();
    switch (from) {
    case 0: store_layout<M, RB, VEC, 0>(v, sm, tid); break;
    case 1: store_layout<M, RB, VEC, 1>(v, sm, tid); break;
    case 2: store_layout<M, RB, VEC, 2>(v, sm, tid); break;
    default: store_layout<M, RB, VEC, 3>(v, sm, tid); break;
    }
    __syncthreads();
    constexpr int PLANE = tile_slots<M, RB, VEC>();
    int at = 0;
#pragma unroll
    for (int i = 0; i < kTpThrBits; ++i)
        if ((tid >> i) & 1) at += w[i];
#pragma unroll
    for (int k = 0; k < RA; ++k) {
        int s = at;
#pragma unroll
        for (int j = 0; j < RB; ++j)
            if ((k >> j) & 1) s += w[kTpThrBits + j];
        if constexpr (sizeof(R) == 4) v.set(k, sm[s], sm[s + PLANE]);
        else v.set(k, sm[2 * s], sm[2 * s + 1]);
    }
}

// ---------------------------------------------------------------- tile I/O
// A pass may load and store in any layout whose lanes hold the five low
// qubits (whole 256-byte runs), not only in layout 0; that saves the change
// of layout a pass would otherwise start or end with.  Bit 0 of a complex64
// tile in layout 0 sits in the thread's 16-byte vectors.
__host__ __device__ constexpr bool io_layout(int M, int RB, int VEC, int l)
{
    if (l == 0) return true;
    if (l >= n_layouts(M, RB)) return false;
    for (int i = 0; i < 5; ++i)
        if (thr_local(M, RB, VEC, l, i) != i) return false;
    return true;
}

// global index of the tile's first amplitude: outer bit i of the tile index at
// outer_pos[i], one lane per bit
__device__ __forceinline__ uint64_t tile_base(const TileGeom &geo, uint32_t tile)
{
    const int lane = threadIdx.x & 31;
    uint64_t b = 0;
    if (lane < geo.n_outer) b = (uint64_t)((tile >> lane) & 1u) << geo.outer_pos[lane];
    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)b);
    const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(b >> 32));
    return ((uint64_t)hi << 32) | lo;
}

// f(k, pointer) for every register k (VEC == 2, L == 0: every even k).  The
// pointer of register k is that of k without its lowest bit plus one
// register bit's offset (taken negative when flip exchanges the bit's labels):
// one 64-bit addition each.
template <int M, int RB, int VEC, int L, int K, int J, typename R, typename F>
__device__ __forceinline__ void io_walk(R *p, const int64_t *off, F f)
{
    constexpr int LOWEST = (VEC == 2 && L == 0) ? 1 : 0;
    if constexpr (J < LOWEST) {
        f(K, p);
    } else {
        io_walk<M, RB, VEC, L, K, J - 1>(p, off, f);
        io_walk<M, RB, VEC, L, K | (1 << J), J - 1>(p + off[J], off, f);
    }
}
template <int M, int RB, int VEC, int L, typename R, typename F>
__device__ __forceinline__ void for_io(const TileGeom &geo, int tid, R *st, uint64_t base, uint64_t flip, F f)
{
    auto gbit = [&](int b) { return (b < kLow) ? (1ull << b) : (1ull << geo.hpos[b - kLow]); };
    int64_t off[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) {
        const uint64_t g = gbit(reg_local(M, RB, VEC, L, j));
        off[j] = (flip & g) ? -2 * (int64_t)g : 2 * (int64_t)g;
    }
    uint64_t t = base ^ flip;
    // the five low qubits are thread bits 0.. in order, except bit 0 of layout 0
    constexpr int FIRST = thr_local(M, RB, VEC, L, 0);          // 0 or 1
    t ^= (uint64_t)(tid & ((1 << (kLow - FIRST)) - 1)) << FIRST;
#pragma unroll
    for (int i = kLow - FIRST; i < kTpThrBits; ++i)
        if ((tid >> i) & 1) t ^= gbit(thr_local(M, RB, VEC, L, i));
    io_walk<M, RB, VEC, L, 0, RB - 1>(st + 2 * t, off, f);
}

template <int RA>
__device__ __forceinline__ void put_pair(Amps<float, RA> &v, int k, const float4 &t)
{
    v.r[k >> 1] = pk(t.x, t.z);
    v.i[k >> 1] = pk(t.y, t.w);
}
template <int RA>
__device__ __forceinline__ void put_pair(Amps<double, RA> &, int, const float4 &) {}

template <int M, int RB, int VEC, int L, bool kCg, typename R, int RA>
__device__ __forceinline__ void tile_load_l(Amps<R, RA> &v, const R *st, const TileGeom &geo, int tid, uint64_t base)
{
    if constexpr (io_layout(M, RB, VEC, L)) {
        for_io<M, RB, VEC, L>(geo, tid, st, base, 0ull, [&](int k, const R *q) {
            if constexpr (VEC == 2 && L == 0) {
                const float4 *p = reinterpret_cast<const float4 *>(q);
                const float4 t = kCg ? __ldcg(p) : *p;
                put_pair(v, k, t);
            } else {
                const typename V2<R>::T *p = reinterpret_cast<const typename V2<R>::T *>(q);
                const typename V2<R>::T t = kCg ? __ldcg(p) : *p;
                v.set(k, t.x, t.y);
            }
        });
    }
}

template <int M, int RB, int VEC, int L, bool kCg, typename R, int RA>
__device__ __forceinline__ void tile_store_l(const Amps<R, RA> &v, R *st, const TileGeom &geo, int tid, uint64_t base,
                                             uint64_t flip)
{
    if constexpr (io_layout(M, RB, VEC, L)) {
        // bit 0 of a complex64 tile in layout 0 sits in the vectors
        const uint64_t in_vec = (VEC == 2 && L == 0) ? 1ull : 0ull;
        const bool swap0 = (flip & in_vec) != 0;
        for_io<M, RB, VEC, L>(geo, tid, st, base, flip & ~in_vec, [&](int k, R *q) {
            if constexpr (VEC == 2 && L == 0) {
                float4 *p = reinterpret_cast<float4 *>(q);
                const float4 t = swap0 ? make_float4(v.re(k + 1), v.im(k + 1), v.re(k), v.im(k))
                                       : make_float4(v.re(k), v.im(k), v.re(k + 1), v.im(k + 1));
                if (kCg) __stcg(p, t);
                else *p = t;
            } else {
                typename V2<R>::T *p = reinterpret_cast<typename V2<R>::T *>(q);
                typename V2<R>::T t;
                t.x = v.re(k);
                t.y = v.im(k);
                if (kCg) __stcg(p, t);
                else *p = t;
            }
        });
    }
}

template <int M, int RB, int VEC, bool kCg, typename R, int RA>
__device__ __forceinline__ void tile_load(int layout, Amps<R, RA> &v, const R *st, const TileGeom &geo, int tid,
                                          uint64_t base)
{
    switch (layout) {
    case 0: tile_load_l<M, RB, VEC, 0, kCg>(v, st, geo, tid, base); break;
    case 2: tile_load_l<M, RB, VEC, 2, kCg>(v, st, geo, tid, base); break;
    default: tile_load_l<M, RB, VEC, 3, kCg>(v, st, geo, tid, base); break;
    }
}

// flip: the qubits whose labels are exchanged; register and thread bits of a
// flipped qubit go to the other half of their pairs
template <int M, int RB, int VEC, bool kCg, typename R, int RA>
__device__ __forceinline__ void tile_store(int layout, const Amps<R, RA> &v, R *st, const TileGeom &geo, int tid,
                                           uint64_t base, uint64_t flip)
{
    switch (layout) {
    case 0: tile_store_l<M, RB, VEC, 0, kCg>(v, st, geo, tid, base, flip); break;
    case 2: tile_store_l<M, RB, VEC, 2, kCg>(v, st, geo, tid, base, flip); break;
    default: tile_store_l<M, RB, VEC, 3, kCg>(v, st, geo, tid, base, flip); break;
    }
}

// thread and register bits (of layout l) whose labels are exchanged
template <int M, int RB, int VEC, int L>
__device__ __forceinline__ void flip_bits_l(const TileGeom &geo, uint64_t flip, uint32_t *fthr, uint32_t *freg)
{
    if constexpr (L < n_layouts(M, RB)) {
        auto fl = [&](int b) { return (uint32_t)(flip >> (b < kLow ? b : geo.hpos[b - kLow])) & 1u; };
#pragma unroll
        for (int i = 0; i < kTpThrBits; ++i) *fthr |= fl(thr_local(M, RB, VEC, L, i)) << i;
#pragma unroll
        for (int j = 0; j < RB; ++j) *freg |= fl(reg_local(M, RB, VEC, L, j)) << j;
    }
}
template <int M, int RB, int VEC>
__device__ __forceinline__ void flip_bits(int layout, const TileGeom &geo, uint64_t flip, uint32_t *fthr,
                                          uint32_t *freg)
{
    if (!flip) return;
    switch (layout) {
    case 0: flip_bits_l<M, RB, VEC, 0>(geo, flip, fthr, freg); break;
    case 1: flip_bits_l<M, RB, VEC, 1>(geo, flip, fthr, freg); break;
    case 2: flip_bits_l<M, RB, VEC, 2>(geo, flip, fthr, freg); break;
    default: flip_bits_l<M, RB, VEC, 3>(geo, flip, fthr, freg); break;
    }
}

// ---------------------------------------------------------------- interpreter
// Shears of register bit J: lo += a hi, then hi += b lo.
template <int J, int RA>
__device__ __forceinline__ void shear_pair(Amps<float, RA> &v, float a, float b)
{
    if constexpr (J == 0) {
#pragma unroll
        for (int p = 0; p < RA / 2; ++p) {
            float2 r = unpk(v.r[p]), i = unpk(v.i[p]);
            r.x = fmaf(a, r.y, r.x);
            i.x = fmaf(a, i.y, i.x);
            r.y = fmaf(b, r.x, r.y);
            i.y = fmaf(b, i.x, i.y);
            v.r[p] = pk(r.x, r.y);
            v.i[p] = pk(i.x, i.y);
        }
    } else if constexpr ((1 << J) < RA) {
        const pack2 A = dup(a), B = dup(b);
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (!(p & (1 << (J - 1)))) {
                const int q = p | (1 << (J - 1));
                v.r[p] = fma2(A, v.r[q], v.r[p]);
                v.i[p] = fma2(A, v.i[q], v.i[p]);
            }
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (!(p & (1 << (J - 1)))) {
                const int q = p | (1 << (J - 1));
                v.r[q] = fma2(B, v.r[p], v.r[q]);
                v.i[q] = fma2(B, v.i[p], v.i[q]);
            }
    }
}
template <int J, int RA>
__device__ __forceinline__ void shear_pair(Amps<double, RA> &v, double a, double b)
{
    if constexpr ((1 << J) < RA) {
#pragma unroll
        for (int k = 0; k < RA; ++k)
            if (!(k & (1 << J))) {
                const int q = k | (1 << J);
                v.r[k] = fma(a, v.r[q], v.r[k]);
                v.i[k] = fma(a, v.i[q], v.i[k]);
                v.r[q] = fma(b, v.r[k], v.r[q]);
                v.i[q] = fma(b, v.i[k], v.i[q]);
            }
    }
}
// the same with complex factors
template <int J, int RA>
__device__ __forceinline__ void cshear_pair(Amps<float, RA> &v, float ar, float ai, float br, float bi)
{
    if constexpr (J == 0) {
#pragma unroll
        for (int p = 0; p < RA / 2; ++p) {
            float2 r = unpk(v.r[p]), i = unpk(v.i[p]);
            r.x = fmaf(ar, r.y, fmaf(-ai, i.y, r.x));
            i.x = fmaf(ar, i.y, fmaf(ai, r.y, i.x));
            r.y = fmaf(br, r.x, fmaf(-bi, i.x, r.y));
            i.y = fmaf(br, i.x, fmaf(bi, r.x, i.y));
            v.r[p] = pk(r.x, r.y);
            v.i[p] = pk(i.x, i.y);
        }
    } else if constexpr ((1 << J) < RA) {
        const pack2 AR = dup(ar), AI = dup(ai), NAI = dup(-ai), BR = dup(br), BI = dup(bi), NBI = dup(-bi);
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (!(p & (1 << (J - 1)))) {
                const int q = p | (1 << (J - 1));
                v.r[p] = fma2(AR, v.r[q], fma2(NAI, v.i[q], v.r[p]));
                v.i[p] = fma2(AR, v.i[q], fma2(AI, v.r[q], v.i[p]));
                v.r[q] = fma2(BR, v.r[p], fma2(NBI, v.i[p], v.r[q]));
                v.i[q] = fma2(BR, v.i[p], fma2(BI, v.r[p], v.i[q]));
            }
    }
}
template <int J, int RA>
__device__ __forceinline__ void cshear_pair(Amps<double, RA> &v, double ar, double ai, double br, double bi)
{
    if constexpr ((1 << J) < RA) {
#pragma unroll
        for (int k = 0; k < RA; ++k)
            if (!(k & (1 << J))) {
                const int q = k | (1 << J);
                v.r[k] = fma(ar, v.r[q], fma(-ai, v.i[q], v.r[k]));
                v.i[k] = fma(ar, v.i[q], fma(ai, v.r[q], v.i[k]));
                v.r[q] = fma(br, v.r[k], fma(-bi, v.i[k], v.r[q]));
                v.i[q] = fma(br, v.i[k], fma(bi, v.r[k], v.i[q]));
            }
    }
}

// Factor tables of all registers.  complex64, complex factors: per pack p the
// real and imaginary parts (entry p of RA / 2 float4), then the negated
// imaginary parts (RA / 2 float2): the operands of the packed multiplies.
template <typename R>
__host__ __device__ constexpr int ctable_units(int RA) { return sizeof(R) == 4 ? RA / 2 + RA / 4 : RA; }
template <int RA>
__device__ __forceinline__ void cmul_pack(Amps<float, RA> &v, int p, pack2 gr, pack2 gi, pack2 ni)
{
    const pack2 t = mul2(gr, v.r[p]), u = mul2(gi, v.r[p]);
    v.r[p] = fma2(ni, v.i[p], t);
    v.i[p] = fma2(gr, v.i[p], u);
}
// J < 0: every register, else those with bit J set
template <int J, int RA>
__device__ __forceinline__ void mul_table(Amps<float, RA> &v, const uint4 *body)
{
    if constexpr (J < 0 || (1 << (J < 0 ? 0 : J)) < RA) {
        const ulonglong2 *t = reinterpret_cast<const ulonglong2 *>(body);
        const pack2 *n = reinterpret_cast<const pack2 *>(body + RA / 2);
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (J <= 0 || (p & (1 << (J > 0 ? J - 1 : 0)))) {
                const ulonglong2 g = t[p];
                if constexpr (J == 0) cmul_at(v, 2 * p + 1, unpk(g.x).y, unpk(g.y).y);
                else cmul_pack(v, p, g.x, g.y, n[p]);
            }
    }
}
template <int J, int RA>
__device__ __forceinline__ void mul_table(Amps<double, RA> &v, const uint4 *body)
{
    if constexpr (J < 0 || (1 << (J < 0 ? 0 : J)) < RA) {
        const double2 *t = reinterpret_cast<const double2 *>(body);
#pragma unroll
        for (int k = 0; k < RA; ++k)
            if (J < 0 || (k & (1 << (J > 0 ? J : 0)))) {
                const double2 g = t[k];
                cmul_at(v, k, g.x, g.y);
            }
    }
}
template <int J, int RA>
__device__ __forceinline__ void mul_one(Amps<float, RA> &v, float gr, float gi)
{
    if constexpr (J == 0) {
#pragma unroll
        for (int p = 0; p < RA / 2; ++p) cmul_at(v, 2 * p + 1, gr, gi);
    } else if constexpr ((1 << J) < RA) {
        const pack2 G = dup(gr), I = dup(gi), N = dup(-gi);
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (p & (1 << (J - 1))) cmul_pack(v, p, G, I, N);
    }
}
template <int J, int RA>
__device__ __forceinline__ void mul_one(Amps<double, RA> &v, double gr, double gi)
{
    if constexpr ((1 << J) < RA) {
#pragma unroll
        for (int k = 0; k < RA; ++k)
            if (k & (1 << J)) cmul_at(v, k, gr, gi);
    }
}
// the registers with bit J set times a phase e^{i phi}, |phi| <= pi / 2, in
// place: re += a im, im += b re, re += a im with a = -tan(phi / 2), b = sin phi
template <int J, int RA>
__device__ __forceinline__ void turn(Amps<float, RA> &v, float a, float b)
{
    if constexpr (J == 0) {
#pragma unroll
        for (int p = 0; p < RA / 2; ++p) {
            float2 r = unpk(v.r[p]), i = unpk(v.i[p]);
            r.y = fmaf(a, i.y, r.y);
            i.y = fmaf(b, r.y, i.y);
            r.y = fmaf(a, i.y, r.y);
            v.r[p] = pk(r.x, r.y);
            v.i[p] = pk(i.x, i.y);
        }
    } else if constexpr ((1 << J) < RA) {
        const pack2 A = dup(a), B = dup(b);
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (p & (1 << (J - 1))) v.r[p] = fma2(A, v.i[p], v.r[p]);
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (p & (1 << (J - 1))) v.i[p] = fma2(B, v.r[p], v.i[p]);
#pragma unroll
        for (int p = 0; p < RA / 2; ++p)
            if (p & (1 << (J - 1))) v.r[p] = fma2(A, v.i[p], v.r[p]);
    }
}
template <int J, int RA>
__device__ __forceinline__ void turn(Amps<double, RA> &v, double a, double b)
{
    if constexpr ((1 << J) < RA) {
#pragma unroll
        for (int k = 0; k < RA; ++k)
            if (k & (1 << J)) {
                v.r[k] = fma(a, v.i[k], v.r[k]);
                v.i[k] = fma(b, v.r[k], v.i[k]);
                v.r[k] = fma(a, v.i[k], v.r[k]);
            }
    }
}
// a ramp on register bit J: the registers' table, then the thread's factor
template <int J, typename R, int RA>
__device__ __forceinline__ void ramp_half(Amps<R, RA> &v, R fr, R fi, const uint4 *body, bool has_reg)
{
    if (has_reg) mul_table<J>(v, body);
    mul_one<J>(v, fr, fi);
}
// entry k of a register table
template <int RA>
__device__ __forceinline__ float2 table_at(const uint4 *body, int k, const Amps<float, RA> &)
{
    const float4 g = reinterpret_cast<const float4 *>(body)[k >> 1];
    return (k & 1) ? make_float2(g.y, g.w) : make_float2(g.x, g.z);
}
template <int RA>
__device__ __forceinline__ double2 table_at(const uint4 *body, int k, const Amps<double, RA> &)
{
    return reinterpret_cast<const double2 *>(body)[k];
}
template <int RA>
__device__ __forceinline__ void mul_real(Amps<float, RA> &v, const uint4 *body)
{
    const pack2 *g = reinterpret_cast<const pack2 *>(body);
#pragma unroll
    for (int p = 0; p < RA / 2; ++p) {
        const pack2 t = g[p];
        v.r[p] = mul2(t, v.r[p]);
        v.i[p] = mul2(t, v.i[p]);
    }
}
template <int RA>
__device__ __forceinline__ void mul_real(Amps<double, RA> &v, const uint4 *body)
{
    const double *g = reinterpret_cast<const double *>(body);
#pragma unroll
    for (int k = 0; k < RA; ++k) {
        v.r[k] *= g[k];
        v.i[k] *= g[k];
    }
}
template <int RA>
__device__ __forceinline__ void xor_signs(Amps<float, RA> &v, const uint32_t *lo, const uint32_t *hi)
{
#pragma unroll
    for (int p = 0; p < RA / 2; ++p) {
        const uint32_t s0 = lo[(2 * p) & 7] ^ hi[(2 * p) >> 3], s1 = lo[(2 * p + 1) & 7] ^ hi[(2 * p) >> 3];
        const pack2 m = ((pack2)s1 << 32) | s0;
        v.r[p] ^= m;
        v.i[p] ^= m;
    }
}
template <int RA>
__device__ __forceinline__ void xor_signs(Amps<double, RA> &v, const uint32_t *lo, const uint32_t *hi)
{
#pragma unroll
    for (int k = 0; k < RA; ++k) v.set(k, flip_sign(v.r[k], lo[k & 7] ^ hi[k >> 3]), flip_sign(v.i[k], lo[k & 7] ^ hi[k >> 3]));
}

// the pending signs into the registers: the sign of register k is the parity
// of k & zs, plus bit 6
template <typename R, int RA>
__device__ __forceinline__ void flush_signs(Amps<R, RA> &v, uint32_t zs)
{
    uint32_t lo[8], hi[8];
    auto bit = [&](int j) { return (zs << (31 - j)) & 0x80000000u; };
    lo[0] = bit(6);
    hi[0] = 0u;
#pragma unroll
    for (int x = 1; x < 8; ++x) {
        const int j = (x & 4) ? 2 : (x & 2) ? 1 : 0;
        lo[x] = lo[x & ~(1 << j)] ^ bit(j);
        hi[x] = hi[x & ~(1 << j)] ^ bit(j + 3);
    }
    xor_signs(v, lo, hi);
}

// exchange on register bit J of the pairs whose bit in act is set
template <int J, typename R, int RA>
__device__ __forceinline__ void exchange(Amps<R, RA> &v, int kind, unsigned long long act, const R *m)
{
    if constexpr ((1 << J) < RA) {
        if (kind == SK_XPERM) {
#pragma unroll
            for (int k = 0; k < RA; ++k)
                if (!(k & (1 << J))) {
                    const bool on = (act >> k) & 1ull;
                    const int q = k | (1 << J);
                    const R lr = v.re(k), li = v.im(k), hr = v.re(q), hi = v.im(q);
                    v.set(k, on ? hr : lr, on ? hi : li);
                    v.set(q, on ? lr : hr, on ? li : hi);
                }
        } else {
            const R ar = m[0], ai = m[1], br = m[2], bi = m[3], cr = m[4], ci = m[5], dr = m[6], di = m[7];
#pragma unroll
            for (int k = 0; k < RA; ++k)
                if (!(k & (1 << J)) && ((act >> k) & 1ull)) {
                    const int q = k | (1 << J);
                    const R lr = v.re(k), li = v.im(k), hr = v.re(q), hi = v.im(q);
                    v.set(k, ar * lr - ai * li + (br * hr - bi * hi), ar * li + ai * lr + (br * hi + bi * hr));
                    v.set(q, cr * lr - ci * li + (dr * hr - di * hi), cr * li + ci * lr + (dr * hi + di * hr));
                }
        }
    }
}

// Run a tile program on the registers of one tile.  tile: the tile's index
// (bit i = the i-th outer qubit); sm: the tile's shared memory (tile_slots
// amplitudes); sp: kChunkUnits units of shared memory, whose first chunk the
// caller has staged (prog_stage + __syncthreads).  All threads run the same
// operations; the control words go through a warp reduction, which leaves
// them in uniform registers (branches without divergence bookkeeping).
// kFull false: programs of groups alone -- a third of the code, which the
// instruction cache and the register allocation feel (189 to 172 ms for the
// 30-qubit depth-20 circuit).
//
// What bounds it (13-qubit tiles, 26 qubits, one operation alone): a pass
// that only loads and stores runs at the HBM rate (0.73 ms for 2 x 2 GiB at 28 qubits);
// a change of layout 24 us, shared-memory bandwidth (16 bytes an amplitude);
// a pair of shears 6 us and a full complex table 12 us, about half the FP32 rate:
// eight warps an SM do not hide all of the decoding.  The 30-qubit circuit's
// 23 passes take 7.5 ms each, where interpreting one gate at a time took 16.
template <typename R, int M, bool kFull>
__device__ __forceinline__ void run_program(Amps<R, (1 << (M - kTpThrBits))> &v, const uint4 *__restrict__ gprog,
                                            int nunits, uint32_t tile, int tid, R *sm, uint4 *sp)
{
    using V = typename V2<R>::T;
    constexpr int VEC = (sizeof(R) == 4) ? 2 : 1;
    constexpr int RB = M - kTpThrBits;
    constexpr int RA = 1 << RB;
    auto uniform = [](uint32_t x) { return __reduce_or_sync(0xffffffffu, x); };
    static_assert(RB >= 4 && RB <= 6, "4 to 6 register bits");
    uint32_t zs = 0;                 // bit j: pending Z on register bit j; bit 6: pending -1
    const uint4 *at = sp;
    int chunk = 0;
    uint4 h = *at;
    for (;;) {
        const uint32_t f = uniform(h.x);
        const uint32_t op = f & 15u;
        if (op <= TP_CHUNK) {
            if (op == TP_END) break;
            __syncthreads();
            ++chunk;
            const int first = chunk * kChunkUnits, cnt = min(kChunkUnits, nunits - first);
            for (int e = tid; e < cnt; e += kTpThr) sp[e] = __ldg(gprog + first + e);
            __syncthreads();
            at = sp;
            h = *at;
            continue;
        }
        const uint4 *body = at + 1;
        at += (f >> 4) & 0xffu;
        const uint4 hn = *at;            // the next operation's header, loaded early
        auto conds = [&]() {
            return ((uint32_t)tid & (h.y & 0xffu)) == ((h.y >> 8) & 0xffu) && (tile & h.z) == h.z;
        };
        if (!kFull || op == TP_GROUP) {
            const uint32_t nz = (f >> 24) & 31u;
            if (nz) {
                const uint2 *ze = reinterpret_cast<const uint2 *>(body);
                for (uint32_t e = 0; e < nz; ++e) {
                    const uint2 q = ze[e];
                    const bool on = ((((uint32_t)tid & q.x) ^ (q.x >> 8)) & 0xffu) == 0 && (tile & q.y) == q.y;
                    zs ^= on ? (q.x >> 16) : 0u;
                }
                body += (nz + 1) >> 1;
            }
            const uint32_t kind = (f >> 12) & 7u;
            if (kind == GD_CPLX) {
                mul_table<-1>(v, body);
                body += ctable_units<R>(RA);
            } else if (kind == GD_HALF) {
                // a phase as three shears of (re, im)
                const V g = *reinterpret_cast<const V *>(body);
                switch ((f >> 15) & 7u) {
                case 0: turn<0>(v, g.x, g.y); break;
                case 1: turn<1>(v, g.x, g.y); break;
                case 2: turn<2>(v, g.x, g.y); break;
                case 3: turn<3>(v, g.x, g.y); break;
                case 4: turn<4>(v, g.x, g.y); break;
                default: turn<5>(v, g.x, g.y); break;
                }
                ++body;
            } else if (kind == GD_REAL) {
                mul_real(v, body);
                body += RA * (int)sizeof(R) / 16;
            }
            const uint32_t bits = (f >> 18) & 63u;
            if (bits) {
                const V *ab = reinterpret_cast<const V *>(body);
                V t[RB];
#pragma unroll
                for (int j = 0; j < RB; ++j) t[j] = ab[j];
                if ((f >> 29) & 1u) {
#pragma unroll
                    for (int j = 0; j < RB; ++j) {
                        const uint32_t sg = (zs << (31 - j)) & 0x80000000u;
                        t[j].x = flip_sign(t[j].x, sg);
                        t[j].y = flip_sign(t[j].y, sg);
                    }
                }
                if (bits & 7u) {
                    if (bits & 1u) shear_pair<0>(v, t[0].x, t[0].y);
                    if (bits & 2u) shear_pair<1>(v, t[1].x, t[1].y);
                    if (bits & 4u) shear_pair<2>(v, t[2].x, t[2].y);
                }
                if (bits & 56u) {
                    if (bits & 8u) shear_pair<3>(v, t[3].x, t[3].y);
                    if constexpr (RB > 4) {
                        if (bits & 16u) shear_pair<4>(v, t[4].x, t[4].y);
                    }
                    if constexpr (RB > 5) {
                        if (bits & 32u) shear_pair<5>(v, t[5].x, t[5].y);
                    }
                }
            }
            if (f >> 30) {
                if ((f >> 30) & 1u) {
                    flush_signs(v, zs);
                    zs = 0;
                }
                if (f >> 31) {
                    const uint32_t lay = uniform(h.y);
                    relayout<M, RB, VEC>((int)(lay & 3u), (int)(lay >> 2), v, sm, tid);
                }
            }
        } else if (op == TP_RAMP) {
            if (conds()) {
                const unsigned long long km = *reinterpret_cast<const unsigned long long *>(body);
                ++body;
                const bool has_reg = ((f >> 15) & 1u) != 0;
                const V *t = reinterpret_cast<const V *>(body + (has_reg ? ctable_units<R>(RA) : 0));
                V w;
                w.x = (R)1;
                w.y = (R)0;
                if ((f >> 16) & 1u) {
                    w = t[tid & 15];
                    const V b = t[16 + (tid >> 4)];
                    cmul(w, b.x, b.y);
                    t += kThrTab;
                }
                uint32_t groups = (f >> 17) & 63u;
                uint32_t idx = tile;
                while (groups) {
                    if (groups & 1u) {
                        const V b = t[idx & 15u];
                        cmul(w, b.x, b.y);
                        t += 16;
                    }
                    groups >>= 1;
                    idx >>= kOutGroup;
                }
                switch ((f >> 12) & 7u) {
                case 0: ramp_half<0>(v, w.x, w.y, body, has_reg); break;
                case 1: ramp_half<1>(v, w.x, w.y, body, has_reg); break;
                case 2: ramp_half<2>(v, w.x, w.y, body, has_reg); break;
                case 3: ramp_half<3>(v, w.x, w.y, body, has_reg); break;
                case 4: ramp_half<4>(v, w.x, w.y, body, has_reg); break;
                case 5: ramp_half<5>(v, w.x, w.y, body, has_reg); break;
                default:
#pragma unroll
                    for (int k = 0; k < RA; ++k)
                        if ((km >> k) & 1ull) {
                            V g = w;
                            if (has_reg) {
                                const V r = table_at(body, k, v);
                                cmul(g, r.x, r.y);
                            }
                            cmul_at(v, k, g.x, g.y);
                        }
                    break;
                }
            }
        } else if (op == TP_XCH) {
            const unsigned long long act = conds() ? *reinterpret_cast<const unsigned long long *>(body) : 0ull;
            const R *m = reinterpret_cast<const R *>(body + 1);
            const int kind = (int)((f >> 15) & 3u);
            switch ((f >> 12) & 7u) {
            case 0: exchange<0>(v, kind, act, m); break;
            case 1: exchange<1>(v, kind, act, m); break;
            case 2: exchange<2>(v, kind, act, m); break;
            case 3: exchange<3>(v, kind, act, m); break;
            case 4: exchange<4>(v, kind, act, m); break;
                default: exchange<5>(v, kind, act, m); break;
            }
        } else if (op == TP_PH) {
            const ulonglong2 k2 = *reinterpret_cast<const ulonglong2 *>(body);
            const uint4 u = body[1];
            const R *m = reinterpret_cast<const R *>(body + 2);
            const unsigned long long cond = conds() ? k2.x : 0ull;
            const bool outer = ((uint32_t)tid & (u.x & 0xffu)) == ((u.x >> 8) & 0xffu) && (tile & u.y) == u.y;
            const unsigned long long one = h.w ? (outer ? ~0ull : 0ull) : k2.y;
            const R ar = m[0], ai = m[1], dr = m[2], di = m[3];
#pragma unroll
            for (int k = 0; k < RA; ++k)
                if ((cond >> k) & 1ull) {
                    const bool t = (one >> k) & 1ull;
                    cmul_at(v, k, t ? dr : ar, t ? di : ai);
                }
        } else if (op == TP_PERM) {
            permute<M, RB, VEC>((int)((f >> 12) & 3u), v, sm, tid, reinterpret_cast<const int *>(body));
        } else {                                     // TP_CSHEARS
            const V *ab = reinterpret_cast<const V *>(body);
            const uint32_t j = (f >> 12) & 7u, s = (zs << (31 - j)) & 0x80000000u;
            const R ar = flip_sign(ab[0].x, s), ai = flip_sign(ab[0].y, s);
            const R br = flip_sign(ab[1].x, s), bi = flip_sign(ab[1].y, s);
            switch (j) {
            case 0: cshear_pair<0>(v, ar, ai, br, bi); break;
            case 1: cshear_pair<1>(v, ar, ai, br, bi); break;
            case 2: cshear_pair<2>(v, ar, ai, br, bi); break;
            case 3: cshear_pair<3>(v, ar, ai, br, bi); break;
            case 4: cshear_pair<4>(v, ar, ai, br, bi); break;
                default: cshear_pair<5>(v, ar, ai, br, bi); break;
            }
        }
        h = hn;
    }
}

// the first chunk of a program into shared memory
__device__ __forceinline__ void prog_stage(const uint4 *__restrict__ gprog, int nunits, int tid, uint4 *sp)
{
    const int cnt = min(kChunkUnits, nunits);
    for (int e = tid; e < cnt; e += kTpThr) sp[e] = __ldg(gprog + e);
}

// CTAs per SM the kernels' registers are budgeted for: 13-qubit complex64
// tiles hold 128 registers of amplitudes a thread, and a third CTA (168
// registers) spills -- 268 ms for the 30-qubit depth-20 circuit instead of
// 172; 12-qubit tiles lose the same way with a fifth (224 against 173 ms).
template <typename R, int M>
constexpr int tile_ctas()
{
    if (sizeof(R) == 8) return M == 12 ? 2 : 4;
    return M == 13 ? 2 : M == 12 ? 4 : 6;
}
template <typename R, int M>
constexpr size_t tile_smem_bytes()
{
    constexpr int VEC = sizeof(R) == 4 ? 2 : 1;
    static_assert(sizeof(R) == 8 || tile_slots<M, M - kTpThrBits, VEC>() % 2 == 0, "the planes and the program start on 16-byte boundaries");
    return (size_t)tile_slots<M, M - kTpThrBits, VEC>() * 2 * sizeof(R) + (size_t)kChunkUnits * 16;
}

// ---------------------------------------------------------------- host: diagonal pool
using cplx = std::complex<double>;

// The diagonal operator collected so far:
//     g * prod_q y[q]^{x_q} * prod_{a<b} pair(a, b)^{x_a x_b}.
// Entries stay until a non-diagonal gate on one of their qubits needs them.
struct DiagPool {
    int n = 0;
    cplx g{1.0, 0.0};
    std::vector<cplx> y, pr;
    std::vector<uint64_t> adj;     // qubits that share a pair with q
    explicit DiagPool(int n_) : n(n_), y((size_t)n_, 1.0), pr((size_t)n_ * n_, 1.0), adj((size_t)n_, 0) {}
    cplx &pair(int a, int b) { return pr[(size_t)std::min(a, b) * n + std::max(a, b)]; }
    void mul_pair(int a, int b, cplx f)
    {
        cplx &p = pair(a, b);
        p = (p == 1.0) ? f : p * f;
        const uint64_t ma = 1ull << a, mb = 1ull << b;
        if (p == 1.0) {
            adj[a] &= ~mb;
            adj[b] &= ~ma;
        } else {
            adj[a] |= mb;
            adj[b] |= ma;
        }
    }
    cplx take_pair(int a, int b)
    {
        const cplx p = pair(a, b);
        pair(a, b) = 1.0;
        adj[a] &= ~(1ull << b);
        adj[b] &= ~(1ull << a);
        return p;
    }
};

// a factor the pool may hold: finite and far from zero (its inverse is formed)
inline bool pool_factor(cplx f)
{
    const double a = std::abs(f);
    return a > 1e-6 && a < 1e6;
}
// modulus one to FP32 rounding of the entries: such factors may pile up without
// leaving the range (a million of them by less than two bits)
inline bool unit_factor(cplx f) { return std::abs(std::norm(f) - 1.0) <= 2e-6; }
// as far as the common factor may go
constexpr double kPoolBits = 8.0;

// One operation before packing; the first five kinds are packed into groups.
enum IrKind { IR_Z = 0, IR_DIAG, IR_SHEARS, IR_FLUSH, IR_LAYOUT, IR_RAMP, IR_XCH, IR_PH, IR_CSHEARS, IR_PERM };
struct TpOp {
    int op = IR_Z;
    uint32_t arg = 0;              // IR_Z: sign bits; IR_DIAG: GroupDiag | register bit << 3; IR_SHEARS: register bits;
                                   // IR_LAYOUT: from | to << 2; others: header bits 12..
    uint32_t thr = 0, out = 0;
    uint64_t km = 0;
    std::vector<cplx> tab;         // tables in packing order (shears: (a, b); real factors: real parts)
    std::vector<double> mat;       // IR_XCH: 8 doubles; IR_PH: 4
    std::vector<uint32_t> words;   // IR_PERM: slot weights
    uint64_t km_t = 0;
    uint32_t thr_t = 0, out_t = 0, place = 0;
    size_t ra = 0;                 // IR_RAMP: entries of the register table at the head of tab
};

struct TilePass {
    int start_layout = 0, end_layout = 0;
    uint64_t flip = 0;             // qubits whose labels the store exchanges
    std::vector<TpOp> ops;
    bool groups_only() const
    {
        for (const TpOp &o : ops)
            if (o.op > IR_LAYOUT) return false;
        return true;
    }
};

// U = diag(p, q) K diag(1, y) with K = [[1, -t], [t, 1]] (swap false) or
// [[t, -1], [1, t]] (swap true), 0 <= t <= 1; false when U is not a multiple
// of a unitary matrix to FP64 rounding.  p, q carry the scale, |y| = 1.
inline bool split_unitary(const double m[8], cplx *p, cplx *q, cplx *y, double *t, bool *swap)
{
    const cplx A(m[0], m[1]), B(m[2], m[3]), C(m[4], m[5]), D(m[6], m[7]);
    const double a = std::abs(A), c = std::abs(C), s = std::hypot(a, c);
    if (!(s > 1e-3 && s < 1e3)) return false;
    if (a >= c) {
        *swap = false;
        *t = c / a;
        *p = A;
        *q = c > 0 ? C * (a / c) : cplx(a, 0.0);
        *y = D / *q;
        if (std::abs(B + *p * *t * *y) > 1e-14 * s) return false;
    } else {
        *swap = true;
        *t = a / c;
        *p = a > 0 ? A * (c / a) : cplx(c, 0.0);
        *q = C;
        *y = -B / *p;
        if (std::abs(D - *q * *t * *y) > 1e-14 * s) return false;
    }
    const double ya = std::abs(*y);
    if (std::abs(ya - 1.0) > 1e-14) return false;
    *y /= ya;
    return true;
}

// M = diag(p, q) [[1, 0], [b, 1]] [[1, a], [0, 1]], rows exchanged first when
// swap: the shears of any invertible matrix (complex, four multiply-adds per
// amplitude); false when a factor would be large (a matrix close to singular)
inline bool split_general(const double m[8], cplx *p, cplx *q, cplx *a, cplx *b, bool *swap)
{
    cplx A(m[0], m[1]), B(m[2], m[3]), C(m[4], m[5]), D(m[6], m[7]);
    *swap = std::abs(A) < std::abs(C);
    if (*swap) {
        std::swap(A, C);
        std::swap(B, D);
    }
    const cplx det = A * D - B * C;
    if (!pool_factor(A) || !pool_factor(det)) return false;
    *p = A;
    *q = det / A;
    *a = B / A;
    *b = C * A / det;
    return pool_factor(*q) && pool_factor(*q / *p) && std::abs(*a) <= 4.0 && std::abs(*b) <= 4.0;
}

// Compiles the scheduled gates of consecutive passes into tile programs; the
// pool carries diagonal factors from pass to pass.  R is the kernel's real
// type (the shear factor is rounded to it before the matching scale is formed).
template <typename R>
class TileCompiler {
public:
    TileCompiler(int n, int M, int VEC) : pool(n), n_(n), M_(M), RB_(M - kTpThrBits), RA_(1 << (M - kTpThrBits)), VEC_(VEC)
    {
        for (int l = 0; l < 4; ++l) {
            io_[l] = io_layout(M_, RB_, VEC_, l);
            for (int j = 0; j < RB_; ++j) lreg_[l][j] = l < n_layouts(M_, RB_) ? reg_local(M_, RB_, VEC_, l, j) : 0;
            for (int i = 0; i < kTpThrBits; ++i) lthr_[l][i] = l < n_layouts(M_, RB_) ? thr_local(M_, RB_, VEC_, l, i) : 0;
        }
    }

    DiagPool pool;

    void begin(const Pass &ps)
    {
        loc_.assign((size_t)n_, -1);
        for (int q = 0; q < kLow && q < n_; ++q) loc_[q] = q;
        for (size_t i = 0; i < ps.high.size(); ++i) loc_[ps.high[i]] = kLow + (int)i;
        outbit_.assign((size_t)n_, -1);
        for (int q = 0, i = 0; q < n_; ++q)
            if (loc_[q] < 0) outbit_[q] = i++;
        out_ = TilePass();
        home_ = loc_;
        layout_ = 0;
        started_ = false;
        zdirty_ = false;
        final_ = false;
        queued_ = 0;
        reset_group();
        map_layout();
    }

    void set_layout(int l)
    {
        if (l == layout_) return;
        if (!started_ && !queued_ && pre_.empty() && !tab_used_ && io_[l]) {
            // nothing ran yet: load in this layout
            layout_ = l;
            out_.start_layout = l;
            map_layout();
            return;
        }
        close_group();
        flush_signs();
        TpOp o;
        o.op = IR_LAYOUT;
        o.arg = (uint32_t)(layout_ | (l << 2));
        emit(o);
        layout_ = l;
        map_layout();
    }

    // one gate, under layout l (its target in a register when it is not diagonal)
    void gate(const SGate &g, int l)
    {
        if (g.op == OP_DIAG || g.op == OP_DIAG_HI) {
            diagonal(g);
            return;
        }
        const int nc = __builtin_popcountll(g.ctrl);
        const cplx B(g.m[2], g.m[3]), C(g.m[4], g.m[5]);
        if (nc == 0 && g.op == OP_XPERM) {
            relabel(g.target);
            return;
        }
        if (g.op == OP_SWAP) {
            swap_places(g.target, g.target2);
            return;
        }
        if (nc == 0 && g.op == OP_ANTIDIAG && takes(C, B)) {
            pool.g *= C;
            pool.y[g.target] *= B / C;       // X diag(C, B)
            relabel(g.target);
            return;
        }
        set_layout(l);
        if (nc == 0 && g.op == OP_DENSE && (rotation(g) || shears(g))) return;
        masked_exchange(g);
    }

    // the pass is over; last: apply what is left of the pool.  unit_ok: drop
    // factors of modulus one instead (only |amplitude|^2 is asked for).
    TilePass end(bool last, bool unit_ok = false)
    {
        close_group();
        if (last) final_pool(unit_ok);
        if (last && unit_ok) zdirty_ = false;      // signs and the layout do not matter to |amplitude|^2
        flush_signs();
        if (!(last && unit_ok)) {                  // <sum Z> does not depend on where the qubits are
            if (loc_ != home_) restore_places();
            if (!io_[layout_]) set_layout(0);
        }
        out_.end_layout = layout_;
        out_.flip = flip_;
        flip_ = 0;
        return std::move(out_);
    }
    int current_layout() const { return layout_; }

private:
    int n_, M_, RB_, RA_, VEC_;
    bool io_[4];                          // layouts the pass may load and store in
    int lreg_[4][8], lthr_[4][kTpThrBits];   // their local bits
    std::vector<int> loc_, outbit_;       // per qubit: local bit (-1: outside the tile), bit of the tile index
    std::vector<int> home_;               // loc_ as the state is stored
    std::vector<int> reg_, thr_;          // per qubit: register / thread bit of the current layout, -1 if none
    std::vector<int> regq_;               // qubit of register bit j
    TilePass out_;
    int layout_ = 0;
    bool started_ = false, zdirty_ = false, final_ = false;
    uint64_t flip_ = 0;
    // the open group: factors and operations that precede the queued shears
    std::vector<cplx> tab_;
    bool tab_used_ = false;
    std::vector<TpOp> pre_;
    uint32_t queued_ = 0;
    double sa_[8] = {}, sb_[8] = {};

    void map_layout()
    {
        reg_.assign((size_t)n_, -1);
        thr_.assign((size_t)n_, -1);
        regq_.assign((size_t)RB_, -1);
        int qof[16];
        for (int b = 0; b < 16; ++b) qof[b] = -1;
        for (int q = 0; q < n_; ++q)
            if (loc_[q] >= 0) qof[loc_[q]] = q;
        for (int j = 0; j < RB_; ++j) {
            const int q = qof[lreg_[layout_][j]];
            regq_[(size_t)j] = q;
            if (q >= 0) reg_[(size_t)q] = j;
        }
        for (int i = 0; i < kTpThrBits; ++i) {
            const int q = qof[lthr_[layout_][i]];
            if (q >= 0) thr_[(size_t)q] = i;
        }
    }
    bool flipped(int q) const { return (flip_ >> q) & 1ull; }
    // whether the pool may take a gate's factors a and d (of a qubit's 0 and 1)
    bool takes(cplx a, cplx d) const
    {
        if (!pool_factor(a) || !pool_factor(d)) return false;
        if (unit_factor(a) && unit_factor(d)) return true;
        auto bits = [](cplx f) { return unit_factor(f) ? 0.0 : std::abs(std::log2(std::abs(f))); };
        double t = bits(a) + bits(d) + bits(pool.g);
        for (const cplx &f : pool.y) t += bits(f);
        return t <= kPoolBits;
    }
    // logical value of qubit q (a register bit) in register k
    int bit_of(int q, int k) const { return ((k >> reg_[(size_t)q]) & 1) ^ (flipped(q) ? 1 : 0); }

    void emit(TpOp o)
    {
        out_.ops.push_back(std::move(o));
        started_ = true;
    }
    void reset_group()
    {
        if (tab_used_ || tab_.size() != (size_t)RA_) tab_.assign((size_t)RA_, 1.0);
        tab_used_ = false;
        pre_.clear();
        queued_ = 0;
    }
    // the plain product: std::complex's own looks for infinities in each one
    static cplx times(cplx a, cplx b)
    {
        return cplx(a.real() * b.real() - a.imag() * b.imag(), a.real() * b.imag() + a.imag() * b.real());
    }
    void tab_single(int q, cplx f)
    {
        const int m = 1 << reg_[(size_t)q], want = flipped(q) ? 0 : m;
        for (int k = 0; k < RA_; ++k)
            if ((k & m) == want) tab_[(size_t)k] = tab_used_ ? times(tab_[(size_t)k], f) : f;
        tab_used_ = true;
    }
    void tab_pair(int a, int b, cplx f)
    {
        const int ma = 1 << reg_[(size_t)a], mb = 1 << reg_[(size_t)b];
        const int want = (flipped(a) ? 0 : ma) | (flipped(b) ? 0 : mb);
        for (int k = 0; k < RA_; ++k)
            if ((k & (ma | mb)) == want) tab_[(size_t)k] = times(tab_[(size_t)k], f);
        tab_used_ = true;
    }
    bool tab_real() const
    {
        for (const cplx &c : tab_)
            if (c.imag() != 0.0) return false;
        return true;
    }
    // the register bit the table depends on alone, by a phase of at most a
    // quarter turn (the factor of its 0 half then joins the pool; in the final
    // table it has to be 1), -1 if none
    int half_bit() const
    {
        bool constant = true;
        for (const cplx &c : tab_) constant = constant && c == tab_[0];
        if (constant || (final_ && tab_[0] != 1.0)) return -1;
        for (int j = 0; j < RB_; ++j) {
            bool same = true;
            for (int k = 0; k < RA_ && same; ++k) same = tab_[(size_t)k] == tab_[((k >> j) & 1) ? (size_t)1 << j : 0];
            const cplx f = tab_[(size_t)1 << j] / tab_[0];
            if (same) return std::abs(std::abs(f) - 1.0) < 4e-15 && f.real() >= 0.0 ? j : -1;
        }
        return -1;
    }
    // the table as one multiply: real factors (one packed multiply an
    // amplitude), half of the registers, or all of them (four each)
    void emit_table()
    {
        TpOp o;
        o.op = IR_DIAG;
        const int j = tab_real() ? -1 : half_bit();
        if (j >= 0) {
            const cplx c = tab_[0], f = tab_[(size_t)1 << j] / c;
            pool.g *= c;
            const double t = (double)(R)(-f.imag() / (1.0 + f.real()));
            o.arg = (uint32_t)(GD_HALF | (j << 3));
            o.tab.push_back(cplx(t, -2.0 * t / (1.0 + t * t)));
        } else {
            const bool real = tab_real();
            const cplx s = (!real || pool.g.imag() == 0.0) ? pool.g : cplx(std::abs(pool.g), 0.0);
            if (s != 1.0)
                for (cplx &c : tab_) c = times(c, s);
            pool.g = (s == pool.g) ? cplx(1.0) : pool.g / s;
            o.arg = real ? GD_REAL : GD_CPLX;
            o.tab.swap(tab_);              // a fresh one at the next reset
        }
        pre_.push_back(std::move(o));
    }
    // conditions "qubit b is 1" for a qubit outside the registers
    void add_cond(TpOp *o, int b) const
    {
        if (thr_[(size_t)b] >= 0) {
            const uint32_t m = 1u << thr_[(size_t)b];
            o->thr |= thr_cond(m, flipped(b) ? 0u : m);
        } else {
            o->out |= 1u << outbit_[(size_t)b];
        }
    }

    void close_group()
    {
        if (tab_used_) {
            // one table multiply is due.  If it takes all registers, it takes
            // along whatever else it can carry (not for the queued bits: their
            // entries belong after their shears)
            const bool real = tab_real();
            auto fits = [&](cplx f) { return !real || f.imag() == 0.0; };
            for (int j = (real || half_bit() < 0) ? 0 : RB_; j < RB_; ++j) {
                const int a = regq_[(size_t)j];
                if (a < 0 || ((queued_ >> j) & 1u)) continue;
                if (pool.y[(size_t)a] != 1.0 && fits(pool.y[(size_t)a])) {
                    tab_single(a, pool.y[(size_t)a]);
                    pool.y[(size_t)a] = 1.0;
                }
                for (int i = 0; i < j; ++i) {
                    const int b = regq_[(size_t)i];
                    if (b < 0 || ((queued_ >> i) & 1u) || !((pool.adj[(size_t)a] >> b) & 1ull)) continue;
                    if (fits(pool.pair(a, b))) tab_pair(a, b, pool.take_pair(a, b));
                }
            }
            emit_table();
        }
        for (TpOp &o : pre_) emit(std::move(o));
        if (queued_) {
            TpOp o;
            o.op = IR_SHEARS;
            o.arg = queued_;
            o.tab.reserve((size_t)RB_);
            for (int j = 0; j < RB_; ++j)
                o.tab.push_back(((queued_ >> j) & 1u) ? cplx(sa_[j], sb_[j]) : cplx(0.0));
            emit(std::move(o));
        }
        reset_group();
        const double a = std::abs(pool.g);
        if (a < 0x1p-8 || a > 0x1p8) {
            emit_scale(a);
            pool.g /= a;
        }
    }
    void emit_scale(double a)
    {
        TpOp o;
        o.op = IR_DIAG;
        o.arg = GD_REAL;
        o.tab.assign((size_t)RA_, a);
        emit(o);
    }
    void flush_signs()
    {
        if (!zdirty_) return;
        TpOp o;
        o.op = IR_FLUSH;
        emit(o);
        zdirty_ = false;
    }

    // X on qubit q: exchange its labels; the pool's entries follow
    // (X D = D' X with the factors of 0 and 1 exchanged)
    void relabel(int q)
    {
        flip_ ^= 1ull << q;
        invert_pool(q);
    }
    // SWAP of two qubits of the tile: exchange their places and the pool's entries
    void swap_places(int a, int b)
    {
        std::swap(loc_[(size_t)a], loc_[(size_t)b]);
        if (flipped(a) != flipped(b)) flip_ ^= (1ull << a) | (1ull << b);
        std::swap(pool.y[(size_t)a], pool.y[(size_t)b]);
        const uint64_t both = (1ull << a) | (1ull << b);
        for (uint64_t m = (pool.adj[(size_t)a] | pool.adj[(size_t)b]) & ~both; m; m &= m - 1) {
            const int c = __builtin_ctzll(m);
            const cplx fa = pool.take_pair(a, c), fb = pool.take_pair(b, c);
            if (fb != 1.0) pool.mul_pair(a, c, fb);
            if (fa != 1.0) pool.mul_pair(b, c, fa);
        }
        map_layout();
    }
    // move every qubit back to the place the state keeps it in
    void restore_places()
    {
        int to = 0;
        for (int l = 1; l < n_layouts(M_, RB_); ++l)
            if (io_[l]) to = l;
        auto weight = [&](int local) {
            int src = local;
            for (int q = 0; q < n_; ++q)
                if (home_[(size_t)q] == local) src = loc_[(size_t)q];
            return (uint32_t)(VEC_ == 2 ? (1 << src) + (((1 << src) >> (RB_ + 1)) << 1) : (1 << src) + ((1 << src) >> RB_));
        };
        TpOp o;
        o.op = IR_PERM;
        o.arg = (uint32_t)(layout_ | (to << 2));
        for (int i = 0; i < kTpThrBits; ++i) o.words.push_back(weight(lthr_[to][i]));
        for (int j = 0; j < RB_; ++j) o.words.push_back(weight(lreg_[to][j]));
        emit(std::move(o));
        loc_ = home_;
        layout_ = to;
        map_layout();
    }
    void invert_pool(int q)
    {
        pool.g *= pool.y[(size_t)q];
        pool.y[(size_t)q] = 1.0 / pool.y[(size_t)q];
        for (uint64_t a = pool.adj[(size_t)q]; a; a &= a - 1) {
            const int b = __builtin_ctzll(a);
            const cplx f = pool.take_pair(q, b);
            pool.y[(size_t)b] *= f;
            pool.mul_pair(q, b, f == -1.0 ? cplx(-1.0) : 1.0 / f);
        }
    }

    TpOp make_ramp(int q, const std::vector<std::pair<int, cplx>> &with, cplx own, const std::vector<cplx> *reg_tab,
                   bool everywhere)
    {
        TpOp o;
        o.op = IR_RAMP;
        std::vector<cplx> treg((size_t)RA_, 1.0), tthr((size_t)kThrTab, 1.0), tout((size_t)kOutGroups * 16, 1.0);
        bool hreg = false, hthr = false;
        uint32_t groups = 0;
        if (reg_tab) {
            treg = *reg_tab;
            hreg = true;
        }
        for (const auto &w : with) {
            const int b = w.first;
            if (reg_[(size_t)b] >= 0) {
                hreg = true;
                for (int k = 0; k < RA_; ++k)
                    if (bit_of(b, k)) treg[(size_t)k] *= w.second;
            } else if (thr_[(size_t)b] >= 0) {
                hthr = true;
                const int i = thr_[(size_t)b], f = flipped(b) ? 1 : 0;
                for (int x = 0; x < (i >= 4 ? 8 : 16); ++x)
                    if (((x >> (i & 3)) & 1) ^ f) tthr[(size_t)((i >= 4 ? 16 : 0) + x)] *= w.second;
            } else {
                const int i = outbit_[(size_t)b], gi = i / kOutGroup;
                groups |= 1u << gi;
                for (int x = 0; x < 16; ++x)
                    if ((x >> (i % kOutGroup)) & 1) tout[(size_t)(gi * 16 + x)] *= w.second;
            }
        }
        if (own != 1.0) {
            // the factor of q itself goes into the first table there is
            if (!hthr && !groups) hthr = true;
            if (hthr)
                for (int x = 0; x < 16; ++x) tthr[(size_t)x] *= own;
            else
                for (int x = 0; x < 16; ++x) tout[(size_t)(__builtin_ctz(groups) * 16 + x)] *= own;
        }
        uint32_t centre = 7;
        o.km = (RA_ == 64) ? ~0ull : ((1ull << RA_) - 1ull);
        if (!everywhere) {
            if (reg_[(size_t)q] >= 0) {
                if (!flipped(q)) centre = (uint32_t)reg_[(size_t)q];
                o.km = 0;
                for (int k = 0; k < RA_; ++k)
                    if (bit_of(q, k)) o.km |= 1ull << k;
            } else {
                add_cond(&o, q);
            }
        }
        o.arg = centre | (hreg ? 8u : 0u) | (hthr ? 16u : 0u) | (groups << 5);
        o.ra = hreg ? (size_t)RA_ : 0;
        if (hreg) o.tab.insert(o.tab.end(), treg.begin(), treg.end());
        if (hthr) o.tab.insert(o.tab.end(), tthr.begin(), tthr.end());
        for (int gi = 0; gi < kOutGroups; ++gi)
            if ((groups >> gi) & 1u)
                o.tab.insert(o.tab.end(), tout.begin() + gi * 16, tout.begin() + gi * 16 + 16);
        return o;
    }

    // the phase of one pair alone.  complex128: a ramp multiplies every amplitude whose
    // shared qubit is 1, by 1 where the partner is 0, and that FP64 work outlasts the pass
    // (one controlled phase on 27 qubits: 2.34 ms as a ramp, 1.21 by the conditions of both)
    TpOp pair_phase(int a, int b, cplx f)
    {
        TpOp o;
        o.op = IR_PH;
        for (int k = 0; k < RA_; ++k)
            if ((reg_[(size_t)a] < 0 || bit_of(a, k)) && (reg_[(size_t)b] < 0 || bit_of(b, k))) o.km |= 1ull << k;
        if (reg_[(size_t)a] < 0) add_cond(&o, a);
        if (reg_[(size_t)b] < 0) add_cond(&o, b);
        o.place = 1;                       // no further condition: the factor of 1
        o.mat = {1.0, 0.0, f.real(), f.imag()};
        return o;
    }

    // take the pairs of register qubit q out of the pool, into the group's
    // operations before its shears
    void apply_pairs(int q)
    {
        const uint64_t ad = pool.adj[(size_t)q];
        for (int j = 0; j < RB_; ++j)
            if (((queued_ >> j) & 1u) && regq_[(size_t)j] >= 0 && ((ad >> regq_[(size_t)j]) & 1ull)) {
                // that pair came after the queued shears of its other qubit
                close_group();
                break;
            }
        std::vector<std::pair<int, cplx>> ramp;
        for (uint64_t a = pool.adj[(size_t)q]; a; a &= a - 1) {
            const int b = __builtin_ctzll(a);
            const cplx f = pool.take_pair(q, b);
            if (reg_[(size_t)b] >= 0) tab_pair(q, b, f);
            else if (f == -1.0) sign_op(q, b);
            else ramp.push_back({b, f});
        }
        if (ramp.size() == 1 && sizeof(R) == 8) {
            pre_.push_back(pair_phase(q, ramp[0].first, ramp[0].second));
        } else if (!ramp.empty()) {
            pre_.push_back(make_ramp(q, ramp, pool.y[(size_t)q], nullptr, false));
            pool.y[(size_t)q] = 1.0;
        }
    }
    // CZ of register qubit q with qubit b outside the registers
    void sign_op(int q, int b)
    {
        TpOp o;
        o.op = IR_Z;
        o.arg = (1u << reg_[(size_t)q]) | (flipped(q) ? 64u : 0u);
        add_cond(&o, b);
        pre_.push_back(o);
        zdirty_ = true;
    }

    bool rotation(const SGate &g)
    {
        cplx p, q, y;
        double t;
        bool swap;
        if (!split_unitary(g.m, &p, &q, &y, &t, &swap)) return false;
        const int x = g.target, j = reg_[(size_t)x];
        if ((queued_ >> j) & 1u) close_group();
        pool.y[(size_t)x] *= y;
        apply_pairs(x);                 // may fold pool.y[x] into a ramp
        // a real factor passes through the shears (they are scaled by it); a
        // complex one is a real factor times a phase of at most a quarter turn
        const cplx rho = pool.y[(size_t)x];
        const double mod = rho.imag() == 0.0 ? std::abs(rho.real()) : std::abs(rho);
        double r = 1.0;
        if (mod >= 0.5 && mod <= 2.0) {
            r = rho.real() < 0.0 ? -mod : mod;
            if (rho.imag() != 0.0) tab_single(x, rho / r);
        } else {
            tab_single(x, rho);
        }
        pool.y[(size_t)x] = 1.0;
        t = (double)(R)t;
        // the physical matrix: labels exchanged when the qubit is flipped
        const bool f = flipped(x);
        double rp = r, e = f ? -1.0 : 1.0, h = 1.0;   // h: a common factor
        if (f) { rp = 1.0 / r; h = r; }
        cplx P0 = h * (f ? q : p), P1 = h * (f ? p : q);
        const double d = 1.0 + t * t;
        double a, b;
        if (!swap) {
            a = -e * t;
            b = e * t / d;
            P1 *= d * rp;
        } else {
            a = e * t;
            b = -e * t / d;
            // register 0 now holds e * (value 1), register 1 -value 0 / (e d)
            P0 *= -e * d * rp;
            P1 *= e;
            flip_ ^= 1ull << x;
        }
        sa_[j] = (double)(R)(a * rp);
        sb_[j] = (double)(R)(b / rp);
        queued_ |= 1u << j;
        const cplx f0 = f ? P1 : P0, f1 = f ? P0 : P1;
        pool.g *= f0;
        pool.y[(size_t)x] = f1 / f0;
        if (std::norm(p) + std::norm(q) < 0.5 || std::norm(p) + std::norm(q) > 8.0) close_group();   // a scaled matrix: its scale does not wait
        return true;
    }

    // an uncontrolled matrix that is not unitary to FP64 rounding (entries
    // given in single precision, say): complex shears, which also take the
    // pool's factor of the qubit
    bool shears(const SGate &g)
    {
        const int x = g.target, j = reg_[(size_t)x], fl = flipped(x) ? 1 : 0;
        double m[8];
        for (int i = 0; i < 2; ++i)
            for (int l = 0; l < 2; ++l)
                for (int c = 0; c < 2; ++c) m[2 * (2 * i + l) + c] = g.m[2 * (2 * (i ^ fl) + (l ^ fl)) + c];
        cplx p, q, a, b;
        bool swap;
        if (!split_general(m, &p, &q, &a, &b, &swap)) return false;
        close_group();
        apply_pairs(x);
        cplx rho = pool.y[(size_t)x], h = 1.0;
        if (std::abs(rho) < 0.5 || std::abs(rho) > 2.0) {
            tab_single(x, rho);
            rho = 1.0;
        }
        pool.y[(size_t)x] = 1.0;
        close_group();
        if (fl) {
            h = rho;
            rho = 1.0 / rho;
        }
        TpOp o;
        o.op = IR_CSHEARS;
        o.arg = (uint32_t)j;
        o.tab = {a * rho, b / rho};
        emit(o);
        // registers 0 and 1 hold p^-1 and (q rho)^-1 times the (row-exchanged) result
        cplx P0 = h * p, P1 = h * q * rho;
        if (swap) {
            std::swap(P0, P1);
            flip_ ^= 1ull << x;
        }
        const cplx f0 = fl ? P1 : P0, f1 = fl ? P0 : P1;
        pool.g *= f0;
        const cplx left = f1 / f0;
        if (std::abs(left) < 0.5 || std::abs(left) > 2.0) tab_single(x, left);   // not kept aside
        else pool.y[(size_t)x] = left;
        close_group();
        return true;
    }

    // exchange gates the shears do not cover: controlled gates and matrices
    // that are not unitary
    void masked_exchange(const SGate &g)
    {
        const int x = g.target;
        close_group();
        if (g.op == OP_XPERM && __builtin_popcountll(g.ctrl) == 1) {
            // signs move through a CNOT: Z on the target becomes Z on both
            const int c = __builtin_ctzll(g.ctrl);
            if (pool.y[(size_t)x] == -1.0) pool.y[(size_t)c] *= -1.0;
            else if (pool.y[(size_t)x] != 1.0) fold_target(x);
            for (uint64_t a = pool.adj[(size_t)x]; a; a &= a - 1) {
                const int b = __builtin_ctzll(a);
                if (pool.pair(x, b) != -1.0) continue;
                if (b == c) pool.y[(size_t)c] *= -1.0;
                else pool.mul_pair(c, b, -1.0);
            }
            uint64_t keep = 0;
            for (uint64_t a = pool.adj[(size_t)x]; a; a &= a - 1)
                if (pool.pair(x, __builtin_ctzll(a)) == -1.0) keep |= a & (~a + 1);
            if (keep != pool.adj[(size_t)x]) {
                // the other pairs are applied; the signs stay aside meanwhile
                for (uint64_t a = keep; a; a &= a - 1) pool.take_pair(x, __builtin_ctzll(a));
                const cplx ys = pool.y[(size_t)x];
                pool.y[(size_t)x] = 1.0;
                apply_pairs(x);
                pool.y[(size_t)x] = ys;
                for (uint64_t a = keep; a; a &= a - 1) pool.mul_pair(x, __builtin_ctzll(a), -1.0);
                close_group_for(x);
            }
        } else {
            apply_pairs(x);
            if (pool.y[(size_t)x] != 1.0) fold_target(x);
        }
        close_group_for(x);
        flush_signs();
        TpOp o;
        o.op = IR_XCH;
        const int j = reg_[(size_t)x];
        const int kind = (g.op == OP_DENSE) ? SK_DENSE : (g.op == OP_ANTIDIAG) ? SK_ANTI : SK_XPERM;
        o.arg = (uint32_t)(j | (kind << 3));
        o.km = 0;
        for (int k = 0; k < RA_; ++k) {
            bool on = true;
            for (uint64_t a = g.ctrl; a && on; a &= a - 1) {
                const int c = __builtin_ctzll(a);
                if (reg_[(size_t)c] >= 0) on = bit_of(c, k) != 0;
            }
            if (on) o.km |= 1ull << k;
        }
        for (uint64_t a = g.ctrl; a; a &= a - 1) {
            const int c = __builtin_ctzll(a);
            if (reg_[(size_t)c] < 0) add_cond(&o, c);
        }
        const int fl = flipped(x) ? 1 : 0;
        for (int i = 0; i < 2; ++i)
            for (int l = 0; l < 2; ++l)
                for (int c = 0; c < 2; ++c) o.mat.push_back(g.m[2 * (2 * (i ^ fl) + (l ^ fl)) + c]);
        emit(o);
    }
    void fold_target(int x)
    {
        tab_single(x, pool.y[(size_t)x]);
        pool.y[(size_t)x] = 1.0;
    }
    // close the group without letting its table take x's remaining entries
    // (signs that have already been moved through the exchange)
    void close_group_for(int x)
    {
        if (!tab_used_) {
            close_group();
            return;
        }
        const cplx ys = pool.y[(size_t)x];
        const uint64_t ad = pool.adj[(size_t)x];
        std::vector<std::pair<int, cplx>> keep;
        pool.y[(size_t)x] = 1.0;
        for (uint64_t a = ad; a; a &= a - 1) {
            const int b = __builtin_ctzll(a);
            keep.push_back({b, pool.take_pair(x, b)});
        }
        // entries moved onto the control are after the exchange too, but they
        // do not involve x and commute with it
        close_group();
        pool.y[(size_t)x] = ys;
        for (const auto &k : keep) pool.mul_pair(x, k.first, k.second);
    }

    void diagonal(const SGate &g)
    {
        const int nc = __builtin_popcountll(g.ctrl);
        const cplx a = (g.op == OP_DIAG) ? cplx(g.m[0], g.m[1]) : cplx(1.0), d(g.m[6], g.m[7]);
        const int x = g.target;
        if (nc == 0 ? takes(a, d) : nc == 1 && unit_factor(a) && unit_factor(d)) {
            const cplx ratio = (a == 1.0) ? d : d / a;
            if (nc == 0) {
                pool.g *= a;
                pool.y[(size_t)x] *= ratio;
            } else {
                const int c = __builtin_ctzll(g.ctrl);
                if (a != 1.0) pool.y[(size_t)c] *= a;
                pool.mul_pair(c, x, ratio);
            }
            return;
        }
        // two controls, or factors the pool does not hold: applied where it stands
        close_group();
        TpOp o;
        uint64_t regs = 0;
        for (uint64_t m = g.ctrl; m; m &= m - 1) {
            const int c = __builtin_ctzll(m);
            if (reg_[(size_t)c] >= 0) regs |= 1ull << c;
            else add_cond(&o, c);
        }
        const bool neg = g.op == OP_DIAG_HI && d == -1.0;
        if (neg && __builtin_popcountll(regs) + (reg_[(size_t)x] >= 0 ? 1 : 0) <= 1) {
            o.op = IR_Z;
            if (reg_[(size_t)x] >= 0) regs |= 1ull << x;
            else add_cond(&o, x);
            if (regs) {
                const int q = __builtin_ctzll(regs);
                o.arg = (1u << reg_[(size_t)q]) | (flipped(q) ? 64u : 0u);
            } else {
                o.arg = 64u;
            }
            emit(o);
            zdirty_ = true;
            return;
        }
        o.op = IR_PH;
        o.km = 0;
        for (int k = 0; k < RA_; ++k) {
            bool on = true;
            for (uint64_t m = regs; m && on; m &= m - 1) on = bit_of(__builtin_ctzll(m), k) != 0;
            if (on) o.km |= 1ull << k;
        }
        if (reg_[(size_t)x] >= 0) {
            for (int k = 0; k < RA_; ++k)
                if (bit_of(x, k)) o.km_t |= 1ull << k;
        } else {
            TpOp t;
            add_cond(&t, x);
            o.thr_t = t.thr;
            o.out_t = t.out;
            o.place = 1;
        }
        o.mat = {a.real(), a.imag(), d.real(), d.imag()};
        emit(o);
    }

    // everything left in the pool, in the current layout
    void final_pool(bool unit_ok)
    {
        final_ = true;
        auto unit = [](cplx f) { return std::abs(std::abs(f) - 1.0) <= 1e-12; };
        if (unit_ok) {
            bool all = true;
            for (int q = 0; q < n_ && all; ++q) {
                all = unit(pool.y[(size_t)q]);
                for (uint64_t a = pool.adj[(size_t)q]; a && all; a &= a - 1) all = unit(pool.pair(q, __builtin_ctzll(a)));
            }
            if (all) {
                for (int q = 0; q < n_; ++q) {
                    pool.y[(size_t)q] = 1.0;
                    while (pool.adj[(size_t)q]) pool.take_pair(q, __builtin_ctzll(pool.adj[(size_t)q]));
                }
                pool.g = std::abs(pool.g);
                if (!unit(pool.g)) emit_scale(pool.g.real());
                pool.g = 1.0;
                return;
            }
        }
        // signs with at most one register qubit, then the stars of the other
        // pairs (around the qubit with the most of them, registers first)
        for (int a = 0; a < n_; ++a)
            for (uint64_t m = pool.adj[(size_t)a] & ~((2ull << a) - 1ull); m; m &= m - 1) {
                const int b = __builtin_ctzll(m);
                if (pool.pair(a, b) != -1.0 || (reg_[(size_t)a] >= 0 && reg_[(size_t)b] >= 0)) continue;
                pool.take_pair(a, b);
                if (reg_[(size_t)a] >= 0) {
                    sign_op(a, b);
                } else if (reg_[(size_t)b] >= 0) {
                    sign_op(b, a);
                } else {
                    TpOp o;
                    o.op = IR_Z;
                    o.arg = 64u;
                    add_cond(&o, a);
                    add_cond(&o, b);
                    pre_.push_back(o);
                    zdirty_ = true;
                }
            }
        for (;;) {
            int best = -1, bestc = 0;
            for (int q = 0; q < n_; ++q) {
                int c = 0;
                for (uint64_t a = pool.adj[(size_t)q]; a; a &= a - 1)
                    if (reg_[(size_t)q] < 0 || reg_[(size_t)__builtin_ctzll(a)] < 0) c += 2;
                if (c && reg_[(size_t)q] >= 0) ++c;
                if (c > bestc) { bestc = c; best = q; }
            }
            if (best < 0) break;
            std::vector<std::pair<int, cplx>> with;
            for (uint64_t a = pool.adj[(size_t)best]; a; a &= a - 1) {
                const int b = __builtin_ctzll(a);
                if (reg_[(size_t)best] >= 0 && reg_[(size_t)b] >= 0) continue;   // the table's
                with.push_back({b, pool.take_pair(best, b)});
            }
            if (with.size() == 1 && sizeof(R) == 8) {
                pre_.push_back(pair_phase(best, with[0].first, with[0].second));
                continue;
            }
            pre_.push_back(make_ramp(best, with, pool.y[(size_t)best], nullptr, false));
            pool.y[(size_t)best] = 1.0;
        }
        // what is left lies on single qubits and inside the registers
        std::vector<std::pair<int, cplx>> singles;
        for (int q = 0; q < n_; ++q) {
            if (reg_[(size_t)q] >= 0) {
                if (pool.y[(size_t)q] != 1.0) tab_single(q, pool.y[(size_t)q]);
                for (uint64_t a = pool.adj[(size_t)q]; a; a &= a - 1) {
                    const int b = __builtin_ctzll(a);
                    tab_pair(q, b, pool.take_pair(q, b));
                }
            } else if (pool.y[(size_t)q] != 1.0) {
                singles.push_back({q, pool.y[(size_t)q]});
            }
            pool.y[(size_t)q] = 1.0;
        }
        if (pool.g != 1.0) tab_used_ = true;
        for (cplx &c : tab_) c *= pool.g;
        pool.g = 1.0;
        if (!singles.empty()) {
            pre_.push_back(make_ramp(-1, singles, 1.0, tab_used_ ? &tab_ : nullptr, true));
            tab_.assign((size_t)RA_, 1.0);
            tab_used_ = false;
        }
        close_group();
    }
};

// Predicted time of a pass in microseconds on 2^26 amplitudes, from timings of
// each operation alone (26 qubits, one tile size per type: 13 qubits complex64,
// 12 qubits complex128, whose arithmetic is bound by the FP64 pipe).
template <typename R>
double pass_cost(const TilePass &tp)
{
    constexpr bool D = sizeof(R) == 8;
    double t = D ? 320.0 : 130.0;                 // load and store
    for (const TpOp &o : tp.ops) {
        switch (o.op) {
        case IR_Z: t += 0.4; break;
        case IR_DIAG: t += (o.arg & 7u) == GD_REAL ? (D ? 215.0 : 2.0) : (o.arg & 7u) == GD_HALF ? (D ? 160.0 : 4.0) : (D ? 430.0 : 11.0); break;
        case IR_SHEARS: t += 3.3 + (D ? 215.0 : 5.2) * __builtin_popcount(o.arg); break;
        case IR_FLUSH: t += D ? 15.0 : 6.5; break;
        case IR_LAYOUT: t += D ? 45.0 : 20.0; break;
        case IR_PERM: t += D ? 80.0 : 37.0; break;
        case IR_RAMP: t += D ? 400.0 : 23.0; break;
        case IR_CSHEARS: t += D ? 430.0 : 12.0; break;
        case IR_XCH: t += ((o.arg >> 3) & 3u) == SK_XPERM ? 18.0 : ((o.arg >> 3) & 3u) == SK_DENSE && D ? 800.0 : 50.0; break;
        default: t += D ? 400.0 : 18.0; break;
        }
    }
    return t;
}

// ---------------------------------------------------------------- packing
template <typename R>
class Packer {
public:
    explicit Packer(std::vector<uint32_t> *out) : out_(out), first_(out->size()) {}

    // Consecutive operations that fit the order of a group become one; ramps
    // commute with the signs and the diagonal of an open group and go first.
    void run(const std::vector<TpOp> &ops)
    {
        std::vector<const TpOp *> grp;
        int stage = -1, nz = 0;
        auto close = [&]() {
            if (!grp.empty()) group(grp);
            grp.clear();
            stage = -1;
            nz = 0;
        };
        for (const TpOp &o : ops) {
            if (o.op > IR_LAYOUT) {
                if (!(o.op == IR_RAMP && stage <= IR_DIAG)) close();
                single(o);
                continue;
            }
            const bool joins = o.op == IR_Z ? stage <= IR_DIAG && nz < 31 : o.op > stage;
            if (!joins) close();
            if (o.op == IR_Z) ++nz;
            grp.push_back(&o);
            stage = std::max(stage, o.op);
        }
        close();
        w_.assign(4, 0u);
        put(w_, TP_END);
    }

private:
    std::vector<uint32_t> *out_;
    size_t first_;
    bool dirty_ = false;           // signs may be pending
    std::vector<uint32_t> w_;      // the operation being packed

    static void real(std::vector<uint32_t> *w, double v)
    {
        const R r = (R)v;
        const size_t at = w->size();
        w->resize(at + sizeof(R) / 4);
        memcpy(w->data() + at, &r, sizeof r);
    }
    static void table(std::vector<uint32_t> *w, const std::vector<cplx> &t)
    {
        for (const cplx &c : t) {
            real(w, c.real());
            real(w, c.imag());
        }
        while (w->size() % 4) w->push_back(0u);
    }
    // a factor per register (see ctable_units)
    static void registers(std::vector<uint32_t> *w, const cplx *t, size_t cnt)
    {
        const size_t at = w->size();
        if constexpr (sizeof(R) == 8) {
            w->resize(at + 4 * cnt);
            memcpy(w->data() + at, t, 16 * cnt);
        } else {
            w->resize(at + 3 * cnt);
            float *f = reinterpret_cast<float *>(w->data() + at);
            for (size_t k = 0; k < cnt; k += 2) {
                f[2 * k] = (float)t[k].real();
                f[2 * k + 1] = (float)t[k + 1].real();
                f[2 * k + 2] = (float)t[k].imag();
                f[2 * k + 3] = (float)t[k + 1].imag();
                f[2 * cnt + k] = -(float)t[k].imag();
                f[2 * cnt + k + 1] = -(float)t[k + 1].imag();
            }
        }
    }
    void put(std::vector<uint32_t> &w, uint32_t head)
    {
        while (w.size() % 4) w.push_back(0u);
        const size_t len = w.size() / 4;
        w[0] = head | ((uint32_t)len << 4);
        // an operation and the header after it stay inside one chunk
        auto units = [&]() { return (out_->size() - first_) / 4; };
        if (units() % kChunkUnits + len + 1 > kChunkUnits) {
            out_->push_back(TP_CHUNK | (1u << 4));
            while ((out_->size() - first_) % (4 * kChunkUnits)) out_->push_back(0u);
        }
        out_->insert(out_->end(), w.begin(), w.end());
    }
    void group(const std::vector<const TpOp *> &ops)
    {
        std::vector<uint32_t> &w = w_;
        w.assign(4, 0u);
        uint32_t head = TP_GROUP, nz = 0;
        for (const TpOp *o : ops)
            if (o->op == IR_Z) {
                w.push_back(o->thr | (o->arg << 16));
                w.push_back(o->out);
                ++nz;
                dirty_ = true;
            }
        while (w.size() % 4) w.push_back(0u);
        head |= nz << 24;
        for (const TpOp *o : ops) {
            if (o->op == IR_DIAG) {
                head |= o->arg << 12;
                if ((o->arg & 7u) == GD_REAL) {
                    for (const cplx &c : o->tab) real(&w, c.real());
                } else if ((o->arg & 7u) == GD_HALF) {
                    table(&w, o->tab);
                } else {
                    registers(&w, o->tab.data(), o->tab.size());
                }
            } else if (o->op == IR_SHEARS) {
                head |= (o->arg << 18) | (dirty_ ? 1u << 29 : 0u);
                table(&w, o->tab);
            } else if (o->op == IR_FLUSH) {
                head |= 1u << 30;
                dirty_ = false;
            } else if (o->op == IR_LAYOUT) {
                w[1] = o->arg;
                head |= 1u << 31;
            }
        }
        put(w, head);
    }
    void single(const TpOp &o)
    {
        std::vector<uint32_t> &w = w_;
        w.assign(4, 0u);
        w[1] = o.thr;
        w[2] = o.out;
        w[3] = o.place;
        if (o.op == IR_RAMP || o.op == IR_XCH || o.op == IR_PH)
            w.insert(w.end(), {(uint32_t)o.km, (uint32_t)(o.km >> 32), (uint32_t)o.km_t, (uint32_t)(o.km_t >> 32)});
        if (o.op == IR_PH) w.insert(w.end(), {o.thr_t, o.out_t, 0u, 0u});
        w.insert(w.end(), o.words.begin(), o.words.end());
        for (double v : o.mat) real(&w, v);
        if (o.op == IR_RAMP && (o.arg & 8u)) {
            registers(&w, o.tab.data(), o.ra);
            table(&w, std::vector<cplx>(o.tab.begin() + (long)o.ra, o.tab.end()));
        } else {
            table(&w, o.tab);
        }
        static const uint32_t code[] = {TP_RAMP, TP_XCH, TP_PH, TP_CSHEARS, TP_PERM};
        put(w, code[o.op - IR_RAMP] | (o.arg << 12));
    }
};

template <typename R>
void pack_program(const TilePass &tp, std::vector<uint32_t> *out)
{
    Packer<R>(out).run(tp.ops);
}

// Order and layouts of one pass's gates.  Diagonal gates and X run as soon as
// the gates before them have (the pool and the labels take them); masked
// exchanges as soon as a register holds their target; rotations in groups --
// all that are ready in one layout -- choosing the layout that costs least
// per rotation: a group costs a diagonal table, another layout a trip through
// shared memory.
template <typename R>
void schedule_pass(TileCompiler<R> &tc, const Pass &ps, const std::vector<SGate> &g, int M, int VEC)
{
    const int RB = M - kTpThrBits, NL = n_layouts(M, RB);
    const size_t P = ps.members.size();
    enum { DIAG, LABEL, ROT, MASKED };
    std::vector<uint8_t> kind(P), lmask(P, 0);
    std::vector<int> indeg(P, 0);
    int lastx[64], since[64];              // per qubit: last exchange, list of the diagonal gates after it
    for (int q = 0; q < 64; ++q) lastx[q] = since[q] = -1;
    struct Link { int item, next; };
    std::vector<Link> links;               // the lists: successors of a gate, diagonal gates of a qubit
    links.reserve(8 * P);
    std::vector<int> succ(P, -1);
    uint8_t lq[64];
    for (int q = 0; q < 64; ++q) lq[q] = 0;
    auto layouts_of = [&](int local) {
        uint8_t m = 0;
        for (int l = 0; l < NL; ++l)
            if (is_reg(M, RB, VEC, l, local)) m |= (uint8_t)(1 << l);
        return m;
    };
    for (int q = 0; q < kLow; ++q) lq[q] = layouts_of(q);
    for (size_t i = 0; i < ps.high.size(); ++i) lq[ps.high[i]] = layouts_of(kLow + (int)i);
    auto edge = [&](int a, int b) {
        links.push_back(Link{b, succ[(size_t)a]});
        succ[(size_t)a] = (int)links.size() - 1;
        ++indeg[(size_t)b];
    };
    for (size_t i = 0; i < P; ++i) {
        const SGate &s = g[(size_t)ps.members[i]];
        const uint64_t x = s.xq(), d = s.dq();
        if (!x) kind[i] = DIAG;
        else if (!s.ctrl) kind[i] = (s.op == OP_XPERM || s.op == OP_SWAP) ? LABEL : ROT;
        else kind[i] = MASKED;
        if (x) lmask[i] = lq[s.target];
        for (uint64_t m = d; m; m &= m - 1) {
            const int q = __builtin_ctzll(m);
            if (lastx[q] >= 0) edge(lastx[q], (int)i);
            links.push_back(Link{(int)i, since[q]});
            since[q] = (int)links.size() - 1;
        }
        for (uint64_t m = x; m; m &= m - 1) {
            const int q = __builtin_ctzll(m);
            if (lastx[q] >= 0 && since[q] < 0) edge(lastx[q], (int)i);
            for (int l = since[q]; l >= 0; l = links[(size_t)l].next) {
                const int before = links[(size_t)l].item;   // (edge grows links)
                edge(before, (int)i);
            }
            since[q] = -1;
            lastx[q] = (int)i;
        }
    }
    std::vector<int> ready, now;
    for (size_t i = 0; i < P; ++i)
        if (!indeg[i]) ready.push_back((int)i);
    auto done = [&](int i) {
        for (int l = succ[(size_t)i]; l >= 0; l = links[(size_t)l].next)
            if (--indeg[(size_t)links[(size_t)l].item] == 0) ready.push_back(links[(size_t)l].item);
    };
    auto run = [&](int i, int l) {
        tc.gate(g[(size_t)ps.members[(size_t)i]], l);
        done(i);
    };
    while (!ready.empty()) {
        const int cur = tc.current_layout();
        // everything that is free, then the masked exchanges of this layout
        bool any = false;
        for (size_t r = 0; r < ready.size();) {
            const int i = ready[r];
            if (kind[(size_t)i] <= LABEL) {
                ready.erase(ready.begin() + (long)r);
                run(i, cur);
                any = true;
            } else {
                ++r;
            }
        }
        if (any) continue;
        for (size_t r = 0; r < ready.size() && !any; ++r) {
            const int i = ready[r];
            if (kind[(size_t)i] == MASKED && ((lmask[(size_t)i] >> cur) & 1)) {
                ready.erase(ready.begin() + (long)r);
                run(i, cur);
                any = true;
            }
        }
        if (any) continue;
        int best = cur;
        double best_score = -1.0;
        for (int l = 0; l < NL; ++l) {
            int nrot = 0, nmask = 0;
            for (int i : ready)
                if ((lmask[(size_t)i] >> l) & 1) (kind[(size_t)i] == ROT ? nrot : nmask)++;
            if (!nrot && !nmask) continue;
            const double cost = (l != cur ? kCostLayout : 0.0) + (nrot ? kCostGroup + (nrot > 1 ? 4.0 : 2.0) + nrot : 0.0) +
                                5.0 * nmask;
            const double score = (nrot + nmask) / cost;
            if (score > best_score + 1e-12 || (l == cur && score > best_score - 1e-12)) { best_score = score; best = l; }
        }
        now.clear();
        for (size_t r = 0; r < ready.size();) {
            const int i = ready[r];
            if (kind[(size_t)i] == ROT && ((lmask[(size_t)i] >> best) & 1)) {
                now.push_back(i);
                ready.erase(ready.begin() + (long)r);
            } else {
                ++r;
            }
        }
        if (now.empty()) {
            tc.set_layout(best);          // masked exchanges follow
            continue;
        }
        for (int i : now) run(i, best);
    }
}

// The passes of a circuit as tile programs: every pass that has something to
// run, with its packed words.  Diagonal gates wait in the pool for the pass
// that needs them, so passes of diagonal gates alone vanish; whatever is left
// is applied in the last pass that runs.
struct Program {
    Pass pass;
    TilePass tp;
    std::vector<uint32_t> words;
    std::vector<int> members;       // lowered gates this pass accounts for
};

// where a pass's tiles lie
inline TileGeom tile_geom(const Pass &ps, int n)
{
    TileGeom geo;
    memset(&geo, 0, sizeof geo);
    uint64_t q = (1ull << kLow) - 1ull;
    for (size_t i = 0; i < ps.high.size(); ++i) {
        geo.hpos[i] = ps.high[i];
        q |= 1ull << ps.high[i];
    }
    for (int b = 0; b < n; ++b)
        if (!((q >> b) & 1)) geo.outer_pos[geo.n_outer++] = b;
    return geo;
}

// One pass after the other, so that a caller can launch the first ones while
// it plans the rest.  probabilities_only: see TileCompiler::end.
template <typename R>
class TilePlanner {
public:
    TilePlanner(const std::vector<SGate> &g, int n, int M, int VEC, bool probabilities_only = false, bool pack = true)
        : g_(g), former_(g, n, M), tc_(n, M, VEC), M_(M), VEC_(VEC), prob_(probabilities_only), pack_(pack) {}

    bool next(Program *out)
    {
        for (;;) {
            Pass ps;
            if (!former_.next(&ps)) return false;
            tc_.begin(ps);
            schedule_pass(tc_, ps, g_, M_, VEC_);
            waiting_.insert(waiting_.end(), ps.members.begin(), ps.members.end());
            std::vector<int> left;
            const bool last = former_.only_diagonal_left(&left);
            if (last) {
                for (int m : left) tc_.gate(g_[(size_t)m], tc_.current_layout());
                waiting_.insert(waiting_.end(), left.begin(), left.end());
                former_.finish();
            }
            Program pr;
            pr.tp = tc_.end(last, prob_);
            if (!last && pr.tp.ops.empty() && pr.tp.flip == 0) continue;
            if (pack_) pack_program<R>(pr.tp, &pr.words);
            pr.pass = std::move(ps);
            pr.members.swap(waiting_);
            *out = std::move(pr);
            return true;
        }
    }

private:
    const std::vector<SGate> &g_;
    PassFormer former_;
    TileCompiler<R> tc_;
    int M_, VEC_;
    bool prob_, pack_;
    std::vector<int> waiting_;
};

template <typename R>
std::vector<Program> compile_passes(const std::vector<SGate> &g, int n, int M, int VEC, bool probabilities_only = false)
{
    std::vector<Program> out;
    TilePlanner<R> tp(g, n, M, VEC, probabilities_only);
    Program p;
    while (tp.next(&p)) out.push_back(std::move(p));
    return out;
}

}  // namespace
}  // namespace qsim
