// reduce.cu -- state initialisation, probabilities, FP64 reductions,
// single-qubit collapse and shot sampling.
//
// Probabilities are |a_j|^2 (App. B.3).  Every sum of probabilities (norm,
// the two halves of a single-qubit measurement, <sum Z>, the sampling CDF) is
// accumulated in FP64 over a fixed grid and a fixed tree, so results are
// bit-reproducible run to run.  complex128 squares are FP64 FMAs; complex64
// squares are exact FP32 products summed with compensation in short chunks
// that are carried into FP64 (see "compensated FP32 sums of squares").
//
// Sampling (§2.4: many outcomes from one state without re-running the gates)
// is an inverse CDF over the FP64 prefix of |a_j|^2 that is never
// materialised for the whole state: sums per sub-block of 256 amplitudes and
// per block of 32 sub-blocks (one read of the state), one scan over the block
// sums, then per shot a search of the block, of the sub-block, of its eighth
// and of the amplitude (256 bytes of complex64 per shot, or 2 KB where the pass has not
// written the sums of the eighths, instead of the whole block).
#include <cmath>

#include "f32x2.cuh"
#include "internal.cuh"

namespace qsim {

namespace {

// ---------------------------------------------------------------- SplitMix64
// Steele, Lea & Flood, OOPSLA 2014: add the golden gamma, then the variant-13
// finaliser.  Uniform draw u = (x >> 11) * 2^-53.
__host__ __device__ __forceinline__ uint64_t smix(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}
__host__ __device__ __forceinline__ double unif(uint64_t seed, uint64_t s)
{
    return (double)(smix(seed + s) >> 11) * 0x1.0p-53;
}

// ---------------------------------------------------------------- init
// Zero the state with 16-byte stores and write amplitude j = 1.
__global__ void k_init_basis(uint4 *__restrict__ st, uint64_t nvec, uint64_t jvec, uint4 jval)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvec;
         i += (uint64_t)gridDim.x * blockDim.x)
        st[i] = (i == jvec) ? jval : make_uint4(0, 0, 0, 0);
}

// ---------------------------------------------------------------- block reduce
template <int NT>
__device__ __forceinline__ void block_sum2(double &a, double &b, double *sh)
{
    // fixed-order tree: warp butterflies, then warp 0 over the warp results
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) { sh[2 * w] = a; sh[2 * w + 1] = b; }
    __syncthreads();
    if (w == 0) {
        a = (l < NT / 32) ? sh[2 * l] : 0.0;
        b = (l < NT / 32) ? sh[2 * l + 1] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
    }
    __syncthreads();
}

template <typename R>
__device__ __forceinline__ double sq(R re, R im)
{
    const double r = (double)re, i = (double)im;
    return fma(r, r, i * i);
}

// FP32 -> FP64 with integer operations (the FP64 pipe of this GPU is narrow,
// so the conversion would cost as much as the arithmetic): a normal float is
// widened exactly by rebiasing the exponent (127 -> 1023) and shifting the
// mantissa; zero and subnormals become 0 (their squares are below 1e-76 and
// do not change an FP64 sum of probabilities); states hold no inf / NaN.
__device__ __forceinline__ double widen(float f)
{
    const uint32_t u = __float_as_uint(f);
    const uint32_t e = (u >> 23) & 0xFFu;
    const uint64_t d = ((uint64_t)(u & 0x80000000u) << 32) | ((uint64_t)(e + 896u) << 52) |
                       ((uint64_t)(u & 0x007FFFFFu) << 29);
    return e ? __longlong_as_double((long long)d) : 0.0;
}

template <>
__device__ __forceinline__ double sq<float>(float re, float im)
{
    const double r = widen(re), i = widen(im);
    return fma(r, r, i * i);
}


// a += |re + i im|^2 as two FP64 FMAs (both squares exact in FP64 for a
// complex64 amplitude)
template <typename R>
__device__ __forceinline__ void acc_sq(double &a, R re, R im)
{
    const double r = (double)re, i = (double)im;
    a = fma(r, r, a);
    a = fma(i, i, a);
}
template <>
__device__ __forceinline__ void acc_sq<float>(double &a, float re, float im)
{
    const double r = widen(re), i = widen(im);
    a = fma(r, r, a);
    a = fma(i, i, a);
}

// ---------------------------------------------------------------- compensated FP32 sums of squares
// The FP64 pipe of this GPU runs at about 1/64 of the FP32 rate, so two FP64
// FMAs per complex64 amplitude make a sum of |a|^2 FP64-bound, at about 2.7x
// the time it takes to read the state.  The complex64 reductions therefore
// take their squares and partial sums with error-free FP32 transformations and
// carry them into FP64 once per 8 amplitudes (16 squares):
//  * a chunk is rescaled by an exact power of two 2^(127 - k), k the exponent
//    of its largest component, so that no square overflows or is lost to
//    underflow (the scaling is undone exactly in the FP64 exponent);
//  * x^2 = h + l exactly, with h = fl(x * x) and l = fma(x, x, -h) (Dekker's
//    product, formed with an FMA); h enters the running sum s through Knuth's
//    TwoSum (s + h = t + err exactly), and err + l accumulate in e: the Dot2
//    scheme of Ogita, Rump & Oishi (SIAM J. Sci. Comput. 26(6), 2005);
//  * for m non-negative terms |(s + e) - sum| <= (m + 1)^2 u^2 sum (u = 2^-24,
//    m = 16: about 1e-12 relative in the worst case, where every rounding
//    error takes its maximum with the same sign; around 1e-15 in practice);
//  * s and e widen to FP64 exactly.
// The __f*_rn intrinsics keep the compiler from contracting a product and a
// sum into one FMA, which would break the exactness of the transformations.
struct Sq32 {
    float s = 0.f, e = 0.f;                  // value = s + e
    __device__ __forceinline__ void two_sum(float h)
    {
        const float t = __fadd_rn(s, h);
        const float z = __fsub_rn(t, s);
        const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(h, z));
        s = t;
        e = __fadd_rn(e, err);
    }
    // += x^2
    __device__ __forceinline__ void add_sq(float x)
    {
        const float h = __fmul_rn(x, x);
        const float l = __fmaf_rn(x, x, -h);
        const float t = __fadd_rn(s, h);
        const float z = __fsub_rn(t, s);
        const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(h, z));
        s = t;
        e = __fadd_rn(e, __fadd_rn(err, l));
    }
    // += a square as split by square2: h = -nh, l
    __device__ __forceinline__ void add_split(float nh, float l)
    {
        const float t = __fsub_rn(s, nh);
        const float z = __fsub_rn(t, s);
        const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(-nh, z));
        s = t;
        e = __fadd_rn(e, __fadd_rn(err, l));
    }
    // += x * w (w a small integer; the product is split exactly like a square)
    __device__ __forceinline__ void add_prod(float x, float w)
    {
        const float h = __fmul_rn(x, w);
        const float l = __fmaf_rn(x, w, -h);
        two_sum(h);
        e = __fadd_rn(e, l);
    }
};

// The same in packs, for the two components of an amplitude at once (an
// addition as a multiply-add with 1 or -1: the same rounding).
struct Split2 {
    pack2 nh, l;               // x^2 = l - nh
};
__device__ __forceinline__ Split2 square2(pack2 x, pack2 c, pack2 nc)      // of c x; nc = -c
{
    const pack2 y = mul2(x, c);
    Split2 r;
    r.nh = mul2(y, mul2(x, nc));
    r.l = fma2(y, y, r.nh);
    return r;
}
struct Sum2 {
    pack2 s = 0, e = 0;
    __device__ __forceinline__ void add_split(pack2 nh, pack2 l)
    {
        const pack2 one = dup(1.f), neg = dup(-1.f);
        const pack2 t = fma2(nh, neg, s);
        const pack2 z = fma2(s, neg, t);
        const pack2 a = fma2(fma2(z, neg, t), neg, s);         // s - (t - z)
        const pack2 err = fma2(fma2(z, one, nh), neg, a);      // a + (h - z)
        s = t;
        e = fma2(fma2(err, one, l), one, e);
    }
    // += x * w, componentwise
    __device__ __forceinline__ void add_weighted(const Sum2 &x, float w)
    {
        const pack2 w2 = dup(w);
        const pack2 nh = mul2(x.s, dup(-w));
        add_split(nh, fma2(x.s, w2, nh));
        e = fma2(x.e, w2, e);
    }
    __device__ __forceinline__ Sq32 total() const
    {
        const float2 a = unpk(s), b = unpk(e);
        Sq32 r;
        r.s = a.x;
        r.e = __fadd_rn(b.x, b.y);
        r.two_sum(a.y);
        return r;
    }
};

// Exact power-of-two rescaling of a chunk.  amax = the largest |component|;
// k = its biased exponent clamped to [1, 253], so 2^(127 - k) is a normal float
// and the largest scaled component lies in [1, 2) (k = 1 covers zero and
// subnormal chunks).  Squares of the scaled chunk are the true squares times
// 2^-sh, with sh = 2 (k - 127).
struct Pow2 {
    float scale;
    int sh;
};
__device__ __forceinline__ Pow2 pow2_for(float amax)
{
    const int k = min(max((int)(__float_as_uint(amax) >> 23), 1), 253);
    return {__uint_as_float((uint32_t)(254 - k) << 23), 2 * (k - 127)};
}
__device__ __forceinline__ float absmax4(float m, const float4 &v)
{
    return fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
}
__device__ __forceinline__ float4 scale4(const float4 &v, float c)
{
    return make_float4(__fmul_rn(v.x, c), __fmul_rn(v.y, c), __fmul_rn(v.z, c), __fmul_rn(v.w, c));
}

// f * 2^sh as an FP64, exactly, by integer operations on the exponent field
// (|sh| <= 252 and f a partial sum of a rescaled chunk, so the FP64 exponent
// stays in range); zero and subnormal f give 0.
__device__ __forceinline__ double widen_pow2(float f, int sh)
{
    const uint32_t u = __float_as_uint(f);
    const uint32_t e = (u >> 23) & 0xFFu;
    const int ex = (int)e + 896 + sh;
    const uint64_t d = ((uint64_t)(u & 0x80000000u) << 32) | ((uint64_t)ex << 52) |
                       ((uint64_t)(u & 0x007FFFFFu) << 29);
    return e ? __longlong_as_double((long long)d) : 0.0;
}
__device__ __forceinline__ double widen_sum(const Sq32 &a, int sh)
{
    return widen_pow2(a.s, sh) + widen_pow2(a.e, sh);
}

// VEC amplitudes per 16-byte vector: 2 for complex64, 1 for complex128.
// raw() issues the load only; sq2() turns it into |a|^2 in FP64.  Callers
// issue a batch of raw loads before any arithmetic so that each thread keeps
// several 16-byte requests in flight.
template <typename R> struct AV;
template <> struct AV<float> {
    static constexpr int VEC = 2;
    using Raw = float4;
    __device__ __forceinline__ static Raw raw(const float *st, uint64_t v) { return reinterpret_cast<const float4 *>(st)[v]; }
    __device__ __forceinline__ static void sq2(const Raw &x, double p[2])
    {
        p[0] = sq<float>(x.x, x.y);
        p[1] = sq<float>(x.z, x.w);
    }
    __device__ __forceinline__ static void load(const float *st, uint64_t v, double p[2]) { sq2(raw(st, v), p); }
    __device__ __forceinline__ static void parts(const Raw &x, float re[2], float im[2])
    {
        re[0] = x.x; im[0] = x.y; re[1] = x.z; im[1] = x.w;
    }
};
template <> struct AV<double> {
    static constexpr int VEC = 1;
    using Raw = double2;
    __device__ __forceinline__ static Raw raw(const double *st, uint64_t v) { return reinterpret_cast<const double2 *>(st)[v]; }
    __device__ __forceinline__ static void sq2(const Raw &x, double p[2])
    {
        p[0] = sq<double>(x.x, x.y);
        p[1] = 0.0;
    }
    __device__ __forceinline__ static void load(const double *st, uint64_t v, double p[2]) { sq2(raw(st, v), p); }
    __device__ __forceinline__ static void parts(const Raw &x, double re[1], double im[1])
    {
        re[0] = x.x; im[0] = x.y;
    }
};

// one amplitude as a vector type
template <typename R> struct Amp;
template <> struct Amp<float> { using T = float2; };
template <> struct Amp<double> { using T = double2; };

constexpr int kBatch = 8;     // 16-byte loads in flight per thread

// Masked FP64 sums over a contiguous range per block.
//   RED_NORM: out0 = sum |a|^2                    (two FP64 FMAs per amplitude)
//   RED_BIT : out0 = sum over bit q = 0, out1 = sum over bit q = 1
//   RED_EXPZ: out0 = sum |a_x|^2 (n - 2 popcount x)  (weights from a table),
//             out1 = sum |a|^2 (the norm, from the same pass)
template <typename R, int MODE>
__global__ void __launch_bounds__(kRedThreads) k_masked_sum(const R *__restrict__ st, uint64_t nvec, uint64_t per,
                                                            int q, int n, double *__restrict__ partial)
{
    constexpr int VEC = AV<R>::VEC;
    __shared__ double sh[2 * kRedThreads / 32];
    __shared__ double wtab[64];                 // RED_EXPZ: wtab[k] = n - 2k
    if (MODE == RED_EXPZ) {
        for (int k = threadIdx.x; k <= n; k += kRedThreads) wtab[k] = (double)(n - 2 * k);
        __syncthreads();
    }
    const uint64_t lo = (uint64_t)blockIdx.x * per;
    const uint64_t hi = min(nvec, lo + per);
    double a = 0.0, b = 0.0;
    auto add = [&](uint64_t v, const typename AV<R>::Raw &x) {
        R re[VEC], im[VEC];
        AV<R>::parts(x, re, im);
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            const uint64_t i = v * VEC + e;
            if (MODE == RED_NORM) {
                acc_sq<R>(a, re[e], im[e]);
            } else if (MODE == RED_BIT) {
                if ((i >> q) & 1ull) acc_sq<R>(b, re[e], im[e]);
                else acc_sq<R>(a, re[e], im[e]);
            } else {
                const double p2 = sq<R>(re[e], im[e]);
                a = fma(p2, wtab[__popcll(i)], a);
                b += p2;
            }
        }
    };
    uint64_t v = lo + threadIdx.x;
    for (; v + (uint64_t)(kBatch - 1) * kRedThreads < hi; v += (uint64_t)kBatch * kRedThreads) {
        typename AV<R>::Raw x[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) x[u] = AV<R>::raw(st, v + (uint64_t)u * kRedThreads);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) add(v + (uint64_t)u * kRedThreads, x[u]);
    }
    for (; v < hi; v += kRedThreads) add(v, AV<R>::raw(st, v));
    block_sum2<kRedThreads>(a, b, sh);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = b;
    }
}

// complex64 norm (MODE RED_NORM) and the two halves of qubit q (RED_BIT) with
// the compensated FP32 sums above: per batch of 8 16-byte vectors (16
// amplitudes) one power-of-two scale, two carries into FP64 (8 amplitudes
// each).  The batches, the grid and the FP64 tree are those of k_masked_sum.
// RED_BIT: bit q is usually the same for all of a thread's batch, which then needs
// no choice of sum per amplitude (28 qubits: 0.43 -> 0.38 ms; the batch's two carries are added
// to each other first, so the last bit can differ from the path below).
template <int MODE>
__global__ void __launch_bounds__(kRedThreads) k_sum_sq32(const float *__restrict__ st, uint64_t nvec, uint64_t per,
                                                          int q, double *__restrict__ partial)
{
    static_assert(MODE == RED_NORM || MODE == RED_BIT, "norm or one qubit's halves");
    __shared__ double sh[2 * kRedThreads / 32];
    const uint64_t lo = (uint64_t)blockIdx.x * per;
    const uint64_t hi = min(nvec, lo + per);
    const float4 *st4 = reinterpret_cast<const float4 *>(st);
    double a = 0.0, b = 0.0;
    // the amplitudes of vector v (indices 2v, 2v + 1) go to A (bit q = 0) or B
    auto add_vec = [&](Sq32 &A, Sq32 &B, uint64_t v, const float4 &y) {
        if (MODE == RED_NORM) {
            A.add_sq(y.x); A.add_sq(y.y); A.add_sq(y.z); A.add_sq(y.w);
        } else {
            const bool b0 = ((2 * v) >> q) & 1ull, b1 = ((2 * v + 1) >> q) & 1ull;
            Sq32 c = b0 ? B : A;
            c.add_sq(y.x); c.add_sq(y.y);
            if (b0) B = c; else A = c;
            c = b1 ? B : A;
            c.add_sq(y.z); c.add_sq(y.w);
            if (b1) B = c; else A = c;
        }
    };
    uint64_t v = lo + threadIdx.x;
    for (; v + (uint64_t)(kBatch - 1) * kRedThreads < hi; v += (uint64_t)kBatch * kRedThreads) {
        float4 x[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) x[u] = st4[v + (uint64_t)u * kRedThreads];
        float m = 0.f;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) m = absmax4(m, x[u]);
        const Pow2 p = pow2_for(m);
        if (MODE == RED_BIT) {
            // bit q of all the batch's vectors: the strides of 2^8 vectors leave the bits below alone,
            // and a bit of 2^11 or more vectors changes at most once over them
            static_assert(kRedThreads == 256 && kBatch == 8, "strides of 2^8, a span below 2^11");
            const uint64_t first = 2 * v, end = 2 * (v + (uint64_t)(kBatch - 1) * kRedThreads);
            if (q >= 1 && (q <= 8 || (q >= 12 && !(((first ^ end) >> q) & 1ull)))) {
                double t = 0.0;
                const pack2 sc = dup(p.scale), nsc = dup(-p.scale);
#pragma unroll
                for (int h = 0; h < kBatch; h += 4) {
                    Sq32 A;
#pragma unroll
                    for (int u = h; u < h + 4; ++u) {
                        const Split2 q0 = square2(pk(x[u].x, x[u].y), sc, nsc);
                        const Split2 q1 = square2(pk(x[u].z, x[u].w), sc, nsc);
                        const float2 h0 = unpk(q0.nh), l0 = unpk(q0.l), h1 = unpk(q1.nh), l1 = unpk(q1.l);
                        A.add_split(h0.x, l0.x); A.add_split(h0.y, l0.y);
                        A.add_split(h1.x, l1.x); A.add_split(h1.y, l1.y);
                    }
                    t += widen_sum(A, p.sh);
                }
                if ((first >> q) & 1ull) b += t;
                else a += t;
                continue;
            }
        }
#pragma unroll
        for (int h = 0; h < kBatch; h += 4) {
            Sq32 A, B;
#pragma unroll
            for (int u = h; u < h + 4; ++u) add_vec(A, B, v + (uint64_t)u * kRedThreads, scale4(x[u], p.scale));
            a += widen_sum(A, p.sh);
            if (MODE == RED_BIT) b += widen_sum(B, p.sh);
        }
    }
    for (; v < hi; v += kRedThreads) {
        const float4 x = st4[v];
        const Pow2 p = pow2_for(absmax4(0.f, x));
        Sq32 A, B;
        add_vec(A, B, v, scale4(x, p.scale));
        a += widen_sum(A, p.sh);
        if (MODE == RED_BIT) b += widen_sum(B, p.sh);
    }
    block_sum2<kRedThreads>(a, b, sh);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = b;
    }
}

// <sum Z> over chunks of 16 consecutive amplitudes (n >= 4): for x = 16 ch +
// e, popcount(x) = popcount(ch) + popcount(e), so a thread sums the squares of
// a chunk into five bins by popcount(e) (two FP64 FMAs per amplitude, e known
// at compile time) and adds bin j with weight n - 2 (popcount(ch) + j): five
// FMAs per 16 amplitudes instead of one weighted FMA each.  The second
// partial is the norm (the bins' sum) from the same pass.
template <typename R>
__global__ void __launch_bounds__(kRedThreads) k_expz_chunks(const R *__restrict__ st, uint64_t nch, uint64_t per,
                                                             int n, double *__restrict__ partial)
{
    using T = typename Amp<R>::T;
    __shared__ double sh[2 * kRedThreads / 32];
    __shared__ double wtab[64];                  // wtab[k] = n - 2k
    for (int k = threadIdx.x; k <= n; k += kRedThreads) wtab[k] = (double)(n - 2 * k);
    __syncthreads();
    const uint64_t lo = (uint64_t)blockIdx.x * per;
    const uint64_t hi = min(nch, lo + per);
    double a = 0.0, b = 0.0;
    for (uint64_t ch = lo + threadIdx.x; ch < hi; ch += kRedThreads) {
        double bin[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        if (sizeof(R) == 4) {
            const float4 *q = reinterpret_cast<const float4 *>(st) + ch * 8;
            float4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = q[u];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                acc_sq<float>(bin[__builtin_popcount(2 * u)], x[u].x, x[u].y);
                acc_sq<float>(bin[__builtin_popcount(2 * u + 1)], x[u].z, x[u].w);
            }
        } else {
            const T *q = reinterpret_cast<const T *>(st) + ch * 16;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                T x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = q[8 * h + u];
#pragma unroll
                for (int u = 0; u < 8; ++u) acc_sq<R>(bin[__builtin_popcount(8 * h + u)], x[u].x, x[u].y);
            }
        }
        const int pc = __popcll(ch);
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            a = fma(wtab[pc + j], bin[j], a);
            b += bin[j];
        }
    }
    block_sum2<kRedThreads>(a, b, sh);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = b;
    }
}

// complex64 <sum Z> over chunks of 16 consecutive amplitudes (n >= 4): the
// same popcount bins as k_expz_chunks, each a compensated FP32 sum of squares
// of the chunk rescaled by one power of two; the bins are weighted by the
// integers n - 2 (popcount(ch) + j) with exact FP32 products into one
// compensated sum, carried into FP64 once per chunk.  Bins hold at most 12
// squares; the weighted sum cancels, so its error is relative to
// sum_j |w_j| bin_j <= n * (the chunk's sum of squares).  The second
// partial is the norm: the bins' compensated sum, carried into FP64 per chunk.
__global__ void __launch_bounds__(kRedThreads) k_expz32(const float *__restrict__ st, uint64_t nch, uint64_t per,
                                                        int n, double *__restrict__ partial)
{
    __shared__ double sh[2 * kRedThreads / 32];
    const uint64_t lo = (uint64_t)blockIdx.x * per;
    const uint64_t hi = min(nch, lo + per);
    const float4 *st4 = reinterpret_cast<const float4 *>(st);
    double a = 0.0, b = 0.0;
    for (uint64_t ch = lo + threadIdx.x; ch < hi; ch += kRedThreads) {
        float4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = st4[ch * 8 + u];
        float m = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) m = absmax4(m, x[u]);
        const Pow2 p = pow2_for(m);
        Sq32 bin[5];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float4 y = scale4(x[u], p.scale);
            bin[__builtin_popcount(2 * u)].add_sq(y.x);
            bin[__builtin_popcount(2 * u)].add_sq(y.y);
            bin[__builtin_popcount(2 * u + 1)].add_sq(y.z);
            bin[__builtin_popcount(2 * u + 1)].add_sq(y.w);
        }
        const int pc = __popcll(ch);
        Sq32 w, t;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const float wj = (float)(n - 2 * (pc + j));
            w.add_prod(bin[j].s, wj);
            w.e = __fmaf_rn(bin[j].e, wj, w.e);
            t.two_sum(bin[j].s);
            t.e = __fadd_rn(t.e, bin[j].e);
        }
        a += widen_sum(w, p.sh);
        b += widen_sum(t, p.sh);
    }
    block_sum2<kRedThreads>(a, b, sh);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = b;
    }
}

__global__ void __launch_bounds__(kRedThreads) k_final_sum(const double *__restrict__ partial, int nblk,
                                                           double *__restrict__ out)
{
    __shared__ double sh[2 * kRedThreads / 32];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nblk; i += kRedThreads) {
        a += partial[2 * i];
        b += partial[2 * i + 1];
    }
    block_sum2<kRedThreads>(a, b, sh);
    if (threadIdx.x == 0) { out[0] = a; out[1] = b; }
}

// ---------------------------------------------------------------- probabilities
// 16-byte vectors of the state (two complex64 amplitudes, one complex128), four
// in flight a thread; HBM-bound (28 qubits complex64: 3.2 GB).  aligned: the
// output takes whole-vector stores.
template <typename R, typename O>
__global__ void __launch_bounds__(256) k_probabilities(const R *__restrict__ st, uint64_t nvec, O *__restrict__ p,
                                                       bool aligned)
{
    constexpr int A = sizeof(R) == 4 ? 2 : 1;          // amplitudes per vector
    constexpr int U = 4;
    struct alignas(16) Vec { R x[2 * A]; };
    struct alignas(A * sizeof(O)) Out { O x[A]; };
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < nvec; i0 += U * step) {
        Vec v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * step < nvec) v[u] = reinterpret_cast<const Vec *>(st)[i0 + u * step];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t i = i0 + u * step;
            if (i >= nvec) break;
            Out o;
#pragma unroll
            for (int a = 0; a < A; ++a) {
                const R re = v[u].x[2 * a], im = v[u].x[2 * a + 1];
                if (sizeof(O) == sizeof(R)) o.x[a] = (O)(re * re + im * im);
                else o.x[a] = (O)sq<R>(re, im);
            }
            if (aligned) {
                reinterpret_cast<Out *>(p)[i] = o;
            } else {
#pragma unroll
                for (int a = 0; a < A; ++a) p[A * i + a] = o.x[a];
            }
        }
    }
}

// ---------------------------------------------------------------- collapse
// 16-byte vectors, four in flight a thread: the kept half is read, scaled and
// written, the other half only written (HBM-bound).
template <typename R>
__global__ void __launch_bounds__(256) k_collapse(R *__restrict__ st, uint64_t nvec, int q, int outcome, R scale)
{
    constexpr int A = sizeof(R) == 4 ? 2 : 1;
    constexpr int U = 4;
    struct alignas(16) Vec { R x[2 * A]; };
    Vec *s = reinterpret_cast<Vec *>(st);
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    const int qv = q - (A - 1);                        // the qubit's bit of a vector index, -1: inside the vector
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < nvec; i0 += U * step) {
        Vec v[U];
        bool keep[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t i = i0 + u * step;
            keep[u] = qv < 0 || (int)((i >> qv) & 1ull) == outcome;
            if (keep[u] && i < nvec) v[u] = s[i];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t i = i0 + u * step;
            if (i >= nvec) break;
            Vec o;
#pragma unroll
            for (int e = 0; e < 2 * A; ++e)
                o.x[e] = (keep[u] && (qv >= 0 || (e >> 1) == outcome)) ? v[u].x[e] * scale : (R)0;
            s[i] = o;
        }
    }
}

// ---------------------------------------------------------------- sampling
constexpr int kSampleLog = 13;             // 8192 amplitudes per sampling block
constexpr int kScanThreads = 1024;

// Sub-blocks: min(256, bs) amplitudes, nsub = bs / sub <= 32 per block; lane
// l of a warp takes amplitudes l*apl .. l*apl + apl - 1 of a sub-block
// (apl = max(1, sub / 32)), so a lane-serial prefix followed by a warp scan
// is the sub-block's prefix in index order.
constexpr int kSubLog = 8;

struct SubGeo {
    uint32_t sub, nsub, apl, lanes;
    __host__ __device__ explicit SubGeo(uint64_t bs)
    {
        sub = (uint32_t)(bs < (1ull << kSubLog) ? bs : (1ull << kSubLog));
        nsub = (uint32_t)(bs / sub);
        apl = sub >= 32 ? sub / 32 : 1;
        lanes = sub / apl;
    }
};


// warp inclusive scan of lanes 0..31, fixed order (shfl_up doubling)
__device__ __forceinline__ double warp_incl_scan(double x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// One CTA (8 warps) per block of bs amplitudes.  Groups of 8 lanes own one
// sub-block each (4 per warp, 32 per CTA): lane g of a group accumulates a
// contiguous eighth of the sub-block (complex64 full sub-blocks: compensated
// FP32 squares carried into FP64 every 8 amplitudes; otherwise two FP64 FMAs
// per amplitude), written to eighth[] where that is not null, and a 3-step xor
// tree inside the group gives the sub-sum.  Warp 0 then scans the block's
// sub-sums (warp_incl_scan); the inclusive scan goes to cum[], its last element
// is the block sum.
// kZ (complex64 full sub-blocks only): the same pass also forms the block's
// <sum Z> partial as k_expz32 does (each 16-amplitude chunk's squares binned
// by the popcount of the local index, weighted by n - 2 popcount, one
// compensated sum carried into FP64), written to zpart[2 b] (zpart[2 b + 1] =
// 0, the pair layout k_final_sum reads).  The sub-sums are computed exactly as
// without it.  The squares are split once for both, in packs; packs take the FP32
// lanes as long as two scalars, so the gain is what is shared (28 qubits, sampling kernels:
// 0.680 -> 0.659 ms).  Four CTAs an SM: 66 registers, three CTAs, take 0.786 ms.
template <typename R, bool kZ = false>
__global__ void __launch_bounds__(256, 4) k_sub_sums(const R *__restrict__ st, uint64_t bs, double *__restrict__ cum,
                                                  double *__restrict__ bsum, double *__restrict__ eighth, int n = 0,
                                                  double *__restrict__ zpart = nullptr)
{
    using T = typename Amp<R>::T;
    const SubGeo g(bs);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t j = (uint32_t)(warp * 4 + (lane >> 3));       // this group's sub-block
    const uint32_t gl = (uint32_t)(lane & 7);                    // lane within the group
    const uint64_t base = (uint64_t)blockIdx.x * bs;
    __shared__ double ss[32];
    __shared__ double zs[8];
    double t = 0.0, z = 0.0;
    if (j < g.nsub) {
        const uint32_t per = g.sub >= 8 ? g.sub / 8 : 1;         // amplitudes per lane
        if (gl * per < g.sub) {
            const T *a = reinterpret_cast<const T *>(st) + base + (uint64_t)j * g.sub + (uint64_t)gl * per;
            if (sizeof(R) == 4 && per == 32) {
                // complex64, full sub-block: 16 aligned 16-byte loads per lane,
                // 8 in flight; compensated FP32 squares, one scale per 16
                // amplitudes, carried into FP64 every 8
                const float4 *a4 = reinterpret_cast<const float4 *>(a);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float4 x[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) x[u] = a4[h * 8 + u];
                    float m = 0.f;
#pragma unroll
                    for (int u = 0; u < 8; ++u) m = absmax4(m, x[u]);
                    const Pow2 pw = pow2_for(m);
                    const pack2 sc = dup(pw.scale), nsc = dup(-pw.scale);
                    Sum2 bin[5];
#pragma unroll
                    for (int c = 0; c < 8; c += 4) {
                        Sq32 A;
#pragma unroll
                        for (int u = c; u < c + 4; ++u) {
                            const Split2 q0 = square2(pk(x[u].x, x[u].y), sc, nsc);
                            const Split2 q1 = square2(pk(x[u].z, x[u].w), sc, nsc);
                            const float2 h0 = unpk(q0.nh), l0 = unpk(q0.l), h1 = unpk(q1.nh), l1 = unpk(q1.l);
                            A.add_split(h0.x, l0.x); A.add_split(h0.y, l0.y);
                            A.add_split(h1.x, l1.x); A.add_split(h1.y, l1.y);
                            if constexpr (kZ) {
                                // x[u] holds local indices 2u, 2u + 1 of 16
                                bin[__builtin_popcount(2 * u)].add_split(q0.nh, q0.l);
                                bin[__builtin_popcount(2 * u + 1)].add_split(q1.nh, q1.l);
                            }
                        }
                        t += widen_sum(A, pw.sh);
                    }
                    if constexpr (kZ) {
                        // amplitudes 16 ch .. 16 ch + 15
                        const uint64_t ch = ((base + (uint64_t)j * g.sub + (uint64_t)gl * per) >> 4) + (uint64_t)h;
                        const int pc = __popcll(ch);
                        Sum2 w;
#pragma unroll
                        for (int b = 0; b < 5; ++b) w.add_weighted(bin[b], (float)(n - 2 * (pc + b)));
                        z += widen_sum(w.total(), pw.sh);
                    }
                }
            } else {
                for (uint32_t e0 = 0; e0 < per; e0 += 8) {
                    T x[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (e0 + u < per) x[u] = a[e0 + u];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (e0 + u < per) acc_sq<R>(t, x[u].x, x[u].y);
                }
            }
        }
    }
    if (eighth && j < g.nsub) eighth[((uint64_t)blockIdx.x * g.nsub + j) * 8 + gl] = t;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (gl == 0 && j < g.nsub) ss[j] = t;
    if constexpr (kZ) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        if (lane == 0) zs[warp] = z;
    }
    __syncthreads();
    if (warp == 0) {
        const double c = warp_incl_scan(((uint32_t)lane < g.nsub) ? ss[lane] : 0.0, lane);
        if ((uint32_t)lane < g.nsub) cum[(uint64_t)blockIdx.x * g.nsub + lane] = c;
        if ((uint32_t)lane == g.nsub - 1) bsum[blockIdx.x] = c;
    }
    if constexpr (kZ) {
        if (threadIdx.x == 0) {
            double zz = 0.0;
#pragma unroll
            for (int w = 0; w < 8; ++w) zz += zs[w];
            zpart[2 * blockIdx.x] = zz;
            zpart[2 * blockIdx.x + 1] = 0.0;
        }
    }
}

// Exclusive scan of nb values in one CTA: contiguous segments per thread,
// serial inside a segment, a fixed Hillis-Steele scan over segment totals.
template <typename T>
__global__ void __launch_bounds__(kScanThreads) k_scan_exclusive(const T *__restrict__ in, T *__restrict__ out,
                                                                 uint64_t nb, T *__restrict__ total)
{
    __shared__ T seg[kScanThreads];
    const uint64_t per = (nb + kScanThreads - 1) / kScanThreads;
    const uint64_t lo = (uint64_t)threadIdx.x * per;
    const uint64_t hi = min(nb, lo + per);
    T loc = 0;
    for (uint64_t i = lo; i < hi; ++i) loc += in[i];
    seg[threadIdx.x] = loc;
    __syncthreads();
    for (int off = 1; off < kScanThreads; off <<= 1) {
        T v = (threadIdx.x >= (unsigned)off) ? seg[threadIdx.x - off] : (T)0;
        __syncthreads();
        seg[threadIdx.x] += v;
        __syncthreads();
    }
    T run = (threadIdx.x > 0) ? seg[threadIdx.x - 1] : (T)0;
    if (threadIdx.x == kScanThreads - 1) *total = seg[kScanThreads - 1];
    T acc = 0;
    for (uint64_t i = lo; i < hi; ++i) {
        out[i] = run + acc;
        acc += in[i];
    }
}

// Exclusive scan over many CTAs (the sampler's block sums are FP64, and one
// CTA adding 2^17 of them ran into the narrow FP64 pipe of a single SM):
// chunks of kScanChunk values, four contiguous values per thread.  Pass 1
// writes each chunk's total, the one-CTA scan above turns the totals into
// chunk offsets (and the grand total), pass 2 repeats the chunk's local scan
// (the same operations, so the same bits) and adds the chunk's offset, writing
// each value's exclusive and inclusive sum.
constexpr int kScanChunk = 1024;

template <typename T>
__device__ __forceinline__ T chunk_local_scan(const T *__restrict__ in, uint64_t nb, T *sh, T &total, T v[4],
                                              uint64_t &lo)
{
    lo = (uint64_t)blockIdx.x * kScanChunk + 4u * threadIdx.x;
    T loc = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        v[e] = (lo + e < nb) ? in[lo + e] : (T)0;
        loc += v[e];
    }
    sh[threadIdx.x] = loc;
    __syncthreads();
    for (int off = 1; off < 256; off <<= 1) {
        const T y = (threadIdx.x >= (unsigned)off) ? sh[threadIdx.x - off] : (T)0;
        __syncthreads();
        sh[threadIdx.x] += y;
        __syncthreads();
    }
    total = sh[255];
    return (threadIdx.x > 0) ? sh[threadIdx.x - 1] : (T)0;
}

template <typename T>
__global__ void __launch_bounds__(256) k_scan_chunk_sums(const T *__restrict__ in, uint64_t nb, T *__restrict__ csum)
{
    __shared__ T sh[256];
    T v[4], total;
    uint64_t lo;
    chunk_local_scan<T>(in, nb, sh, total, v, lo);
    if (threadIdx.x == 0) csum[blockIdx.x] = total;
}

template <typename T>
__global__ void __launch_bounds__(256) k_scan_chunk_out(const T *__restrict__ in, uint64_t nb,
                                                        const T *__restrict__ cexcl, T *__restrict__ out,
                                                        T *__restrict__ incl)
{
    __shared__ T sh[256];
    T v[4], total;
    uint64_t lo;
    T run = chunk_local_scan<T>(in, nb, sh, total, v, lo) + cexcl[blockIdx.x];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (lo + e < nb) out[lo + e] = run;
        run += v[e];
        if (lo + e < nb) incl[lo + e] = run;
    }
}

// last block with a non-zero sum (0: none), 1024 at a time from the end
__global__ void __launch_bounds__(1024) k_last_nonzero(const double *__restrict__ bsum, uint64_t nb,
                                                       uint64_t *__restrict__ out)
{
    for (uint64_t end = nb;; end -= 1024) {
        const uint64_t i = end - 1 - threadIdx.x;
        const bool nz = threadIdx.x < end && bsum[i] > 0.0;
        if (__syncthreads_or(nz) || end <= 1024) {
            if (threadIdx.x == 0) *out = 0;
            __syncthreads();
            if (nz) atomicMax((unsigned long long *)out, (unsigned long long)i);
            return;
        }
    }
}

// a power of two 2^d as a float for d <= 127; 0 below -126 (a lane that
// small against the largest one contributes nothing measurable)
__device__ __forceinline__ float pow2f(int d)
{
    return d < -126 ? 0.f : __uint_as_float((uint32_t)(127 + min(d, 127)) << 23);
}

// s + t as an unevaluated pair (hi, lo) (Knuth's TwoSum) added to (hi, lo)
__device__ __forceinline__ void df_add(float &hi, float &lo, float th, float tl)
{
    const float u = __fadd_rn(hi, th);
    const float z = __fsub_rn(u, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(u, z)), __fsub_rn(th, z));
    hi = u;
    lo = __fadd_rn(__fadd_rn(lo, tl), err);
}

// A non-negative finite double orders like its bits as a signed integer; a
// negative one has negative bits, below all of them.  So a > b for a >= 0
// takes two integer instructions instead of one on the FP64 pipe, which
// issues one warp instruction every 16 cycles per SM.
__device__ __forceinline__ bool above(double a, double b)
{
    return __double_as_longlong(a) > __double_as_longlong(b);
}

// a shot's target relative to its sub-block: (hi + lo) 2^e, |hi| in [1, 2]
struct Target {
    float hi, lo;
    int e;
};

__device__ __forceinline__ Target split_target(double d)
{
    const uint64_t b = (uint64_t)__double_as_longlong(d);
    const int f = (int)((b >> 52) & 0x7ffu);
    if (f == 0) return {0.f, 0.f, 0};
    const double m = __longlong_as_double((long long)((b & 0x800fffffffffffffull) | (1023ull << 52)));
    const float hi = __double2float_rn(m);
    return {hi, __double2float_rn(m - (double)hi), f - 1023};
}

// complex64: the first of the 32 amplitudes of an eighth (four in each of
// eight lanes, gl = lane within the group) whose prefix exceeds the target.
// The lane's prefix is kept as compensated FP32 partial sums of its squares rescaled
// by a power of two (2^-sh, from the lane's largest component).  The lanes' totals are
// brought to one scale (the group's largest sh) by exact powers of two and
// scanned across the group as FP32 pairs (TwoSum).  The target, brought to
// that scale, relative to the lane's start and rescaled back to the lane's
// units, is compared with each partial sum as a float pair.  An amplitude that
// is exactly zero leaves the prefix unchanged and is never the first
// crossing.  Returns the first crossing in the lane (-1: none).
__device__ __forceinline__ int lane_locate(const float4 x[2], int gl, const Target &tg)
{
    const Pow2 pw = pow2_for(absmax4(absmax4(0.f, x[0]), x[1]));
    float cs[4], ce[4];
    Sq32 A;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float4 y = scale4(x[u], pw.scale);
        A.add_sq(y.x); A.add_sq(y.y);
        cs[2 * u] = A.s; ce[2 * u] = A.e;
        A.add_sq(y.z); A.add_sq(y.w);
        cs[2 * u + 1] = A.s; ce[2 * u + 1] = A.e;
    }
    // the lane's total in the group's common units 2^shm (shm >= pw.sh)
    int shm = pw.sh;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) shm = max(shm, __shfl_xor_sync(0xffffffffu, shm, o));
    const float down = pow2f(pw.sh - shm);
    float ih = __fmul_rn(A.s, down), il = __fmul_rn(A.e, down);
    // inclusive scan of the pairs over the group, then each lane's start = the
    // previous lane's inclusive sum
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const float yh = __shfl_up_sync(0xffffffffu, ih, o, 8);
        const float yl = __shfl_up_sync(0xffffffffu, il, o, 8);
        if (gl >= o) df_add(ih, il, yh, yl);
    }
    float sh0 = __shfl_up_sync(0xffffffffu, ih, 1, 8), sl0 = __shfl_up_sync(0xffffffffu, il, 1, 8);
    if (gl == 0) { sh0 = 0.f; sl0 = 0.f; }
    // the target in common units (beyond 2^100: past every sum), minus the
    // lane's start, back in the lane's units
    const float unit = pow2f(min(tg.e - shm, 100));
    float rh = __fmul_rn(tg.hi, unit), rl = __fmul_rn(tg.lo, unit);
    df_add(rh, rl, -sh0, -sl0);
    const float up = pow2f(shm - pw.sh);
    const bool far = shm - pw.sh > 127;            // the lane is negligible next to the largest
    rh = far ? (rh > 0.f ? INFINITY : -INFINITY) : __fmul_rn(rh, up);
    rl = far ? 0.f : __fmul_rn(rl, up);
    int first = -1;
#pragma unroll
    for (int e = 3; e >= 0; --e) {
        const float4 &v = x[e >> 1];
        const bool nz = (e & 1) ? (v.z != 0.f || v.w != 0.f) : (v.x != 0.f || v.y != 0.f);
        if (nz && __fadd_rn(__fsub_rn(cs[e], rh), __fsub_rn(ce[e], rl)) > 0.f) first = e;
    }
    return first;
}

// complex128: the same in FP64
__device__ __forceinline__ int lane_locate(const double2 x[4], int gl, double target)
{
    double c[4], run = 0.0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        acc_sq<double>(run, x[e].x, x[e].y);
        c[e] = run;
    }
    double incl = run;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, incl, o, 8);
        if (gl >= o) incl += y;
    }
    const double r = target - (incl - run);
    int first = -1;
#pragma unroll
    for (int e = 3; e >= 0; --e)
        if (above(c[e], r) && above(c[e], e ? c[e - 1] : 0.0)) first = e;
    return first;
}

// Shots of a register of at least 2^8 amplitudes.  Shot s takes t = u_s total
// and the first index whose prefix sum of |a|^2 exceeds t, found level by level:
// the block (bexcl, bincl), the sub-block (cum, inclusive within the block), the
// eighth of it, the amplitude.  Where rounding leaves no crossing (t within an ulp of a
// boundary), the last one with non-zero probability is taken.

// the tables of the first two levels
struct ShotTables {
    uint32_t nsub;
    uint64_t nb;
    const double *bexcl, *bincl, *cum;
    const uint64_t *last;
};

// the sub-block (counted over the register) that holds t; d = t relative to its start
__device__ __forceinline__ uint64_t find_sub(const ShotTables &T, double t, double &d)
{
    uint64_t lo = 0, hi = T.nb;
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (above(T.bincl[mid], t)) hi = mid; else lo = mid + 1;
    }
    const uint64_t b = lo < T.nb ? lo : *T.last;
    const double be = T.bexcl[b];
    const double *P = T.cum + b * T.nsub;
    uint32_t j = 0, je = T.nsub;
    while (j < je) {
        const uint32_t mid = (j + je) >> 1;
        if (above(be + P[mid], t)) je = mid; else j = mid + 1;
    }
    if (j == T.nsub)
        for (--j; j > 0 && !(P[j] > P[j - 1]);) --j;
    d = t - (be + (j > 0 ? P[j - 1] : 0.0));
    return b * T.nsub + j;
}

// the last eighth that is not empty and starts at or before the target; d becomes relative to it
__device__ __forceinline__ uint32_t find_eighth(const double ev[8], double &d)
{
    double acc = 0.0, gp = 0.0;
    int g = -1;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (above(ev[k], 0.0) && (g < 0 || !above(acc, d))) {
            g = k;
            gp = acc;
        }
        if (k < 7) acc += ev[k];
    }
    d -= gp;
    return (uint32_t)max(g, 0);
}

// the amplitude within the eighth, from the crossing in each of its eight lanes (-1: none)
template <typename V, int NV>
__device__ __forceinline__ uint32_t find_amplitude(const V (&x)[NV], int hit, int gr)
{
    uint32_t fl = (__ballot_sync(0xffffffffu, hit >= 0) >> (8 * gr)) & 0xffu;
    if (__any_sync(0xffffffffu, fl == 0)) {        // no crossing: the last one that is not zero
        int nz = -1;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if constexpr (NV == 2) {
                const float4 &v = x[e >> 1];
                if ((e & 1) ? (v.z != 0.f || v.w != 0.f) : (v.x != 0.f || v.y != 0.f)) nz = e;
            } else {
                double p2 = 0.0;
                acc_sq<double>(p2, x[e].x, x[e].y);
                if (p2 > 0.0) nz = e;
            }
        }
        const uint32_t nl = (__ballot_sync(0xffffffffu, nz >= 0) >> (8 * gr)) & 0xffu;
        if (fl == 0) {
            hit = max(nz, 0);
            fl = nl ? 1u << (31 - __clz(nl)) : 1u;
        }
    }
    const int L = __ffs(fl) - 1;
    return (uint32_t)(4 * L + __shfl_sync(0xffffffffu, hit, 8 * gr + L));
}

// Many shots: the pass over the state has left the sums of the eighths.
// A lane looks up the first three levels of its own shot; then eight
// lanes read the 32 amplitudes of a shot's eighth, four shots of the warp at a time.
// The FP64 pipe (one warp instruction every 16 cycles per SM) is kept to what a lane
// needs for its shot.  When shots were sorted by block and a warp searched the
// 256 amplitudes of one sub-block per shot (14 FP64 instructions a shot, 480 in all),
// the sampling kernels took for a million shots 1.28 ms at 20 qubits (0.35 of it
// sorting) and 1.61 at 28, complex64, and 4.2 ms at 27, complex128; now 0.14, 0.68
// (0.55 the pass over the state) and 0.74.  The reads are as random as the shots
// either way, 256 bytes (512) per shot.
template <typename R>
__global__ void __launch_bounds__(256) k_shots(const R *__restrict__ st, ShotTables T, uint64_t seed,
                                               const double *__restrict__ total, const double *__restrict__ eighth,
                                               uint64_t shots, uint64_t *__restrict__ out)
{
    using V = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
    constexpr int NV = sizeof(R) == 4 ? 2 : 4;         // 16-byte vectors of a lane's four amplitudes
    const double tot = *total;
    if (!(tot > 0.0)) return;
    const int lane = threadIdx.x & 31, gr = lane >> 3, gl = lane & 7;
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t c0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); c0 < shots; c0 += step) {
        const uint64_t s = min(c0 + (uint64_t)lane, shots - 1);
        double rel;
        const uint64_t q = find_sub(T, unif(seed, s) * tot, rel);
        const double2 *e2 = reinterpret_cast<const double2 *>(eighth + 8 * q);
        double ev[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double2 y = e2[k];
            ev[2 * k] = y.x;
            ev[2 * k + 1] = y.y;
        }
        const uint32_t part = (uint32_t)(q * 8) + find_eighth(ev, rel);   // 32 amplitudes each
        Target tl = {0.f, 0.f, 0};
        if constexpr (sizeof(R) == 4) tl = split_target(rel);
        const V *av = reinterpret_cast<const V *>(st) + gl * NV;
        V nx[NV];
        {
            const uint64_t p = __shfl_sync(0xffffffffu, part, gr);
#pragma unroll
            for (int u = 0; u < NV; ++u) nx[u] = av[p * (8 * NV) + u];
        }
        uint32_t idx = 0;
#pragma unroll 1
        for (int it = 0; it < 8; ++it) {
            const int i = it * 4 + gr;
            V x[NV];
#pragma unroll
            for (int u = 0; u < NV; ++u) x[u] = nx[u];
            const uint64_t p = __shfl_sync(0xffffffffu, part, min(i + 4, 28 + gr));
#pragma unroll
            for (int u = 0; u < NV; ++u) nx[u] = av[p * (8 * NV) + u];
            int hit;
            if constexpr (sizeof(R) == 4)
                hit = lane_locate(x, gl, Target{__shfl_sync(0xffffffffu, tl.hi, i), __shfl_sync(0xffffffffu, tl.lo, i),
                                                __shfl_sync(0xffffffffu, tl.e, i)});
            else
                hit = lane_locate(x, gl, __shfl_sync(0xffffffffu, rel, i));
            const uint32_t found = find_amplitude(x, hit, gr);
            const uint32_t mine = __shfl_sync(0xffffffffu, found, 8 * (lane & 3));
            if ((lane >> 2) == it) idx = mine;
        }
        if (c0 + (uint64_t)lane < shots) out[s] = (uint64_t)part * 32 + idx;
    }
}

// sum of |a|^2 over the 32 amplitudes at p, by the operations of k_sub_sums
__device__ __forceinline__ double eighth_sum(const float *p)
{
    const float4 *a4 = reinterpret_cast<const float4 *>(p);
    double t = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = a4[h * 8 + u];
        float m = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) m = absmax4(m, x[u]);
        const Pow2 pw = pow2_for(m);
        const pack2 sc = dup(pw.scale), nsc = dup(-pw.scale);
#pragma unroll
        for (int c = 0; c < 8; c += 4) {
            Sq32 A;
#pragma unroll
            for (int u = c; u < c + 4; ++u) {
                const Split2 q0 = square2(pk(x[u].x, x[u].y), sc, nsc);
                const Split2 q1 = square2(pk(x[u].z, x[u].w), sc, nsc);
                const float2 h0 = unpk(q0.nh), l0 = unpk(q0.l), h1 = unpk(q1.nh), l1 = unpk(q1.l);
                A.add_split(h0.x, l0.x); A.add_split(h0.y, l0.y);
                A.add_split(h1.x, l1.x); A.add_split(h1.y, l1.y);
            }
            t += widen_sum(A, pw.sh);
        }
    }
    return t;
}
__device__ __forceinline__ double eighth_sum(const double *p)
{
    const double2 *a = reinterpret_cast<const double2 *>(p);
    double t = 0.0;
#pragma unroll
    for (int e0 = 0; e0 < 32; e0 += 8) {
        double2 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = a[e0 + u];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc_sq<double>(t, x[u].x, x[u].y);
    }
    return t;
}

// Few shots for the register's size: the pass over the state has not written the eighths
// (see kEighthsPer64), so eight lanes take one shot and form those of its sub-block
// from all 256 amplitudes.
template <typename R>
__global__ void __launch_bounds__(256) k_shots_read(const R *__restrict__ st, ShotTables T, uint64_t seed,
                                                    const double *__restrict__ total, uint64_t shots,
                                                    uint64_t *__restrict__ out)
{
    using V = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
    constexpr int NV = sizeof(R) == 4 ? 2 : 4;
    const double tot = *total;
    if (!(tot > 0.0)) return;
    const int lane = threadIdx.x & 31, gr = lane >> 3, gl = lane & 7;
    const uint64_t step = (uint64_t)gridDim.x * (blockDim.x >> 3);
    for (uint64_t c0 = ((uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) >> 3; c0 < shots; c0 += step) {
        const uint64_t s = min(c0 + (uint64_t)gr, shots - 1);
        double rel, ev[8];
        const uint64_t q = find_sub(T, unif(seed, s) * tot, rel);
        __syncwarp();
        const double e = eighth_sum(st + 2 * ((q << kSubLog) + 32 * (uint64_t)gl));
#pragma unroll
        for (int k = 0; k < 8; ++k) ev[k] = __shfl_sync(0xffffffffu, e, 8 * gr + k);
        const uint64_t part = q * 8 + find_eighth(ev, rel);
        const V *av = reinterpret_cast<const V *>(st) + part * (8 * NV) + gl * NV;
        V x[NV];
#pragma unroll
        for (int u = 0; u < NV; ++u) x[u] = av[u];
        int hit;
        if constexpr (sizeof(R) == 4) hit = lane_locate(x, gl, split_target(rel));
        else hit = lane_locate(x, gl, rel);
        const uint32_t found = find_amplitude(x, hit, gr);
        if (gl == 0 && c0 + (uint64_t)gr < shots) out[s] = part * 32 + found;
    }
}

// the same for a register of fewer than 2^8 amplitudes: their prefix in shared
// memory, a thread per shot
template <typename R>
__global__ void __launch_bounds__(256) k_shots_small(const R *__restrict__ st, uint32_t N, uint64_t seed,
                                                     const double *__restrict__ total, uint64_t shots,
                                                     uint64_t *__restrict__ out)
{
    __shared__ double pre[128];
    __shared__ uint32_t last;
    const double tot = *total;
    if (!(tot > 0.0)) return;
    if (threadIdx.x == 0) {
        double run = 0.0;
        last = 0;
        for (uint32_t i = 0; i < N; ++i) {
            double p = 0.0;
            acc_sq<R>(p, st[2 * i], st[2 * i + 1]);
            run += p;
            pre[i] = run;
            if (p > 0.0) last = i;
        }
    }
    __syncthreads();
    for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < shots;
         s += (uint64_t)gridDim.x * blockDim.x) {
        const double t = unif(seed, s) * tot;
        uint32_t lo = 0, hi = N;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (above(pre[mid], t)) hi = mid; else lo = mid + 1;
        }
        out[s] = lo < N ? lo : last;
    }
}

unsigned grid_for(uint64_t work, int threads, int num_sms)
{
    uint64_t g = (work + threads - 1) / threads;
    const uint64_t cap = (uint64_t)num_sms * 32;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

// exclusive scan of nb values into out, inclusive into incl and their total
// into *total, on the handle's stream; cs holds 2 * ceil(nb / kScanChunk) values of scratch
template <typename T>
int scan_sums(qsim_state *s, const T *in, T *out, T *incl, uint64_t nb, T *total, T *cs, const char *what)
{
    const uint64_t nc = (nb + kScanChunk - 1) / kScanChunk;
    launch_begin(s, KC_SAMPLE);
    k_scan_chunk_sums<T><<<(unsigned)nc, 256, 0, s->stream>>>(in, nb, cs);
    if (int rc = launch_end(s, what)) return rc;
    launch_begin(s, KC_SAMPLE);
    k_scan_exclusive<T><<<1, kScanThreads, 0, s->stream>>>(cs, cs + nc, nc, total);
    if (int rc = launch_end(s, what)) return rc;
    launch_begin(s, KC_SAMPLE);
    k_scan_chunk_out<T><<<(unsigned)nc, 256, 0, s->stream>>>(in, nb, cs + nc, out, incl);
    return launch_end(s, what);
}

}  // namespace

uint64_t splitmix64_host(uint64_t x) { return smix(x); }
double uniform_host(uint64_t seed, uint64_t s) { return unif(seed, s); }

int launch_init_basis(qsim_state *s, uint64_t j)
{
    const size_t amp = (s->dtype == SIM_C128) ? 16 : 8;
    const uint64_t nvec = (uint64_t)(s->bytes / 16);
    uint64_t jvec;
    uint4 jval = make_uint4(0, 0, 0, 0);
    if (amp == 16) {
        jvec = j;
        const double one = 1.0;
        uint64_t bits;
        memcpy(&bits, &one, 8);
        jval.x = (uint32_t)bits; jval.y = (uint32_t)(bits >> 32);
    } else {
        jvec = j / 2;
        const float one = 1.0f;
        uint32_t bits;
        memcpy(&bits, &one, 4);
        if (j & 1) jval.z = bits; else jval.x = bits;
    }
    launch_begin(s, KC_INIT, (double)s->bytes);
    k_init_basis<<<grid_for(nvec, 256, s->num_sms), 256, 0, s->stream>>>((uint4 *)s->amps, nvec, jvec, jval);
    return launch_end(s, "init basis");
}

int reduce_sums(qsim_state *s, int mode, int qubit, double out[2])
{
    const uint64_t N = 1ull << s->n;
    const uint64_t nvec = (s->dtype == SIM_C128) ? N : N / 2;
    const uint64_t per = (nvec + kRedBlocks - 1) / kRedBlocks;
    launch_begin(s, KC_REDUCE, (double)s->bytes);
    if (s->dtype == SIM_C128) {
        const double *st = (const double *)s->amps;
        if (mode == RED_NORM) k_masked_sum<double, RED_NORM><<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, nvec, per, qubit, s->n, s->red_partial);
        else if (mode == RED_BIT) k_masked_sum<double, RED_BIT><<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, nvec, per, qubit, s->n, s->red_partial);
        else if (s->n >= 4) k_expz_chunks<double><<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, N / 16, (N / 16 + kRedBlocks - 1) / kRedBlocks, s->n, s->red_partial);
        else k_masked_sum<double, RED_EXPZ><<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, nvec, per, qubit, s->n, s->red_partial);
    } else {
        const float *st = (const float *)s->amps;
        if (mode == RED_NORM) k_sum_sq32<RED_NORM><<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, nvec, per, qubit, s->red_partial);
        else if (mode == RED_BIT) k_sum_sq32<RED_BIT><<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, nvec, per, qubit, s->red_partial);
        else if (s->n >= 4) k_expz32<<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, N / 16, (N / 16 + kRedBlocks - 1) / kRedBlocks, s->n, s->red_partial);
        else k_masked_sum<float, RED_EXPZ><<<kRedBlocks, kRedThreads, 0, s->stream>>>(st, nvec, per, qubit, s->n, s->red_partial);
    }
    int rc = launch_end(s, "masked sum");
    if (rc) return rc;
    launch_begin(s, KC_REDUCE);
    k_final_sum<<<1, kRedThreads, 0, s->stream>>>(s->red_partial, kRedBlocks, s->red_out);
    rc = launch_end(s, "final sum");
    if (rc) return rc;
    QSIM_CUDA(cudaMemcpyAsync(s->host_red, s->red_out, 2 * sizeof(double), cudaMemcpyDeviceToHost, s->stream));
    QSIM_CUDA(cudaStreamSynchronize(s->stream));
    out[0] = s->host_red[0];
    out[1] = s->host_red[1];
    return SIM_OK;
}

// sum_j |a_j|^2 into s->red_out[0] on the device (accumulated as for
// sim_norm), for kernels that read it later in stream order; no host sync
int reduce_norm_device(qsim_state *s)
{
    const uint64_t N = 1ull << s->n;
    const uint64_t nvec = (s->dtype == SIM_C128) ? N : N / 2;
    const uint64_t per = (nvec + kRedBlocks - 1) / kRedBlocks;
    launch_begin(s, KC_REDUCE, (double)s->bytes);
    if (s->dtype == SIM_C128)
        k_masked_sum<double, RED_NORM><<<kRedBlocks, kRedThreads, 0, s->stream>>>((const double *)s->amps, nvec, per, 0,
                                                                                  s->n, s->red_partial);
    else
        k_sum_sq32<RED_NORM><<<kRedBlocks, kRedThreads, 0, s->stream>>>((const float *)s->amps, nvec, per, 0,
                                                                       s->red_partial);
    if (int rc = launch_end(s, "norm pass")) return rc;
    launch_begin(s, KC_REDUCE);
    k_final_sum<<<1, kRedThreads, 0, s->stream>>>(s->red_partial, kRedBlocks, s->red_out);
    return launch_end(s, "norm final sum");
}

int launch_probabilities(qsim_state *s, void *dev_out, int out_real)
{
    const uint64_t N = 1ull << s->n;
    const uint64_t nvec = (s->dtype == SIM_C128) ? N : N / 2;
    const unsigned g = grid_for(nvec, 256, s->num_sms);
    const bool aligned = ((uintptr_t)dev_out & 15u) == 0;
    launch_begin(s, KC_PROB, (double)s->bytes + (double)N * (out_real == SIM_F64 ? 8.0 : 4.0));
    if (s->dtype == SIM_C128) {
        if (out_real == SIM_F64) k_probabilities<double, double><<<g, 256, 0, s->stream>>>((const double *)s->amps, nvec, (double *)dev_out, aligned);
        else k_probabilities<double, float><<<g, 256, 0, s->stream>>>((const double *)s->amps, nvec, (float *)dev_out, aligned);
    } else {
        if (out_real == SIM_F64) k_probabilities<float, double><<<g, 256, 0, s->stream>>>((const float *)s->amps, nvec, (double *)dev_out, aligned);
        else k_probabilities<float, float><<<g, 256, 0, s->stream>>>((const float *)s->amps, nvec, (float *)dev_out, aligned);
    }
    return launch_end(s, "probabilities");
}

int launch_collapse(qsim_state *s, int qubit, int outcome, double scale)
{
    const uint64_t N = 1ull << s->n;
    const uint64_t nvec = (s->dtype == SIM_C128) ? N : N / 2;
    const unsigned g = grid_for(nvec, 256, s->num_sms);
    launch_begin(s, KC_COLLAPSE, 1.5 * (double)s->bytes);
    if (s->dtype == SIM_C128)
        k_collapse<double><<<g, 256, 0, s->stream>>>((double *)s->amps, nvec, qubit, outcome, scale);
    else
        k_collapse<float><<<g, 256, 0, s->stream>>>((float *)s->amps, nvec, qubit, outcome, (float)scale);
    return launch_end(s, "collapse");
}

bool sample_observe_fused(const qsim_state *s)
{
    return s->dtype == SIM_C64 && s->n >= kSampleLog && SubGeo(1ull << kSampleLog).sub == 256;
}

// The pass over the state writes the sums of its eighths (8 bytes per 32 amplitudes:
// 8-11 % of its time for complex64) where the shots pay for them: a shot reads 256 bytes
// with them and 2 KB without (512 and 4 KB).  For a million shots, with / without (and
// one shot in a warp, sorted by block, before there were eighths): complex64 28 qubits 0.80 / 1.26 (1.83)
// ms, 30 2.31 / 2.65 (3.37), 33 16.2 / 15.2 (16.1); complex128 30 4.36 / 5.23 (7.84).  For 10^4:
// 0.69 / 0.62 (0.65), 2.20 / 1.97 (2.01), 16.1 / 14.4 (14.6); 4.14 / 3.93 (3.96).  The two
// are even at about one shot in 2300 amplitudes (complex64, 27 qubits and more) and
// one in 3600-6700 (complex128).
constexpr uint64_t kEighthsPer64 = 2048, kEighthsPer128 = 4096;

int run_sample(qsim_state *s, uint64_t shots, uint64_t seed, uint64_t *out, int out_on_device, double *norm_out,
               double *expz_out)
{
    if (shots == 0) return SIM_OK;
    const bool obs = expz_out != nullptr;
    if (obs && !sample_observe_fused(s)) return fail(SIM_EINVAL, "sample with <sum Z>: complex64, n >= 13 only");
    if (shots > 0xFFFFFFFFull) return fail(SIM_EINVAL, "sim_sample: at most 2^32 - 1 shots per call");
    const uint64_t N = 1ull << s->n;
    const uint64_t bs = (s->n >= kSampleLog) ? (1ull << kSampleLog) : N;
    const uint64_t nb = N / bs;
    const SubGeo sg(bs);
    // scratch: scanned sub-sums and eighths of full sub-blocks, block sums and
    // their scans (nb doubles each), total, last block and <sum Z>, chunk
    // totals and offsets of the scan, shots for host output
    const bool full = sg.sub == (1u << kSubLog);
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
    const size_t o_cum = take(nb * sg.nsub * 8);
    const size_t o_bsum = take(nb * 8), o_bexcl = take(nb * 8), o_bincl = take(nb * 8), o_tot = take(4 * 8);
    const uint64_t nchunk = (nb + kScanChunk - 1) / kScanChunk;
    const size_t o_cs = take(2 * nchunk * 8);
    const size_t o_zpart = obs ? take(2 * nb * 8) : 0;
    const size_t o_out = out_on_device ? 0 : take(shots * 8);
    const bool c128 = s->dtype == SIM_C128;
    bool stored = full && shots >= N / (c128 ? kEighthsPer128 : kEighthsPer64);
    const size_t o_eig = off;
    char *scratch = nullptr;
    if (stored && cudaMallocAsync((void **)&scratch, off + nb * sg.nsub * 64, s->stream) != cudaSuccess) {
        cudaGetLastError();
        stored = false;                // the eighths do not fit beside the state: do without
    }
    if (!stored) QSIM_CUDA(cudaMallocAsync((void **)&scratch, off, s->stream));
    double *cum = (double *)(scratch + o_cum), *eighth = stored ? (double *)(scratch + o_eig) : nullptr;
    double *bsum = (double *)(scratch + o_bsum), *bexcl = (double *)(scratch + o_bexcl);
    double *bincl = (double *)(scratch + o_bincl);
    double *tot = (double *)(scratch + o_tot), *zout = tot + 2;        // zout: two values
    uint64_t *last = (uint64_t *)(tot + 1);
    uint64_t *dout = out_on_device ? out : (uint64_t *)(scratch + o_out);
    double *cs = (double *)(scratch + o_cs);
    double *zpart = obs ? (double *)(scratch + o_zpart) : nullptr;
    const ShotTables tables{sg.nsub, nb, bexcl, bincl, cum, last};
    int rc = SIM_OK;
    do {
        launch_begin(s, KC_SAMPLE, (double)s->bytes);
        if (c128) k_sub_sums<double><<<(unsigned)nb, 256, 0, s->stream>>>((const double *)s->amps, bs, cum, bsum, eighth);
        else if (obs)
            k_sub_sums<float, true><<<(unsigned)nb, 256, 0, s->stream>>>((const float *)s->amps, bs, cum, bsum, eighth,
                                                                       s->n, zpart);
        else k_sub_sums<float><<<(unsigned)nb, 256, 0, s->stream>>>((const float *)s->amps, bs, cum, bsum, eighth);
        if ((rc = launch_end(s, "sub-block sums"))) break;
        if (obs) {
            launch_begin(s, KC_REDUCE);
            k_final_sum<<<1, kRedThreads, 0, s->stream>>>(zpart, (int)nb, zout);
            if ((rc = launch_end(s, "<sum Z> total"))) break;
        }
        if ((rc = scan_sums<double>(s, bsum, bexcl, bincl, nb, tot, cs, "block scan"))) break;
        launch_begin(s, KC_SAMPLE);
        k_last_nonzero<<<1, 1024, 0, s->stream>>>(bsum, nb, last);
        if ((rc = launch_end(s, "last nonzero"))) break;
        // per shot 32 amplitudes (256 without the eighths); a zero norm writes none
        launch_begin(s, KC_SAMPLE, (double)shots * (stored ? 32.0 : full ? 256.0 : 0.0) * (c128 ? 16.0 : 8.0));
        const unsigned grid = grid_for(full && !stored ? 8 * shots : shots, 256, s->num_sms);
        if (stored && c128)
            k_shots<double><<<grid, 256, 0, s->stream>>>((const double *)s->amps, tables, seed, tot, eighth, shots, dout);
        else if (stored)
            k_shots<float><<<grid, 256, 0, s->stream>>>((const float *)s->amps, tables, seed, tot, eighth, shots, dout);
        else if (full && c128)
            k_shots_read<double><<<grid, 256, 0, s->stream>>>((const double *)s->amps, tables, seed, tot, shots, dout);
        else if (full)
            k_shots_read<float><<<grid, 256, 0, s->stream>>>((const float *)s->amps, tables, seed, tot, shots, dout);
        else if (c128)
            k_shots_small<double><<<grid, 256, 0, s->stream>>>((const double *)s->amps, (uint32_t)N, seed, tot, shots,
                                                               dout);
        else
            k_shots_small<float><<<grid, 256, 0, s->stream>>>((const float *)s->amps, (uint32_t)N, seed, tot, shots,
                                                              dout);
        if ((rc = launch_end(s, "shots"))) break;
        double *host = s->host_red;
        if (cudaMemcpyAsync(host, tot, (obs ? 3 : 1) * 8, cudaMemcpyDeviceToHost, s->stream) != cudaSuccess ||
            cudaStreamSynchronize(s->stream) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "sample readback");
            break;
        }
        if (norm_out) *norm_out = host[0];
        if (expz_out) *expz_out = host[2];
        if (!(host[0] > 0.0)) { rc = fail(SIM_EINVAL, "sim_sample: the state has zero norm"); break; }
        if (!out_on_device) {
            if (cudaMemcpyAsync(out, dout, shots * 8, cudaMemcpyDeviceToHost, s->stream) != cudaSuccess) {
                rc = cuda_fail(cudaGetLastError(), "shots readback");
                break;
            }
        }
    } while (0);
    cudaFreeAsync(scratch, s->stream);
    if (rc == SIM_OK && !out_on_device) QSIM_CUDA(cudaStreamSynchronize(s->stream));
    return rc;
}

}  // namespace qsim
