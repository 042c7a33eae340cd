// Plain conjugate gradients on M^T M v = b with the whole iteration state of a
// right-hand side on chip: one thread-block cluster per right-hand side, one
// launch per solve. The two-kernel iteration streams the same state through L2
// (or, past 129 MB, HBM) twice per iteration and pays two launches' latencies.
//
// Work split. A cluster of CS blocks owns one right-hand side; block c owns the
// slices [T c / CS, T (c + 1) / CS). A lane group (RGeo) holds one slice: every
// lane a two-column strip of one chunk of rows, so one shuffle pair per row
// serves the odd x-bonds. r and the vector being formed (M r, then A r) stay in
// registers; p, x and the diagonal stay in tensor memory (or shared memory and
// registers, where 16 values per lane or fewer are held); s = A p in shared
// memory, in the lanes' own order. The slices of a block meet in one exchange
// buffer: slot j takes C r_{t-1} for slice j, then (once slice j has read it)
// C^T s D w of slice j for slice j - 1: one slot per slice and one more.
//
// Iteration. The single-reduction form of CG (Chronopoulos and Gear): from
// u = A r, gamma = (r, r) and delta = (r, A r) = |M r|^2 follow beta, alpha and
// then s = u + beta s, p = r + beta p, x += alpha p, r -= alpha s. Each block
// also keeps r and s of its two neighbour slices, updated from their u, so that
// an iteration crosses the cluster once: two sums per block and two boundary
// slices, all asynchronous and awaited together.
//
// Scale. The iteration runs on b over a power of two near |b| (pow2_hi), so it
// takes the same steps whatever the scale of b.
//
// Control. After every check_every iterations the recursive residual is
// compared with tol; at the check after the first one below tol, as in the
// two-kernel iteration, or after reliable_every iterations, x is folded into the FP64 solution and r is replaced by the FP64 true residual (the
// reliable update of cg_solve), computed by the same cluster. p is kept and
// re-conjugated, beta = -(r, A p) / (p, A p), with A p formed anew. Clusters take
// right-hand sides from a table of states (ready / running / done), fewest
// iterations first; between two segments a cluster hands its unfinished
// right-hand side back when another one is ready and continues with it
// otherwise, so nothing ever waits for work. Which cluster runs a segment does
// not change its arithmetic.
//
// Bounds and measurements (GB300, us per iteration of all right-hand sides,
// solves to 1e-10, against the two-kernel iteration): L = 4, Ltau = 40, 1 rhs
// 1.5 / 8.6 (a chain of block barriers and the scalar step, some 3000 cycles);
// L = 16, Ltau = 160, 2 rhs 2.6 / 9.8; L = 28, Ltau = 120, 128 rhs 52 / 101
// and L = 32, Ltau = 200, 16 rhs 14.3 / 22 (issue slots and shared memory of the
// multiprocessors that clusters of 9 and 16 blocks reach, 135 and 112 of 152; a
// quarter of it the FP64 true residual, bound by the FP64 pipes). FP64
// iterations, L = 4: 5.5 / 11.7.
#pragma once

#include <cooperative_groups.h>
#include <string.h>

#include "cb.cuh"
#include "internal.cuh"
#include "strip.cuh"

namespace hol {

// Launch parameters of one solve.
struct ResArgs {
    const double* b;       // [n_rhs][T][N]
    double* v;             // solution, FP64
    void* r;               // saved state between segments, [n_rhs][T][N] (float or double)
    void* p;
    double* t64;           // scratch of the true residual, [n_rhs][T][N]
    const void* ev;        // exp(-dtau V) in the iteration's precision
    const double* ev64;
    int T, n_rhs, max_iter, chk, rel_every;
    int slots;             // most slices of one block
    int tm_cols;           // tensor-memory columns (TM instances)
    int wait_tries;        // of a wait for the other blocks (mb_wait)
    double tol, th;
    DcgState d;
};

enum ResState { RS_READY = 0, RS_RUNNING = 1, RS_DONE = 2 };

// A kernel instance: values stored per slice, slices per warp and register set,
// values per lane, and the kernel (null when that K is not built).
struct ResKernel {
    int sl, g, e;
    void (*fn)(ResArgs);
};
// tm: the variant with x and p in tensor memory (FP32, at least 16 values per lane)
ResKernel resident_kernel_f32_large(int L, int K, bool tm);   // resident32l.cu: L >= 24
ResKernel resident_kernel_f32_mid(int L, int K, bool tm);     // resident32m.cu: 14 <= L <= 22
ResKernel resident_kernel_f32_small(int L, int K, bool tm);   // resident32s.cu: L <= 12
ResKernel resident_kernel_f64(int L, int K);                  // resident64.cu: L <= 20

namespace {

namespace cgp = cooperative_groups;

// Sums of the iteration's dot products: a compensated float pair in the FP32
// iteration (cb.cuh), FP64 in the FP64 one. (r, r) is summed in FP32 by groups of
// four, as in the two-kernel iteration, |M r|^2 by two chains per lane and
// slice (one there). The partials of a reduction are sums of many terms of
// similar size, so their pairs are added without renormalising: only the leading
// sums form the dependent chain. Relative error of (r, r) against 64 bits, rms over
// 200 random vectors of n = 640 / 7,680 / 40,960 / 94,080 / 204,800 values: 38 / 10 / 4.6 /
// 3.0 / 2.1 e-10, the two-kernel sums (pairs in a block, FP64 over the blocks) the same
// digits, since the products' own rounding is nearly all of it; with two long chains per
// lane 36 / 14 / 9.5 / 9.3 / 6.6 e-10. The groups cost 2 % of the iteration at L = 28 and 32.
template <typename R>
struct Acc;
template <>
struct Acc<float> {
    using T = F2;
    static __device__ __forceinline__ T zero() { return F2{0.0f, 0.0f}; }
    static __device__ __forceinline__ T add(T a, T b)
    {
        const F2 s = f2_two_sum(a.hi, b.hi);
        return F2{s.hi, s.lo + (a.lo + b.lo)};
    }
    static __device__ __forceinline__ T addv(T a, float b)
    {
        const F2 s = f2_two_sum(a.hi, b);
        return F2{s.hi, s.lo + a.lo};
    }
    static __device__ __forceinline__ T shfl(T a, int o)
    {
        return F2{__shfl_xor_sync(kFull, a.hi, o), __shfl_xor_sync(kFull, a.lo, o)};
    }
    static __device__ __forceinline__ double val(T a) { return f2_to_double(a); }
    // 2: not finite, 1: below the limit, else 0
    static __device__ __forceinline__ int stop(T a, double limit)
    {
        const float h = (float)limit;
        return !isfinite(a.hi) ? 2 : (a.hi - h) + a.lo < 0.0f ? 1 : 0;
    }
};
template <>
struct Acc<double> {
    using T = double;
    static __device__ __forceinline__ T zero() { return 0.0; }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    static __device__ __forceinline__ T addv(T a, double b) { return a + b; }
    static __device__ __forceinline__ T shfl(T a, int o) { return __shfl_xor_sync(kFull, a, o); }
    static __device__ __forceinline__ double val(T a) { return a; }
    static __device__ __forceinline__ int stop(T a, double limit)
    {
        return !isfinite(a) ? 2 : a < limit ? 1 : 0;
    }
};

// The scalars of the single-reduction iteration, formed by one warp of every
// block. With gamma = (r, r) and delta = (r, A r): beta = gamma / gamma_old,
// (p, A p) = delta - beta gamma / alpha_old, alpha = gamma / (p, A p). Kept
// between iterations: ig = 1 / gamma and kap = 1 / (gamma alpha) of the last
// one. FP32 iteration: pairs of floats throughout (some 45 bits), because an
// FP64 division is ten dependent operations on the scarce FP64 pipe, between
// the reduction and the update. Before the rounding to FP32 that alpha and beta
// take in either iteration the pairs are off by at most 6e-14 (beta) and 1e-13 times
// delta / (p, A p) (alpha) over 200,000 random steps; after it not one differs from the
// rounded 64-bit quotient. A ratio that is not finite is 0, as cg_ratio's.
__device__ __forceinline__ F2 p_norm(float h, float l)
{
    const float s = h + l;
    return F2{s, l - (s - h)};
}
__device__ __forceinline__ F2 p_mul(F2 a, F2 b)
{
    const float h = a.hi * b.hi;
    return p_norm(h, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -h))));
}
// 1 / a: the hardware's approximate reciprocal and one Newton step in pairs
__device__ __forceinline__ F2 p_inv(F2 a)
{
    float q;
    asm("rcp.approx.f32 %0, %1;" : "=f"(q) : "f"(a.hi));
    const float e = fmaf(-q, a.lo, fmaf(-q, a.hi, 1.0f));   // 1 - q a
    return p_norm(q, q * e);
}
template <typename R>
struct Steps;
template <>
struct Steps<float> {
    F2 ig, kap;
    __device__ __forceinline__ void start()
    {
        ig = F2{0.0f, 0.0f};
        kap = F2{0.0f, 0.0f};
    }
    // given: beta already chosen with (p, A p) = delta + corr (restart)
    __device__ __forceinline__ void step(F2 g, F2 d, bool given, float beta_in, double corr,
                                         float& alpha, float& beta)
    {
        g = p_norm(g.hi, g.lo);
        d = p_norm(d.hi, d.lo);
        if (given) {
            beta = beta_in;
            const double t = f2_to_double(d) + corr;
            pap.hi = (float)t;
            pap.lo = (float)(t - (double)pap.hi);
        } else {
            const F2 b2 = p_mul(g, ig);
            beta = b2.hi + b2.lo;
            const F2 t = p_mul(g, p_mul(g, kap));
            const F2 s2 = f2_two_sum(d.hi, -t.hi);
            pap = p_norm(s2.hi, s2.lo + (d.lo - t.lo));
        }
        const F2 a2 = p_mul(g, p_inv(pap));
        alpha = a2.hi + a2.lo;
        if (!isfinite(alpha)) alpha = 0.0f;
        if (!isfinite(beta)) beta = 0.0f;
    }
    // what the next step needs, off the way to this one's update
    __device__ __forceinline__ void keep(F2 g)
    {
        ig = p_inv(p_norm(g.hi, g.lo));
        kap = p_mul(p_mul(pap, ig), ig);
    }
    F2 pap;
};
template <>
struct Steps<double> {
    double ig, kap, pap;
    __device__ __forceinline__ void start()
    {
        ig = 0.0;
        kap = 0.0;
    }
    __device__ __forceinline__ void step(double g, double d, bool given, double beta_in, double corr,
                                         double& alpha, double& beta)
    {
        if (given) {
            beta = beta_in;
            pap = d + corr;
        } else {
            beta = g * ig;
            pap = d - g * (g * kap);
        }
        if (!isfinite(beta)) beta = 0.0;
        alpha = cg_ratio(g, pap);
    }
    __device__ __forceinline__ void keep(double g)
    {
        ig = 1.0 / g;
        kap = (pap * ig) * ig;
    }
};

// Tensor memory as the lanes' private store: column c of a warp's window is
// one more 32-bit register of every lane. x and p go there (TM): nothing but
// their own lane ever reads them, and shared memory's bandwidth, which bounds
// the iteration, is left to the exchange. N columns of two windows at a time; a
// pass that reads what an earlier pass stored starts with tm_stored().
__device__ __forceinline__ void tm_stored()
{
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void tm_ld2(unsigned a, unsigned b, float (&p)[N], float (&x)[N])
{
    static_assert(N == 4 || N == 8, "columns per access");
    unsigned u[N], v[N];
    if constexpr (N == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%8];\n"
                     "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%9];\n"
                     "tcgen05.wait::ld.sync.aligned;\n"
                     : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(v[0]), "=r"(v[1]),
                       "=r"(v[2]), "=r"(v[3])
                     : "r"(a), "r"(b)
                     : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n"
                     "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n"
                     "tcgen05.wait::ld.sync.aligned;\n"
                     : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]),
                       "=r"(u[6]), "=r"(u[7]), "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]),
                       "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                     : "r"(a), "r"(b)
                     : "memory");
#pragma unroll
    for (int k = 0; k < N; ++k) {
        p[k] = __uint_as_float(u[k]);
        x[k] = __uint_as_float(v[k]);
    }
}
template <int N>
__device__ __forceinline__ void tm_st(unsigned a, const float (&p)[N])
{
    if constexpr (N == 4)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(a),
                     "r"(__float_as_uint(p[0])), "r"(__float_as_uint(p[1])),
                     "r"(__float_as_uint(p[2])), "r"(__float_as_uint(p[3]))
                     : "memory");
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(a),
                     "r"(__float_as_uint(p[0])), "r"(__float_as_uint(p[1])),
                     "r"(__float_as_uint(p[2])), "r"(__float_as_uint(p[3])),
                     "r"(__float_as_uint(p[4])), "r"(__float_as_uint(p[5])),
                     "r"(__float_as_uint(p[6])), "r"(__float_as_uint(p[7]))
                     : "memory");
}

// Within the iterations the blocks of a cluster exchange their sums as
// asynchronous remote stores and their boundary slices as bulk copies between
// shared memories; both complete on a barrier of the receiving block, whose wait
// is the only one (a cluster barrier costs a fence of everything before it, some
// thousand cycles, each time). Two barriers take turns: a block two exchanges
// ahead of another cannot exist, one ahead can. A cluster's blocks are resident
// together, so a wait ends by completion; it is bounded all the same (wait_tries of
// kMbTryNs each). A block whose wait runs out ends its segment and waits once more,
// kMbDrain tries, for the copies on their way to it; the others then run out of
// their waits, so every block reaches the cluster barriers that follow, and the solve
// ends with HOL_ETIMEOUT.
__device__ __forceinline__ unsigned sm_addr(const void* p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned sm_remote(unsigned a, int rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void mb_init(unsigned mb, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mb), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mb_expect(unsigned mb, int bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mb), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_push(unsigned dst, unsigned src, int bytes, unsigned mb)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, "
                 "[%3];\n" ::"r"(dst),
                 "r"(src), "r"(bytes), "r"(mb)
                 : "memory");
}
template <typename T8>
__device__ __forceinline__ void st_async8(unsigned dst, T8 v, unsigned mb)
{
    static_assert(sizeof(T8) == 8, "one 8-byte value");
    unsigned long long u;
    memcpy(&u, &v, 8);
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n" ::"r"(dst),
                 "l"(u), "r"(mb)
                 : "memory");
}
constexpr int kMbTryNs = 20000;
constexpr int kMbDrain = 50000;     // one second
__device__ __forceinline__ bool mb_wait(unsigned mb, int parity, int tries)
{
    for (int k = 0; k < tries; ++k) {
        int ok;
        asm volatile("{\n.reg .pred p;\n"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
                     "selp.b32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok)
                     : "r"(mb), "r"(parity), "r"(kMbTryNs)
                     : "memory");
        if (ok) return true;
    }
    return false;
}

// After a wait that ran out: waits for what is still on its way into this block
// (barriers mb[0], mb[1], exchanges so far n), then sets the flag in every block of the
// cluster. Out of line: inlined, never executed, it changed the iteration's code
// (L = 18, Ltau = 160, 8 rhs: 3.40 -> 3.66 us per iteration).
static __device__ __noinline__ void mb_gave_up(unsigned mb, unsigned n, unsigned flag, int cs)
{
    if ((int)threadIdx.x >= cs) return;
    for (unsigned x = n > 2 ? n - 2 : 0; x < n; ++x) mb_wait(mb + 8 * (x & 1), (int)(x >> 1) & 1, kMbDrain);
    asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(sm_remote(flag, threadIdx.x)), "r"(1) : "memory");
}

// A right-hand side is solved as b / 2^ex, ex the exponent of |b|, so that the FP32
// sums and their reciprocals stay in range whatever the scale of b. Every vector on
// chip and v between segments are on that scale; v goes back to b's with the last
// segment. All exact. The exponent is kept as a difference of high words, ex << 20.
__device__ __forceinline__ unsigned exp_hi(double x) { return ((unsigned)__double2hiint(x) & 0x7ff00000u) - 0x3ff00000u; }
__device__ __forceinline__ double pow2_hi(unsigned xs) { return __hiloint2double((int)(0x3ff00000u + xs), 0); }

// FP32 <-> FP64 on the integer pipes for the usual exponents: a conversion
// instruction takes the FP64 pipe as long as an addition. Same values (round to
// nearest even); zeros, subnormals, infinities and NaN take the instruction.
__device__ __forceinline__ double to_f64(float x)
{
    const unsigned u = __float_as_uint(x);
    if (((u >> 23) & 255u) - 1u < 254u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                                (int)(u << 29));
    return (double)x;
}
__device__ __forceinline__ double to_f64(double x) { return x; }
template <typename R>
__device__ __forceinline__ R from_f64(double x);
template <>
__device__ __forceinline__ double from_f64<double>(double x) { return x; }
template <>
__device__ __forceinline__ float from_f64<float>(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e - 897u < 253u) {   // a normal float even after rounding up
        const unsigned m = ((hi & 0x7fffffffu) - (896u << 20)) << 3 | lo >> 29;
        const unsigned rem = lo << 3;                      // what falls off, left aligned
        const unsigned up = rem > 0x80000000u || (rem == 0x80000000u && (m & 1u));
        return __uint_as_float((hi & 0x80000000u) | (m + up));
    }
    return (float)x;
}

// A lane's E values of one slot, in the lanes' own order: four at a time, the
// lanes of a slice side by side.
template <typename R, int L>
__device__ __forceinline__ void slot_ld(const R* s, int ll, R (&v)[RGeo<L>::E])
{
    using K = RGeo<L>;
    using V2 = typename Vec2<R>::T;
#pragma unroll
    for (int e = 0; e < K::E; e += 4) {
        const R* q = s + (e * K::LS + 4 * ll);
        if constexpr (sizeof(R) == 4) {
            const float4 t = *reinterpret_cast<const float4*>(q);
            v[e] = t.x; v[e + 1] = t.y; v[e + 2] = t.z; v[e + 3] = t.w;
        } else {
            const V2 t0 = *reinterpret_cast<const V2*>(q), t1 = *reinterpret_cast<const V2*>(q + 2);
            v[e] = t0.x; v[e + 1] = t0.y; v[e + 2] = t1.x; v[e + 3] = t1.y;
        }
    }
}
template <typename R, int L>
__device__ __forceinline__ void slot_st(R* s, int ll, const R (&v)[RGeo<L>::E])
{
    using K = RGeo<L>;
    using V2 = typename Vec2<R>::T;
#pragma unroll
    for (int e = 0; e < K::E; e += 4) {
        R* q = s + (e * K::LS + 4 * ll);
        if constexpr (sizeof(R) == 4) {
            *reinterpret_cast<float4*>(q) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        } else {
            V2 t0, t1;
            t0.x = v[e]; t0.y = v[e + 1]; t1.x = v[e + 2]; t1.y = v[e + 3];
            *reinterpret_cast<V2*>(q) = t0;
            *reinterpret_cast<V2*>(q + 2) = t1;
        }
    }
}

// CH of them, from value e on
template <typename R, int L, int CH>
__device__ __forceinline__ void slot_get(const R* s, int ll, int e, R (&v)[CH])
{
    using V2 = typename Vec2<R>::T;
#pragma unroll
    for (int q = 0; q < CH; q += 4) {
        const R* p = s + ((e + q) * RGeo<L>::LS + 4 * ll);
        if constexpr (sizeof(R) == 4) {
            const float4 t = *reinterpret_cast<const float4*>(p);
            v[q] = t.x; v[q + 1] = t.y; v[q + 2] = t.z; v[q + 3] = t.w;
        } else {
            const V2 t0 = *reinterpret_cast<const V2*>(p), t1 = *reinterpret_cast<const V2*>(p + 2);
            v[q] = t0.x; v[q + 1] = t0.y; v[q + 2] = t1.x; v[q + 3] = t1.y;
        }
    }
}
template <typename R, int L, int CH>
__device__ __forceinline__ void slot_put(R* s, int ll, int e, const R (&v)[CH])
{
    using V2 = typename Vec2<R>::T;
#pragma unroll
    for (int q = 0; q < CH; q += 4) {
        R* p = s + ((e + q) * RGeo<L>::LS + 4 * ll);
        if constexpr (sizeof(R) == 4) {
            *reinterpret_cast<float4*>(p) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
        } else {
            V2 t0, t1;
            t0.x = v[q]; t0.y = v[q + 1]; t1.x = v[q + 2]; t1.y = v[q + 3];
            *reinterpret_cast<V2*>(p) = t0;
            *reinterpret_cast<V2*>(p + 2) = t1;
        }
    }
}

template <typename R, int L, int K, bool TM>
__global__ void __launch_bounds__(512, 1) k_cg_resident(ResArgs a)
{
    using Geo = RGeo<L>;
    using A = Acc<R>;
    using AT = typename A::T;
    using V2 = typename Vec2<R>::T;
    constexpr int E = Geo::E, RT = Geo::RT, SL = Geo::SL, G = Geo::G, N = L * L;
    constexpr int CH = E % 8 == 0 ? 8 : 4;      // values per step of the update
    const cgp::cluster_group cl = cgp::this_cluster();
    const int cs = (int)cl.num_blocks(), crank = (int)cl.block_rank();
    const int nw = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Geo geo;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // slots of one slice: [exchange: slots + 1][s: slots + 2][boundary
    // slices out: 2 x 2, in: 2 x 2] and,
    // without tensor memory, [p: slots][x: slots]; the FP64 exchange of the true
    // residual takes the first two in the FP32 iteration (s is rebuilt after it)
    R* ex = reinterpret_cast<R*>(smem_raw);
    R* ss = ex + (long)(a.slots + 1) * SL;
    R* hb = ss + (long)(a.slots + 2) * SL;
    R* hin = hb + 4L * SL;
    R* ps = hin + 4L * SL;
    R* xs = ps + (long)a.slots * SL;
    double* ex64 = reinterpret_cast<double*>(smem_raw);
    const R* hb_prev;   // the neighbour blocks' boundary slices
    const R* hb_next;
    __shared__ AT red_w[2][16];           // [sum][warp of the block]
    __shared__ AT red_c[2][2][16];        // [parity][sum][block of the cluster]
    __shared__ double red64[2][16 * 16];
    __shared__ R s_step[2];               // alpha, beta
    __shared__ int s_stop;                // 1: end of the segment, 2: not finite, 3: a wait ran out
    __shared__ __align__(8) unsigned long long s_mb[2];
    __shared__ int s_item;
    __shared__ int s_lost;                // a wait of some block of the cluster ran out
    // |b|, (tol |b|)^2 on the scale of r, the exponent of |b| (pow2_hi): of the item in
    // hand, here and not in registers of the iteration
    __shared__ double s_bnorm, s_limit;
    __shared__ unsigned s_bxs;
    __shared__ unsigned s_tm;

    const int t0 = (int)((long)a.T * crank / cs), t1 = (int)((long)a.T * (crank + 1) / cs);
    const int nc = t1 - t0;
    const int prev = crank == 0 ? cs - 1 : crank - 1, next = crank + 1 == cs ? 0 : crank + 1;
    const int prev_nc = (int)((long)a.T * (prev + 1) / cs) - (int)((long)a.T * prev / cs);
    hb_prev = cl.map_shared_rank(hb, prev);
    hb_next = cl.map_shared_rank(hb, next);
    // lane groups hold the slices -1 .. nc (-1 and nc: copies of the neighbour
    // blocks' last and first slice, which this block updates for itself)
    auto slice = [&](int k) { return (wid * K + k) * G + geo.g - 1; };
    auto held = [&](int k) { return geo.ok && slice(k) <= nc; };
    auto own = [&](int k) { return geo.ok && slice(k) >= 0 && slice(k) < nc; };
    auto tau_of = [&](int j) {
        const int t = t0 + j;
        return t < 0 ? t + a.T : t >= a.T ? t - a.T : t;
    };

    // tensor-memory window of this warp (its lane quarter; K E columns each of p,
    // x and s D)
    unsigned tmw = 0;
    const int tm_cols = TM ? a.tm_cols : 0;
    if constexpr (TM) {
        if (wid == 0) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(&s_tm);
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(dst),
                         "r"(tm_cols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        }
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        tmw = s_tm + ((unsigned)(wid & 3) << 21) + (unsigned)((wid >> 2) * (3 * K * E));
    }
    auto tp = [&](int k, int e) { return tmw + (unsigned)(k * E + e); };
    auto tx = [&](int k, int e) { return tmw + (unsigned)((K + k) * E + e); };
    auto td = [&](int k, int e) { return tmw + (unsigned)((2 * K + k) * E + e); };
    auto get_tm = [&](unsigned at, R (&v)[E]) {
        if constexpr (TM) {
#pragma unroll
            for (int e = 0; e + CH < E; e += 2 * CH) {
                R u[CH], v2[CH];
                tm_ld2<CH>(at + e, at + e + CH, u, v2);
#pragma unroll
                for (int q = 0; q < CH; ++q) {
                    v[e + q] = u[q];
                    v[e + CH + q] = v2[q];
                }
            }
            if constexpr ((E / CH) % 2 == 1) {
                R u[CH], v2[CH];
                tm_ld2<CH>(at + E - CH, at + E - CH, u, v2);
#pragma unroll
                for (int q = 0; q < CH; ++q) v[E - CH + q] = u[q];
            }
        }
    };
    // the lane's p of set k (every lane of the warp calls it)
    auto get_p = [&](int k, R (&p)[E]) {
        if constexpr (TM) {
            tm_stored();
            get_tm(tp(k, 0), p);
        } else {
            if (own(k)) slot_ld<R, L>(ps + (long)slice(k) * SL, geo.ll, p);
        }
    };

    const R th = (R)a.th;
    const R* ev = reinterpret_cast<const R*>(a.ev);
    R* rsave = reinterpret_cast<R*>(a.r);
    R* psave = reinterpret_cast<R*>(a.p);
    R r[K][E], w[K][E];
    // s D of the slices: in tensor memory beside p and x, in registers (FP32
    // without tensor memory), or read again (FP64, bound by its arithmetic): a
    // cluster barrier drops the L1 lines, so a load in the iteration is one of
    // L2 latency ahead of a block barrier
    constexpr bool DREG = sizeof(R) == 4 && !TM;
    R dreg[DREG ? K : 1][DREG ? E : 1];
    auto load_d = [&](int k, int q) -> V2 {
        V2 d;
        d.x = d.y = R(0);
        const int j = slice(k);
        if (held(k) && j >= 0 && geo.has(q)) {
            const int tau = tau_of(j);
            d = __ldg(reinterpret_cast<const V2*>(ev + (long)tau * N + geo.site(q)));
            if (tau != 0) {
                d.x = -d.x;
                d.y = -d.y;
            }
        }
        return d;
    };
    if constexpr (TM || DREG) {
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int e = 0; e < E; e += CH) {
                R u[CH];
#pragma unroll
                for (int q = 0; q < CH; q += 2) {
                    const V2 d = load_d(k, (e + q) / 2);
                    u[q] = d.x;
                    u[q + 1] = d.y;
                    if constexpr (DREG) {
                        dreg[k][e + q] = d.x;
                        dreg[k][e + q + 1] = d.y;
                    }
                }
                if constexpr (TM) tm_st<CH>(td(k, e), u);
            }
    }
    if constexpr (TM) tm_stored();

    // The sums over the cluster of two partials per lane, in warp 0 of every
    // block: lanes below 16 carry the first, the others the second; warps, then
    // blocks, always in the same order. Every block has passed its barrier when
    // its sums arrive, so its boundary slices are written and its reads of the
    // previous exchange done; the parity keeps a fast block's next sums off a slow
    // one's read. One warp does the scalar work: in every warp it cost more issue
    // slots than the barrier it saves.
    int par = 0;
    if (threadIdx.x < 2) mb_init(sm_addr(&s_mb[threadIdx.x]), 1);
    if (threadIdx.x == 0) s_stop = s_lost = 0;
    cl.sync();
    bool lost = false;      // a wait of this block ran out (warp 0; never in a working cluster)
    unsigned mbk = 0;       // exchanges so far: barrier mbk & 1, its phase mbk >> 1
    auto half_sum = [&](AT v) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v = A::add(v, A::shfl(v, o));
        return v;
    };
    auto reduce = [&](AT& x0, AT& x1) {
        const int which = lane >> 4, l16 = lane & 15;
        AT v = which ? x1 : x0;
        v = half_sum(A::add(v, A::shfl(which ? x0 : x1, 16)));
        if (l16 == 0) red_w[which][wid] = v;
        __syncthreads();
        if (wid == 0) {
            v = half_sum(l16 < nw ? red_w[which][l16] : A::zero());
            if (cs > 1) {
                const unsigned mb = sm_addr(&s_mb[mbk & 1]);
                if (lane == 0) mb_expect(mb, 16 * cs + 2 * SL * (int)sizeof(R));
                if (l16 < cs)
                    st_async8(sm_remote(sm_addr(&red_c[par][which][crank]), l16), v,
                              sm_remote(mb, l16));
                if (!lost) lost = !mb_wait(mb, (int)(mbk >> 1) & 1, a.wait_tries);
                v = half_sum(l16 < cs ? red_c[par][which][l16] : A::zero());
            }
            const AT o = A::shfl(v, 16);
            x0 = which ? o : v;
            x1 = which ? v : o;
        }
        ++mbk;
        par ^= 1;
    };
    int par64 = 0;
    auto reduce64 = [&](double x0) -> double {
        x0 = warp_sum(x0);
        if (lane < cs) *cl.map_shared_rank(&red64[par64][crank * nw + wid], lane) = x0;
        cl.sync();
        double s = 0.0;
        for (int k = lane; k < cs * nw; k += 32) s += red64[par64][k];
        s = warp_sum(s);
        par64 ^= 1;
        return s;
    };
    // Boundary slices, [parity][0: the block's first, 1: its last] on their way
    // out: pushed into the neighbours' `in` slots as part of the next reduction,
    // or read by the neighbours after a cluster barrier (between iterations). The
    // parity alternates with every exchange.
    int hpar = 0;
    auto halo_send = [&](int k, const R (&v)[E], bool push) {
        const int j = slice(k);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const bool mine = own(k) && j == (side == 0 ? 0 : nc - 1);
            R* src = hb + (long)(2 * hpar + side) * SL;
            if (mine) slot_st<R, L>(src, geo.ll, v);
            if (push && cs > 1 && __any_sync(kFull, mine)) {
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if (mine && geo.ll == 0) {
                    const int to = side == 0 ? prev : next;   // its slice after / before its own
                    bulk_push(sm_remote(sm_addr(hin + (long)(2 * hpar + 1 - side) * SL), to), sm_addr(src),
                              SL * (int)sizeof(R), sm_remote(sm_addr(&s_mb[mbk & 1]), to));
                }
            }
        }
    };
    // the copies' new values: in [parity][0: slice -1, 1: slice nc], or the
    // neighbours' outgoing slots
    auto halo_recv = [&](int k, int hp, R (&v)[E], bool pushed) {
        if (held(k) && !own(k)) {
            const bool first = slice(k) < 0;
            const R* s = pushed && cs > 1 ? hin + (long)(2 * hp + (first ? 0 : 1)) * SL
                         : first          ? hb_prev + (long)(2 * hp + 1) * SL
                                          : hb_next + (long)(2 * hp + 0) * SL;
            slot_ld<R, L>(s, geo.ll, v);
        }
    };
    // w <- A v on the own slices (v: r, or with `conj` the operand already in
    // w); returns the lane's |M v|^2. The boundary slices go to the neighbours'
    // halo slots.
    auto apply = [&](bool conj) -> AT {
#pragma unroll
        for (int k = 0; k < K; ++k) {   // C v to the successor
            const int j = slice(k);
            R t[E];
#pragma unroll
            for (int e = 0; e < E; ++e) t[e] = conj ? w[k][e] : r[k][e];
            rc_apply<R, L>(t, geo, th);
            if (geo.ok && j < nc) slot_st<R, L>(ex + (long)(j + 1) * SL, geo.ll, t);
            if constexpr (TM)   // w is free here unless it holds the operand
                if (!conj) get_tm(td(k, 0), w[k]);
        }
        __syncthreads();
        AT acc = A::zero();
#pragma unroll
        for (int k = 0; k < K; ++k) {   // M v, and C^T s D M v to the predecessor
            const int j = slice(k);
            const bool on = held(k) && j >= 0;
            R t[E], dd[TM ? E : 1];
#pragma unroll
            for (int e = 0; e < E; ++e) t[e] = R(0);
            if (on) slot_ld<R, L>(ex + (long)j * SL, geo.ll, t);
            if constexpr (TM)
                if (conj) get_tm(td(k, 0), dd);
#pragma unroll
            for (int q = 0; q < RT; ++q) {
                V2 d;
                if constexpr (TM) {
                    d.x = conj ? dd[2 * q] : w[k][2 * q];
                    d.y = conj ? dd[2 * q + 1] : w[k][2 * q + 1];
                } else if constexpr (DREG) {
                    d.x = dreg[k][2 * q];
                    d.y = dreg[k][2 * q + 1];
                } else {
                    d = load_d(k, q);
                }
                w[k][2 * q] = fma(d.x, t[2 * q], conj ? w[k][2 * q] : r[k][2 * q]);
                w[k][2 * q + 1] = fma(d.y, t[2 * q + 1], conj ? w[k][2 * q + 1] : r[k][2 * q + 1]);
                t[2 * q] = d.x * w[k][2 * q];
                t[2 * q + 1] = d.y * w[k][2 * q + 1];
            }
            if (own(k)) {
                R p0 = R(0), p1 = R(0);
#pragma unroll
                for (int e = 0; e < E; e += 2) {
                    p0 = fma(w[k][e], w[k][e], p0);
                    p1 = fma(w[k][e + 1], w[k][e + 1], p1);
                }
                acc = A::addv(acc, p0 + p1);
            }
            rc_apply_t<R, L>(t, geo, th);
            if (on) slot_st<R, L>(ex + (long)j * SL, geo.ll, t);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < K; ++k)
        {
            if (own(k)) {
                const R* s = ex + (long)(slice(k) + 1) * SL;
                R y[E];
                slot_ld<R, L>(s, geo.ll, y);
#pragma unroll
                for (int q = 0; q < RT; ++q) {
                    const bool h = geo.has(q);   // an unused row pair stays zero
                    w[k][2 * q] = h ? w[k][2 * q] + y[2 * q] : R(0);
                    w[k][2 * q + 1] = h ? w[k][2 * q + 1] + y[2 * q + 1] : R(0);
                }
            }
            halo_send(k, w[k], true);
        }
        return acc;
    };
    auto own_dot = [&](const R (&x0)[K][E], const R (&y0)[K][E]) -> AT {
        AT acc = A::zero();
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (own(k)) {
#pragma unroll
                for (int e = 0; e < E; e += 4) {
                    R s4 = x0[k][e] * y0[k][e];
#pragma unroll
                    for (int q = 1; q < 4; ++q) s4 = fma(x0[k][e + q], y0[k][e + q], s4);
                    acc = A::addv(acc, s4);
                }
            }
        return acc;
    };

    // the failure flags of the solve: of several clusters' failures the code that counts
    // is a timeout, then a number that is not finite, then a missed tolerance, whichever
    // comes last (the codes fall in that order)
    static_assert(HOL_ETIMEOUT < HOL_ENUMERIC && HOL_ENUMERIC < HOL_ENOTCONV && HOL_ENOTCONV < 0, "order");
    auto fail = [&](int code, int rhs) {
        if (code != HOL_ENOTCONV) {
            a.d.g[DCG_ERR_RHS] = rhs;   // one failing rhs (any); reported only
            atomicMin(&a.d.g[DCG_ERR], code);
        }
        atomicMin(&a.d.g[DCG_STICKY], code);
    };
    int item = -1;          // right-hand side in hand (uniform over the cluster)
    bool loaded = false;    // its r and p are on chip
    int it = 0;
    for (;;) {
        // ------------------------------------------------ the next segment's item
        if (crank == 0 && wid == 0) {
            // the ready right-hand side with the fewest iterations; an
            // unfinished one in hand (left running) is given back for it
            // (none after a wait ran out: the cluster's exchanges are no longer in step)
            int pick = -1;
            for (int tries = s_lost ? a.n_rhs : 0; tries < a.n_rhs && pick < 0; ++tries) {
                int best = 0x7fffffff, bi = -1;
                for (int k = lane; k < a.n_rhs; k += 32)
                    if (__ldcg(a.d.rstate + k) == RS_READY) {
                        const int c = __ldcg(a.d.it + k);
                        if (c < best) {
                            best = c;
                            bi = k;
                        }
                    }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const int ob = __shfl_xor_sync(kFull, best, o), oi = __shfl_xor_sync(kFull, bi, o);
                    if (oi >= 0 && (bi < 0 || ob < best || (ob == best && oi < bi))) {
                        best = ob;
                        bi = oi;
                    }
                }
                if (bi < 0) break;
                int won = 0;
                if (lane == 0) won = atomicCAS(a.d.rstate + bi, RS_READY, RS_RUNNING) == RS_READY;
                if (__shfl_sync(kFull, won, 0)) pick = bi;
            }
            if (pick < 0 && item >= 0) pick = item;   // nothing else: go on with it
            if (lane < cs) *cl.map_shared_rank(&s_item, lane) = pick;
        }
        cl.sync();
        const int nxt = s_item;
        if (item >= 0 && nxt != item) {
            // hand the unfinished one back: r and p to memory, then ready
            const long base = ((long)item * a.T + t0) * N;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                R p[E];
                get_p(k, p);
                if (own(k)) {
                    const long o = base + (long)slice(k) * N;
#pragma unroll
                    for (int q = 0; q < RT; ++q)
                        if (geo.has(q)) {
                            V2 t;
                            t.x = r[k][2 * q]; t.y = r[k][2 * q + 1];
                            __stcg(reinterpret_cast<V2*>(rsave + o + geo.site(q)), t);
                            t.x = p[2 * q]; t.y = p[2 * q + 1];
                            __stcg(reinterpret_cast<V2*>(psave + o + geo.site(q)), t);
                        }
                }
            }
            __threadfence();
            cl.sync();
            if (crank == 0 && threadIdx.x == 0) {
                a.d.it[item] = it;
                a.d.bnorm[item] = s_bnorm;
                __threadfence();
                atomicExch(a.d.rstate + item, RS_READY);
            }
        }
        if (nxt < 0) break;
        if (nxt != item) loaded = false;
        item = nxt;
        __threadfence();
        const long rbase = (long)item * a.T * N, base = rbase + (long)t0 * N;
        if (!loaded) {
            it = __ldcg(a.d.it + item);
            double bnorm = __ldcg(a.d.bnorm + item);
            if (it == 0) {
                double bb = 0.0;
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (own(k))
#pragma unroll
                        for (int q = 0; q < RT; ++q)
                            if (geo.has(q)) {
                                const double2 t = *reinterpret_cast<const double2*>(
                                    a.b + base + (long)slice(k) * N + geo.site(q));
                                bb = fma(t.x, t.x, bb);
                                bb = fma(t.y, t.y, bb);
                            }
                bnorm = sqrt(reduce64(bb));
                if (bnorm == 0.0 || !isfinite(bnorm)) {   // v = 0 is exact, or nothing is
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (own(k))
#pragma unroll
                            for (int q = 0; q < RT; ++q)
                                if (geo.has(q))
                                    __stcg(reinterpret_cast<double2*>(
                                               a.v + base + (long)slice(k) * N + geo.site(q)),
                                           make_double2(0.0, 0.0));
                    if (crank == 0 && threadIdx.x == 0) {
                        const bool z = bnorm == 0.0;
                        a.d.tres[item] = z ? 0.0 : bnorm;
                        a.d.done[item] = z;
                        a.d.rstate[item] = RS_DONE;
                        if (!z) fail(HOL_ENUMERIC, item);
                    }
                    item = -1;
                    continue;
                }
            }
            const unsigned bxs = exp_hi(bnorm);
            if (threadIdx.x == 0) {
                // a tolerance far below the FP64 rounding of b still folds before the
                // sums leave their range
                const double tb = a.tol * (bnorm * pow2_hi(0u - bxs));
                s_bnorm = bnorm;
                s_limit = fmax(tb * tb, sizeof(R) == 4 ? 1e-34 : 1e-290);
                s_bxs = bxs;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < K; ++k) {
                R p[E];
                const long o = rbase + (held(k) ? (long)tau_of(slice(k)) * N : 0L);
#pragma unroll
                for (int q = 0; q < RT; ++q) {
                    V2 tr, tq;
                    tr.x = tr.y = tq.x = tq.y = R(0);
                    if (held(k) && geo.has(q)) {
                        if (it == 0) {
                            const double2 t = *reinterpret_cast<const double2*>(a.b + o + geo.site(q));
                            tr.x = from_f64<R>(t.x * pow2_hi(0u - bxs));
                            tr.y = from_f64<R>(t.y * pow2_hi(0u - bxs));
                        } else {
                            tr = __ldcg(reinterpret_cast<const V2*>(rsave + o + geo.site(q)));
                            tq = __ldcg(reinterpret_cast<const V2*>(psave + o + geo.site(q)));
                        }
                    }
                    r[k][2 * q] = tr.x; r[k][2 * q + 1] = tr.y;
                    p[2 * q] = tq.x; p[2 * q + 1] = tq.y;
                }
                if constexpr (TM) {
#pragma unroll
                    for (int e = 0; e < E; e += CH) {
                        R u[CH];
#pragma unroll
                        for (int q = 0; q < CH; ++q) u[q] = p[e + q];
                        tm_st<CH>(tp(k, e), u);
                    }
                } else {
                    if (own(k)) slot_st<R, L>(ps + (long)slice(k) * SL, geo.ll, p);
                }
            }
            loaded = true;
        }
        // x = 0; the FP64 solution is not yet defined before the first fold
        const bool fresh = it == 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if constexpr (TM) {
                R z[CH];
#pragma unroll
                for (int q = 0; q < CH; ++q) z[q] = R(0);
#pragma unroll
                for (int e = 0; e < E; e += CH) tm_st<CH>(tx(k, e), z);
            } else {
                R z[E];
#pragma unroll
                for (int e = 0; e < E; ++e) z[e] = R(0);
                if (own(k)) slot_st<R, L>(xs + (long)slice(k) * SL, geo.ll, z);
            }
        }
        // ------------------------------------------------ direction to go on with
        Steps<R> st;
        st.start();
        bool given = false;
        R beta0 = R(0);
        double corr = 0.0;
        if (fresh) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                R z[E];
#pragma unroll
                for (int e = 0; e < E; ++e) z[e] = R(0);
                if (held(k)) slot_st<R, L>(ss + (long)(slice(k) + 1) * SL, geo.ll, z);
            }
        } else {
            // s = A p for the kept p, re-conjugated against the replaced r:
            // beta = -(r, s) / (p, s), so (p, A p) = delta + beta (r, s)
#pragma unroll
            for (int k = 0; k < K; ++k) {
#pragma unroll
                for (int e = 0; e < E; ++e) w[k][e] = R(0);
                get_p(k, w[k]);
                halo_send(k, w[k], false);
            }
            cl.sync();
#pragma unroll
            for (int k = 0; k < K; ++k) halo_recv(k, hpar, w[k], false);
            hpar ^= 1;
            AT pi = apply(true);
            AT rho = own_dot(r, w);
            reduce(pi, rho);
            __syncthreads();
#pragma unroll
            for (int k = 0; k < K; ++k) {
                halo_recv(k, hpar, w[k], true);
                if (held(k)) slot_st<R, L>(ss + (long)(slice(k) + 1) * SL, geo.ll, w[k]);
            }
            hpar ^= 1;
            given = true;
            if (wid == 0) {
                const double bq = cg_ratio(-A::val(rho), A::val(pi));
                beta0 = (R)bq;
                corr = bq * A::val(rho);
            }
        }
        AT gpart = own_dot(r, r);

        // ------------------------------------------------ iterations
        int since = 0;
        bool bad = false;
        bool below = false;   // below tol at the last check (warp 0)
        for (;;) {
            if (it >= a.max_iter || (since >= a.rel_every && since % a.chk == 0)) break;
            AT delta = apply(false);
            AT gamma = gpart;
            reduce(gamma, delta);
            if (wid == 0) {
                // |r| / |b| < tol, as gamma against (tol |b|)^2. The two-kernel iteration has
                // the next check_every iterations in flight when it reads this, so a solution
                // that stops here at once is further from the exact one (1.05 to 1.5 times
                // on average, at L = 32 to 4)
                int stop = lost ? 3 : 0;
                if (!lost && since > 0 && since % a.chk == 0) {
                    stop = A::stop(gamma, s_limit);
                    const bool first = stop == 1 && !below;
                    below = first;
                    if (first) stop = 0;
                }
                R al, be;
                st.step(gamma, delta, given, beta0, corr, al, be);
                if (lane == 0) {
                    s_step[0] = al;
                    s_step[1] = be;
                    s_stop = stop;
                }
            }
            __syncthreads();
            if (s_stop) {
                bad = s_stop >= 2;
                hpar ^= 1;
                break;
            }
            const R alpha = s_step[0], beta = s_step[1];
            given = false;
            if (wid == 0) st.keep(gamma);
            // s = A r + beta s, p = r + beta p, x += alpha p, r -= alpha s
            gpart = A::zero();
            if constexpr (TM) tm_stored();
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int j = slice(k);
                const bool hk = held(k), ok = own(k);
                halo_recv(k, hpar, w[k], true);
                R* sk = ss + (long)(j + 1) * SL;
                R* pk = ps + (long)j * SL;
                R* xk = xs + (long)j * SL;
                AT gk = A::zero();
#pragma unroll
                for (int e = 0; e < E; e += CH) {
                    R p[CH], x[CH], s[CH];
                    if constexpr (TM) {
                        tm_ld2<CH>(tp(k, e), tx(k, e), p, x);
                    } else if (ok) {
                        slot_get<R, L, CH>(pk, geo.ll, e, p);
                        slot_get<R, L, CH>(xk, geo.ll, e, x);
                    }
                    if (hk) {
                        slot_get<R, L, CH>(sk, geo.ll, e, s);
#pragma unroll
                        for (int q = 0; q < CH; ++q) s[q] = fma(beta, s[q], w[k][e + q]);
                        slot_put<R, L, CH>(sk, geo.ll, e, s);
                    } else {
#pragma unroll
                        for (int q = 0; q < CH; ++q) s[q] = R(0);
                    }
#pragma unroll
                    for (int q = 0; q < CH; ++q) {
                        p[q] = fma(beta, p[q], r[k][e + q]);
                        x[q] = fma(alpha, p[q], x[q]);
                        r[k][e + q] = fma(-alpha, s[q], r[k][e + q]);
                    }
                    if constexpr (TM) {
                        tm_st<CH>(tp(k, e), p);
                        tm_st<CH>(tx(k, e), x);
                    } else if (ok) {
                        slot_put<R, L, CH>(pk, geo.ll, e, p);
                        slot_put<R, L, CH>(xk, geo.ll, e, x);
                    }
#pragma unroll
                    for (int q0 = 0; q0 < CH; q0 += 4) {
                        R s4 = r[k][e + q0] * r[k][e + q0];
#pragma unroll
                        for (int q = 1; q < 4; ++q) s4 = fma(r[k][e + q0 + q], r[k][e + q0 + q], s4);
                        gk = A::addv(gk, s4);
                    }
                }
                if (ok) gpart = A::add(gpart, gk);
            }
            hpar ^= 1;
            ++it;
            ++since;
        }

        // ------------------------------------------------ fold and true residual
        // every block has read its exchange slots and s: the FP64 exchange takes
        // their place. v += x, C v to the successor
        if (s_stop == 3) mb_gave_up(sm_addr(s_mb), mbk, sm_addr(&s_lost), cs);
        cl.sync();
        const double down = pow2_hi(0u - s_bxs);
        double* const ex64_next0 = cl.map_shared_rank(ex64, next);
        double* const ex64_prevn = cl.map_shared_rank(ex64, prev) + (long)prev_nc * SL;
        if constexpr (TM) tm_stored();
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = slice(k);
            double t[E];
            double* vo = a.v + base + (long)j * N;
#pragma unroll
            for (int e = 0; e < E; e += CH) {
                R x[CH];
                double2 u[CH / 2];
#pragma unroll
                for (int q = 0; q < CH / 2; ++q) {
                    u[q] = make_double2(0.0, 0.0);
                    if (!fresh && own(k) && geo.has(e / 2 + q))
                        u[q] = __ldcg(reinterpret_cast<const double2*>(vo + geo.site(e / 2 + q)));
                }
                if constexpr (TM) {
                    R x2[CH];
                    tm_ld2<CH>(tx(k, e), tx(k, e), x, x2);
                } else if (own(k)) {
                    slot_get<R, L, CH>(xs + (long)j * SL, geo.ll, e, x);
                }
#pragma unroll
                for (int q = 0; q < CH / 2; ++q) {
                    if (own(k) && geo.has(e / 2 + q)) {
                        u[q].x += to_f64(x[2 * q]);
                        u[q].y += to_f64(x[2 * q + 1]);
                        __stcg(reinterpret_cast<double2*>(vo + geo.site(e / 2 + q)), u[q]);
                    }
                    t[e + 2 * q] = u[q].x;
                    t[e + 2 * q + 1] = u[q].y;
                }
            }
            rc_apply<double, L>(t, geo, a.th);
            if (own(k))
                slot_st<double, L>(j + 1 == nc ? ex64_next0 : ex64 + (long)(j + 1) * SL, geo.ll, t);
        }
        cl.sync();
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = slice(k);
            double t[E];
            if (own(k)) {
                const bool neg = t0 + j != 0;
                const long o = base + (long)j * N;
                slot_ld<double, L>(ex64 + (long)j * SL, geo.ll, t);
                const double* dj = a.ev64 + (long)(t0 + j) * N;
#pragma unroll
                for (int q0 = 0; q0 < RT; q0 += 2) {   // two rows' loads ahead of their stores
                    double2 d[2], u[2], bv[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        d[q] = make_double2(0.0, 0.0);
                        u[q] = d[q];
                        bv[q] = d[q];
                        if (geo.has(q0 + q)) {
                            const int so = geo.site(q0 + q);
                            d[q] = __ldg(reinterpret_cast<const double2*>(dj + so));
                            u[q] = __ldcg(reinterpret_cast<const double2*>(a.v + o + so));
                            bv[q] = __ldg(reinterpret_cast<const double2*>(a.b + o + so));
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const double dx = neg ? -d[q].x : d[q].x, dy = neg ? -d[q].y : d[q].y;
                        double* tq = t + 2 * (q0 + q);
                        const double wx = fma(dx, tq[0], u[q].x), wy = fma(dy, tq[1], u[q].y);
                        if (geo.has(q0 + q))
                            __stcg(reinterpret_cast<double2*>(a.t64 + o + geo.site(q0 + q)),
                                   make_double2(fma(bv[q].x, down, -wx), fma(bv[q].y, down, -wy)));
                        tq[0] = dx * wx;
                        tq[1] = dy * wy;
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) t[e] = 0.0;
            }
            rc_apply_t<double, L>(t, geo, a.th);
            if (own(k)) slot_st<double, L>(j == 0 ? ex64_prevn : ex64 + (long)j * SL, geo.ll, t);
        }
        cl.sync();
        double tr = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (own(k)) {
                const double* to = a.t64 + base + (long)slice(k) * N;
                const double* ys = ex64 + (long)(slice(k) + 1) * SL;
#pragma unroll
                for (int e = 0; e < E; e += 4) {
                    double y[4];
                    slot_get<double, L, 4>(ys, geo.ll, e, y);
#pragma unroll
                    for (int q = 0; q < 4; q += 2)
                        if (geo.has((e + q) / 2)) {
                            const double2 u =
                                __ldcg(reinterpret_cast<const double2*>(to + geo.site((e + q) / 2)));
                            const double rx = u.x - y[q], ry = u.y - y[q + 1];
                            tr = fma(rx, rx, tr);
                            tr = fma(ry, ry, tr);
                            r[k][e + q] = from_f64<R>(rx);
                            r[k][e + q + 1] = from_f64<R>(ry);
                        }
                }
            }
            halo_send(k, r[k], false);
        }
        const double tres = sqrt(reduce64(tr)) / (s_bnorm * pow2_hi(0u - s_bxs));
#pragma unroll
        for (int k = 0; k < K; ++k) halo_recv(k, hpar, r[k], false);
        hpar ^= 1;
        const bool timeout = s_lost != 0;
        bad = bad || timeout || !isfinite(tres);
        if (bad || tres < a.tol || it >= a.max_iter) {
            const unsigned bxs = s_bxs;
            if (bxs != 0)   // v on the scale of b
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (own(k))
#pragma unroll
                        for (int q = 0; q < RT; ++q)
                            if (geo.has(q)) {
                                double2* vq = reinterpret_cast<double2*>(
                                    a.v + base + (long)slice(k) * N + geo.site(q));
                                double2 u = __ldcg(vq);
                                u.x *= pow2_hi(bxs);
                                u.y *= pow2_hi(bxs);
                                __stcg(vq, u);
                            }
            if (crank == 0 && threadIdx.x == 0) {
                const bool ok = !bad && tres < a.tol;
                a.d.it[item] = it;
                a.d.tres[item] = tres;
                a.d.done[item] = ok;
                a.d.rstate[item] = RS_DONE;
                if (!ok) fail(timeout ? HOL_ETIMEOUT : bad ? HOL_ENUMERIC : HOL_ENOTCONV, item);
            }
            item = -1;
        }
    }
    if constexpr (TM) {
        asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
        __syncthreads();
        if (wid == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(s_tm),
                         "r"(tm_cols));
    }
}

// r and the applied direction stay in registers: at most 32 values of each
// per lane in FP32, 16 in FP64
template <typename R, int L, int K>
constexpr bool res_fits = K * RGeo<L>::E <= (sizeof(R) == 4 ? 32 : 16);
template <typename R, int L, int K>   // without tensor memory s D takes registers too
constexpr bool res_plain = res_fits<R, L, K> && K * RGeo<L>::E <= 16;

template <typename R, int L>
ResKernel resident_instance(int K, bool tm)
{
    ResKernel k{RGeo<L>::SL, RGeo<L>::G, RGeo<L>::E, nullptr};
#define HOL_RES_K(KK)                                                               \
    if constexpr (res_fits<R, L, KK>) {                                             \
        if constexpr (res_plain<R, L, KK>)                                          \
            if (K == KK && !tm) k.fn = k_cg_resident<R, L, KK, false>;              \
        if constexpr (sizeof(R) == 4 && KK * RGeo<L>::E >= 16)                      \
            if (K == KK && tm) k.fn = k_cg_resident<R, L, KK, true>;                \
    }
    HOL_RES_K(1)
    HOL_RES_K(2)
    HOL_RES_K(4)
#undef HOL_RES_K
    return k;
}

}  // namespace
}  // namespace hol
