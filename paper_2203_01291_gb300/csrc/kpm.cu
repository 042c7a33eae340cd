// Chebyshev kernels of the adiabatic preconditioner (App. C), one problem being
// the series of one (omega, right-hand side): sum_m c_m T_m(A) u for a complex
// N-vector u, A = 2 (Bbar - bmin) / db - 1 (precond.cu). Bbar is real, so the
// real and imaginary parts run the same real recurrence independently and meet
// only in the complex coefficients: each part accumulates sum c_m.re T_m u and
// sum c_m.im T_m u, and the two exchange the latter once per series.
//
// What bounds both kernels is the chain of dependent Bbar applications of omega
// = 0 (N_P falls like 1 / (omega + 1/2), so its two series are several times
// longer than the next); all other problems fit beside it. Against the older kernels
// (kpm_registers 0..3), P^{-1} P^{-T} at Ltau = 120 for every even L from 4 to 32 on 2 and
// 16 right-hand sides: FP32 as fast at L = 4 and 6 (14 us, launches), else 1.04 to 2.2 times
// as fast as the best of them; FP64 1.1 to 2.6 times. They remain for callers that
// select them.
//   k_kpm_strip (FP32, L <= 18): one warp per part with the slice in the strip
//   layout (strip.cuh), so a step has no barrier: about 150 cycles a step, the
//   latency of its shuffles and dependent multiply-adds. Steps carry the
//   recurrence x = d2 Bbar' t + (2 c0 t - prev), the factor 2 a folded into the
//   diagonal, on packed FP32 pairs; 2 c0 as two floats, since its rounding, the
//   same at every site and step, would be the largest error of a long series
//   (relative error of a series, mean over seven shapes: 6.4e-7, 1.1e-6 with
//   one float or with the older kernels' unfolded constants). P^{-1} P^{-T} at
//   L = 16, Ltau = 160 on 2 rhs 15.2 us (30.4 with the one-column layout
//   k_kpm_lane); 14.2 with the set-up ahead of the wait for the forward transform.
//   k_kpm_rows (FP32, L >= 20): the strip over several warps per part, since one
//   warp's issue slots would bound a step (L = 32: 500 cycles); one exchange of
//   edge rows per step. L = 32, Ltau = 200: 23.2 us on 2 rhs (42.2 with
//   k_kpm_reg), 40.0 on 16 (57.7).
//   k_kpm_pair (FP64): a step is bound by the FP64 pipe (an FP64 instruction
//   holds its quarter of a multiprocessor for sixty cycles), so a problem's two
//   parts take one multiprocessor each (a cluster of two blocks) and a part is
//   cut into row pairs over all four quarters: one or two columns by two rows
//   per lane, the odd y-bonds through shared memory (one block barrier per
//   step). L = 20, Ltau = 120, 2 rhs: 108 us for this kernel (279 in the
//   shared-memory kernel); L = 16, Ltau = 160, 2 rhs: 74 (149 with k_kpm_band).
#include <cooperative_groups.h>

#include <type_traits>

#include "cb.cuh"
#include "fft.cuh"
#include "internal.cuh"
#include "strip.cuh"

namespace hol {
namespace {

namespace cgp = cooperative_groups;

// ---------------------------------------------------------------- FP32 strips
// Block: two warps, one per part; the warp's lane groups hold the same omega of
// consecutive right-hand sides (an idle group repeats the last one).
template <int L>
__global__ void __launch_bounds__(64)
    k_kpm_strip(const float2* __restrict__ vin, float2* __restrict__ vout,
                const float* __restrict__ dk, const int* __restrict__ npv,
                const float4* __restrict__ coef, int n_rhs, int Th,
                int max_np, int mode, float th)
{
    using K = RGeo<L>;
    constexpr int N = L * L, RT = K::RT;
    const K geo;
    const int part = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rpb = (n_rhs + K::G - 1) / K::G;       // blocks per omega, longest series first
    const int wq = blockIdx.x / rpb;
    const int rhs_raw = (blockIdx.x - wq * rpb) * K::G + geo.g;
    const bool own = geo.ok && rhs_raw < n_rhs;
    const int rhs = rhs_raw < n_rhs ? rhs_raw : n_rhs - 1;
    const long off = ((long)rhs * Th + wq) * N;
    extern __shared__ __align__(16) float4 ks_smem[];
    float4* cw = ks_smem;                                            // (re, re, im, im)
    f32p* xb = reinterpret_cast<f32p*>(cw + max_np);                 // [series][part][RT][32]
    const int np = npv[wq];
    for (int m = threadIdx.x; m < np; m += 64) cw[m] = coef[(long)wq * max_np + m];
    const float c2 = dk[N];
    const f32p c02 = pk(c2, c2), c02l = pk(dk[N + 1], dk[N + 1]), th2 = pk(th, th);
    const f32p m1 = pk(-1.0f, -1.0f), half = pk(0.5f, 0.5f);
    f32p t[RT], d[RT];
#pragma unroll
    for (int q = 0; q < RT; ++q) {
        d[q] = 0;
        if (geo.has(q)) {
            const float2 db2 = *reinterpret_cast<const float2*>(dk + geo.site(q));
            d[q] = pk(db2.x, db2.y);
        }
    }
    pdl_wait();      // the input comes from the previous kernel of the stream
    pdl_trigger();   // the next kernel's blocks may take their places (it waits for this one's end)
#pragma unroll
    for (int q = 0; q < RT; ++q) {
        t[q] = 0;
        if (geo.has(q)) {
            const float4 v = *reinterpret_cast<const float4*>(vin + off + geo.site(q));
            t[q] = part ? pk(v.y, v.w) : pk(v.x, v.z);
        }
    }
    __syncthreads();
    // one series; the direction is a compile-time constant
    auto series = [&](auto trans_c, int sidx) {
        constexpr bool trans = decltype(trans_c)::value;
        const float4 c0 = cw[0];
        f32p A[RT], B[RT], nprev[RT];   // minus the one before
        // T_1 u = A u = 2 A (u / 2) - 0: the recurrence from t = u / 2, prev = 0
#pragma unroll
        for (int q = 0; q < RT; ++q) {
            A[q] = mul2(pk(c0.x, c0.y), t[q]);
            B[q] = mul2(pk(c0.z, c0.w), t[q]);
            t[q] = mul2(half, t[q]);
            nprev[q] = 0;
        }
        for (int m = 1; m < np; ++m) {
            const float4 cm = cw[m];
            const f32p cr = pk(cm.x, cm.y), ci = pk(cm.z, cm.w);
            f32p b[RT];
#pragma unroll
            for (int q = 0; q < RT; ++q) b[q] = trans ? mul2(d[q], t[q]) : t[q];
            if constexpr (trans) {
                py_odd<L>(b, geo, th2);
                py_even<L>(b, th2);
                px_odd<L>(b, geo, th2);
                px_even<L>(b, th);
                if constexpr (K::NL < K::H) {
#pragma unroll
                    for (int q = RT - 2; q < RT; ++q) b[q] = geo.shortc ? 0 : b[q];   // unused rows
                }
            } else {
                px_even<L>(b, th);
                px_odd<L>(b, geo, th2);
                py_even<L>(b, th2);
                py_odd<L>(b, geo, th2);
            }
#pragma unroll
            for (int q = 0; q < RT; ++q) {
                const f32p y = fma2(c02, t[q], fma2(c02l, t[q], nprev[q]));
                const f32p x = trans ? add2(b[q], y) : fma2(d[q], b[q], y);
                nprev[q] = mul2(m1, t[q]);
                t[q] = x;
                A[q] = fma2(cr, x, A[q]);
                B[q] = fma2(ci, x, B[q]);
            }
            if (m == 1)
#pragma unroll
                for (int q = 0; q < RT; ++q) nprev[q] = add2(nprev[q], nprev[q]);   // T_0 u = u
        }
        // re = A_re - s B_im, im = A_im + s B_re; s = -1 for the conjugate
        // coefficients of the transpose
        f32p* mine = xb + (long)((sidx * 2 + part) * RT) * 32 + lane;
        const f32p* oth = xb + (long)((sidx * 2 + 1 - part) * RT) * 32 + lane;
#pragma unroll
        for (int q = 0; q < RT; ++q) mine[q * 32] = B[q];
        __syncthreads();
        const float s = (part == 0) == trans ? 1.0f : -1.0f;
#pragma unroll
        for (int q = 0; q < RT; ++q) t[q] = fma2(pk(s, s), oth[q * 32], A[q]);
    };
    if (mode & 1) series(std::true_type{}, 0);
    if (mode & 2) series(std::false_type{}, 1);
    if (own) {
        float* o = reinterpret_cast<float*>(vout + off) + part;
#pragma unroll
        for (int q = 0; q < RT; ++q)
            if (geo.has(q)) {
                float x, y;
                upk(t[q], x, y);
                o[2 * geo.site(q)] = x;
                o[2 * geo.site(q) + 2] = y;
            }
    }
}

template <int L>
int run_strip(const hol_ctx* c, const float2* in, float2* out, int n_rhs, int mode, cudaStream_t s)
{
    using K = RGeo<L>;
    const int Th = c->T / 2, max_np = c->kpm.max_np;
    const size_t sm = (size_t)max_np * sizeof(float4) + (size_t)4 * K::RT * 32 * sizeof(f32p);
    if (int rc = smem_raise((const void*)k_kpm_strip<L>, sm)) return rc;
    const int grid = Th * ((n_rhs + K::G - 1) / K::G);
    HOL_CUDA(launch_pdl(c, k_kpm_strip<L>, grid, 64, sm, s, in, out, c->kpm.dk32, c->kpm.np,
                        c->kpm.coef32, n_rhs, Th, max_np, mode, (float)c->th));
    HOL_CHECK_LAUNCH("k_kpm_strip");
    return HOL_OK;
}

// ---------------------------------------------------------------- FP32 bands
// The strip of L >= 20 over several warps per part: a lane holds two columns of
// RP row pairs, NCH chunks over W warps. The odd y-bonds across chunks go
// through shared memory behind a barrier of the part's own warps; a warp's
// share of a step (E = 4 RP values) is then as short as that exchange.
template <int L>
struct BGeo {
    static constexpr int LP = L / 2;
    static constexpr int RP = (L / 2) % 2 == 0 ? 2 : L == 30 ? 3 : 1;   // divides L / 2
    static constexpr int NCH = (L / 2) / RP;
    static constexpr int HM = 32 / LP;
    static constexpr int W = (NCH + HM - 1) / HM;        // warps per part
    static constexpr int H = (NCH + W - 1) / W;
};

template <int L, bool CL>
__global__ void __launch_bounds__(32 * BGeo<L>::W * (CL ? 1 : 2))
    k_kpm_rows(const float2* __restrict__ vin, float2* __restrict__ vout,
               const float* __restrict__ dk, const int* __restrict__ npv,
               const float4* __restrict__ coef, int n_rhs, int Th,
               int max_np, int mode, float th)
{
    using P = BGeo<L>;
    constexpr int N = L * L, LP = P::LP, RT = 2 * P::RP, NT = 32 * P::W;
    // CL: a cluster of two blocks, one per part; else both parts in one block
    const int rank = CL ? (int)(blockIdx.x & 1) : 0;
    const int part = CL ? rank : (int)(threadIdx.x >= NT);
    const int tid = threadIdx.x - (CL ? 0 : part * NT);
    const int lane = tid & 31, wid = tid >> 5;
    const int h = lane / LP;
    const int ch_raw = wid * P::H + h;
    const bool live = h < P::H && ch_raw < P::NCH;
    const int ch = live ? ch_raw : 0;                    // idle lanes repeat the first chunk
    const int base = h < P::H ? h * LP : 0;
    const int cx = lane % LP;
    const int left = base + (cx == 0 ? LP - 1 : cx - 1);
    const int right = base + (cx + 1 == LP ? 0 : cx + 1);
    const int prob = CL ? blockIdx.x >> 1 : blockIdx.x;  // longest series first
    const int wq = prob / n_rhs, rhs = prob - wq * n_rhs;
    const long off = ((long)rhs * Th + wq) * N;
    const int site0 = ch * RT * L + 2 * cx;
    extern __shared__ __align__(16) float4 kr_smem[];
    float4* cw = kr_smem;                                            // (re, re, im, im)
    // edge rows [part of the block][2][chunk][row][LP], exchange [series][part][RT][NT]
    constexpr int EB = 2 * P::NCH * 2 * LP;
    const int slot = CL ? 0 : part;
    f32p* eb = reinterpret_cast<f32p*>(cw + max_np) + slot * EB;
    f32p* xb = reinterpret_cast<f32p*>(cw + max_np) + (CL ? 1 : 2) * EB;
    const int np = npv[wq];
    for (int m = threadIdx.x; m < np; m += blockDim.x) cw[m] = coef[(long)wq * max_np + m];
    const float c2 = dk[N];
    const f32p c02 = pk(c2, c2), c02l = pk(dk[N + 1], dk[N + 1]), th2 = pk(th, th);
    const f32p m1 = pk(-1.0f, -1.0f), half = pk(0.5f, 0.5f);
    f32p t[RT], d[RT];
#pragma unroll
    for (int q = 0; q < RT; ++q) {
        const float2 db2 = *reinterpret_cast<const float2*>(dk + site0 + q * L);
        d[q] = pk(db2.x, db2.y);
    }
    pdl_wait();      // the input comes from the previous kernel of the stream
    pdl_trigger();   // the next kernel's blocks may take their places (it waits for this one's end)
#pragma unroll
    for (int q = 0; q < RT; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(vin + off + site0 + q * L);
        t[q] = part ? pk(v.y, v.w) : pk(v.x, v.z);
    }
    __syncthreads();
    int par = 0;
    const int dn = ch + 1 == P::NCH ? 0 : ch + 1, up = ch == 0 ? P::NCH - 1 : ch - 1;
    auto y_odd = [&](f32p (&v)[RT]) {
        f32p* e = eb + par * (P::NCH * 2 * LP);
        if (live) {
            e[(ch * 2 + 0) * LP + cx] = v[0];
            e[(ch * 2 + 1) * LP + cx] = v[RT - 1];
        }
        if constexpr (CL)
            __syncthreads();
        else   // this part's warps only
            asm volatile("bar.sync %0, %1;\n" ::"r"(1 + part), "r"(NT) : "memory");
        const f32p vd = e[(dn * 2 + 0) * LP + cx], vu = e[(up * 2 + 1) * LP + cx];
#pragma unroll
        for (int q = 1; q + 1 < RT; q += 2) {
            const f32p a = v[q], b = v[q + 1];
            v[q] = fma2(b, th2, a);
            v[q + 1] = fma2(a, th2, b);
        }
        v[RT - 1] = fma2(vd, th2, v[RT - 1]);
        v[0] = fma2(vu, th2, v[0]);
        par ^= 1;
    };
    auto y_even = [&](f32p (&v)[RT]) {
#pragma unroll
        for (int q = 0; q < RT; q += 2) {
            const f32p a = v[q], b = v[q + 1];
            v[q] = fma2(b, th2, a);
            v[q + 1] = fma2(a, th2, b);
        }
    };
    auto x_even = [&](f32p (&v)[RT]) {
#pragma unroll
        for (int q = 0; q < RT; ++q) {
            float a, b;
            upk(v[q], a, b);
            v[q] = pk(fmaf(th, b, a), fmaf(th, a, b));
        }
    };
    auto x_odd = [&](f32p (&v)[RT]) {
#pragma unroll
        for (int q = 0; q < RT; ++q) {
            float a, b;
            upk(v[q], a, b);
            const float rt = __shfl_sync(kFull, a, right);
            const float lf = __shfl_sync(kFull, b, left);
            v[q] = fma2(pk(lf, rt), th2, v[q]);
        }
    };
    auto series = [&](auto trans_c, int sidx) {
        constexpr bool trans = decltype(trans_c)::value;
        const float4 c0 = cw[0];
        f32p A[RT], B[RT], nprev[RT];   // minus the one before
#pragma unroll
        for (int q = 0; q < RT; ++q) {   // T_1 u = 2 A (u / 2) - 0, as in k_kpm_strip
            A[q] = mul2(pk(c0.x, c0.y), t[q]);
            B[q] = mul2(pk(c0.z, c0.w), t[q]);
            t[q] = mul2(half, t[q]);
            nprev[q] = 0;
        }
        for (int m = 1; m < np; ++m) {
            const float4 cm = cw[m];
            const f32p cr = pk(cm.x, cm.y), ci = pk(cm.z, cm.w);
            f32p b[RT];
#pragma unroll
            for (int q = 0; q < RT; ++q) b[q] = trans ? mul2(d[q], t[q]) : t[q];
            if constexpr (trans) {
                y_odd(b);
                y_even(b);
                x_odd(b);
                x_even(b);
            } else {
                x_even(b);
                x_odd(b);
                y_even(b);
                y_odd(b);
            }
#pragma unroll
            for (int q = 0; q < RT; ++q) {
                const f32p y = fma2(c02, t[q], fma2(c02l, t[q], nprev[q]));
                const f32p x = trans ? add2(b[q], y) : fma2(d[q], b[q], y);
                nprev[q] = mul2(m1, t[q]);
                t[q] = x;
                A[q] = fma2(cr, x, A[q]);
                B[q] = fma2(ci, x, B[q]);
            }
            if (m == 1)
#pragma unroll
                for (int q = 0; q < RT; ++q) nprev[q] = add2(nprev[q], nprev[q]);
        }
        f32p* mine = xb + (long)((CL ? sidx : 2 * sidx + part) * RT) * NT + tid;
        const f32p* oth = mine + (CL ? 0 : (1 - 2 * part) * RT * NT);
#pragma unroll
        for (int q = 0; q < RT; ++q) mine[q * NT] = B[q];
        if constexpr (CL) {
            const cgp::cluster_group cl = cgp::this_cluster();
            cl.sync();
            oth = cl.map_shared_rank(mine, 1 - rank);
        } else {
            __syncthreads();
        }
        const float s = (part == 0) == trans ? 1.0f : -1.0f;
#pragma unroll
        for (int q = 0; q < RT; ++q) t[q] = fma2(pk(s, s), oth[q * NT], A[q]);
    };
    if (mode & 1) series(std::true_type{}, 0);
    if (mode & 2) series(std::false_type{}, 1);
    if (live) {
        float* o = reinterpret_cast<float*>(vout + off) + part;
#pragma unroll
        for (int q = 0; q < RT; ++q) {
            float x, y;
            upk(t[q], x, y);
            o[2 * (site0 + q * L)] = x;
            o[2 * (site0 + q * L) + 2] = y;
        }
    }
    if constexpr (CL) cgp::this_cluster().sync();   // the other part has read this block's exchange
}

// Launch of two-block clusters (one block per part), with programmatic
// dependent launch when the context enables it.
template <typename... KArgs, typename... Args>
cudaError_t launch_pair(const hol_ctx* c, void (*kernel)(KArgs...), int problems, int threads,
                        size_t smem, cudaStream_t s, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * problems);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = c->pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <int L>
int run_rows(const hol_ctx* c, const float2* in, float2* out, int n_rhs, int mode, cudaStream_t s)
{
    using P = BGeo<L>;
    const int Th = c->T / 2, max_np = c->kpm.max_np;
    // one multiprocessor per part while every warp of the launch is resident at
    // once (L = 32, Ltau = 200: 16.5 against 21.7 us on 2 rhs); beyond that the
    // blocks queue and half as many of them do better (38.4 against 30.0 us on
    // 16 rhs)
    const bool cl = 2L * P::W * Th * n_rhs <= 64L * c->sms;
    const size_t sm = (size_t)max_np * sizeof(float4) +
                      (size_t)(cl ? 1 : 2) * (2 * P::NCH * 2 * P::LP + 4 * P::RP * 32 * P::W) *
                          sizeof(f32p);
    if (int rc = smem_raise((const void*)(cl ? k_kpm_rows<L, true> : k_kpm_rows<L, false>), sm))
        return rc;
    if (cl)
        HOL_CUDA(launch_pair(c, k_kpm_rows<L, true>, Th * n_rhs, 32 * P::W, sm, s, in, out,
                             c->kpm.dk32, c->kpm.np, c->kpm.coef32, n_rhs, Th, max_np, mode, (float)c->th));
    else
        HOL_CUDA(launch_pdl(c, k_kpm_rows<L, false>, Th * n_rhs, 64 * P::W, sm, s, in, out,
                            c->kpm.dk32, c->kpm.np, c->kpm.coef32, n_rhs, Th, max_np, mode, (float)c->th));
    HOL_CHECK_LAUNCH("k_kpm_rows");
    return HOL_OK;
}

// ---------------------------------------------------------------- FP64 pairs
// A part in row pairs: chunk q holds rows 2 q, 2 q + 1; a lane COLS of their
// columns. COLS = 1 up to L = 16, where it spreads a part over four warps.
template <int L>
struct PGeo {
    static constexpr int COLS = L <= 16 ? 1 : 2;
    static constexpr int LP = L / COLS;                  // lanes per row pair
    static constexpr int NCH = L / 2;
    static constexpr int HM = 32 / LP;                   // most row pairs per warp
    static constexpr int W = (NCH + HM - 1) / HM;        // warps per part
    static constexpr int H = (NCH + W - 1) / W;          // row pairs per warp, evened out
};

template <int L>
__global__ void __launch_bounds__(32 * PGeo<L>::W)
    k_kpm_pair(const double2* __restrict__ vin, double2* __restrict__ vout,
               const double* __restrict__ dk, const int* __restrict__ npv,
               const double2* __restrict__ coef, int n_rhs, int Th,
               int max_np, int mode, double th)
{
    using P = PGeo<L>;
    constexpr int N = L * L, C = P::COLS, LP = P::LP;
    const cgp::cluster_group cl = cgp::this_cluster();
    const int part = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int h = lane / LP, cx = lane - h * LP;
    const int ch_raw = wid * P::H + h;
    const bool live = h < P::H && ch_raw < P::NCH;
    const int ch = live ? ch_raw : 0;                    // idle lanes repeat the first chunk
    const int base = h < P::H ? h * LP : 0;              // (their shuffles stay inside the warp)
    const int cxs = h < P::H ? cx : cx % LP;
    // colour 1 pairs columns (even, odd), colour 2 (odd, even): the partners
    const int p1 = base + (cxs ^ 1);                                            // C = 1
    const int p2 = base + ((cxs & 1) ? (cxs + 1 == LP ? 0 : cxs + 1) : (cxs == 0 ? LP - 1 : cxs - 1));
    const int left = base + (cxs == 0 ? LP - 1 : cxs - 1);                      // C = 2
    const int right = base + (cxs + 1 == LP ? 0 : cxs + 1);
    const int prob = blockIdx.x >> 1;                    // omega slowest, longest series first
    const int wq = prob / n_rhs, rhs = prob - wq * n_rhs;
    const long off = ((long)rhs * Th + wq) * N;
    const int site0 = 2 * ch * L + C * cxs;
    extern __shared__ __align__(16) unsigned char kp_smem[];
    double2* cw = reinterpret_cast<double2*>(kp_smem);
    double* eb = reinterpret_cast<double*>(cw + max_np);            // [2][chunk][row][L]
    double* xb = eb + 2 * P::NCH * 2 * L;                           // [series][2 C][threads]
    const int np = npv[wq];
    for (int m = threadIdx.x; m < np; m += blockDim.x) cw[m] = coef[(long)wq * max_np + m];
    const double c02 = dk[N];
    const double* vf = reinterpret_cast<const double*>(vin);
    double t[2][C], d[2][C];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k = 0; k < C; ++k) d[r][k] = dk[site0 + r * L + k];
    pdl_wait();      // the input comes from the previous kernel of the stream
    const PdlTriggerAtExit pdl_at_exit;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k = 0; k < C; ++k) t[r][k] = vf[2 * (off + site0 + r * L + k) + part];
    __syncthreads();
    int par = 0;
    // odd y-bonds: this chunk's rows with its neighbours' (through shared memory)
    auto y_odd = [&](double (&v)[2][C]) {
        double* e = eb + (long)par * P::NCH * 2 * L;
        if (live)
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < C; ++k) e[(ch * 2 + r) * L + C * cxs + k] = v[r][k];
        __syncthreads();
        const int dn = ch + 1 == P::NCH ? 0 : ch + 1, up = ch == 0 ? P::NCH - 1 : ch - 1;
#pragma unroll
        for (int k = 0; k < C; ++k) {
            v[1][k] = fma(th, e[(dn * 2 + 0) * L + C * cxs + k], v[1][k]);
            v[0][k] = fma(th, e[(up * 2 + 1) * L + C * cxs + k], v[0][k]);
        }
        par ^= 1;
    };
    auto y_even = [&](double (&v)[2][C]) {
#pragma unroll
        for (int k = 0; k < C; ++k) {
            const double x = v[0][k], y = v[1][k];
            v[0][k] = fma(th, y, x);
            v[1][k] = fma(th, x, y);
        }
    };
    auto x_even = [&](double (&v)[2][C]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if constexpr (C == 1) {
                v[r][0] = fma(th, __shfl_sync(kFull, v[r][0], p1), v[r][0]);
            } else {
                const double x = v[r][0], y = v[r][C - 1];
                v[r][0] = fma(th, y, x);
                v[r][C - 1] = fma(th, x, y);
            }
        }
    };
    auto x_odd = [&](double (&v)[2][C]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if constexpr (C == 1) {
                v[r][0] = fma(th, __shfl_sync(kFull, v[r][0], p2), v[r][0]);
            } else {
                const double rt = __shfl_sync(kFull, v[r][0], right);
                const double lf = __shfl_sync(kFull, v[r][C - 1], left);
                v[r][0] = fma(th, lf, v[r][0]);
                v[r][C - 1] = fma(th, rt, v[r][C - 1]);
            }
        }
    };
    auto series = [&](auto trans_c, int sidx) {
        constexpr bool trans = decltype(trans_c)::value;
        const double2 c0 = cw[0];
        double A[2][C], B[2][C], prev[2][C];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < C; ++k) {
                A[r][k] = c0.x * t[r][k];
                B[r][k] = c0.y * t[r][k];
                t[r][k] *= 0.5;          // T_1 u = 2 A (u / 2) - 0
                prev[r][k] = 0.0;
            }
        for (int m = 1; m < np; ++m) {
            const double2 cm = cw[m];
            double b[2][C];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < C; ++k) b[r][k] = trans ? d[r][k] * t[r][k] : t[r][k];
            if constexpr (trans) {
                y_odd(b);
                y_even(b);
                x_odd(b);
                x_even(b);
            } else {
                x_even(b);
                x_odd(b);
                y_even(b);
                y_odd(b);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < C; ++k) {
                    const double y = fma(c02, t[r][k], -prev[r][k]);
                    const double x = trans ? b[r][k] + y : fma(d[r][k], b[r][k], y);
                    prev[r][k] = t[r][k];
                    t[r][k] = x;
                    A[r][k] = fma(cm.x, x, A[r][k]);
                    B[r][k] = fma(cm.y, x, B[r][k]);
                }
            if (m == 1)
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int k = 0; k < C; ++k) prev[r][k] += prev[r][k];   // T_0 u = u
        }
        // re = A_re - s B_im, im = A_im + s B_re (s = -1 for the transpose)
        double* mine = xb + (long)sidx * 2 * C * blockDim.x;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < C; ++k) mine[(r * C + k) * blockDim.x + threadIdx.x] = B[r][k];
        cl.sync();
        const double* oth = cl.map_shared_rank(mine, 1 - part);
        const bool neg = (part == 0) != trans;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < C; ++k) {
                const double o = oth[(r * C + k) * blockDim.x + threadIdx.x];
                t[r][k] = neg ? A[r][k] - o : A[r][k] + o;
            }
    };
    if (mode & 1) series(std::true_type{}, 0);
    if (mode & 2) series(std::false_type{}, 1);
    if (live) {
        double* o = reinterpret_cast<double*>(vout);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < C; ++k) o[2 * (off + site0 + r * L + k) + part] = t[r][k];
    }
    cl.sync();   // the other part has read this block's exchange
}

template <int L>
int run_pair(const hol_ctx* c, const double2* in, double2* out, int n_rhs, int mode, cudaStream_t s)
{
    using P = PGeo<L>;
    const int Th = c->T / 2, max_np = c->kpm.max_np;
    const size_t sm = (size_t)max_np * sizeof(double2) +
                      (size_t)(2 * P::NCH * 2 * L + 2 * 2 * P::COLS * 32 * P::W) * sizeof(double);
    if (int rc = smem_raise((const void*)k_kpm_pair<L>, sm)) return rc;
    HOL_CUDA(launch_pair(c, k_kpm_pair<L>, Th * n_rhs, 32 * P::W, sm, s, in, out, c->kpm.dk64,
                         c->kpm.np, c->kpm.coef, n_rhs, Th, max_np, mode, c->th));
    HOL_CHECK_LAUNCH("k_kpm_pair");
    return HOL_OK;
}

}  // namespace

int kpm_strip(const hol_ctx* c, const float2* in, float2* out, int n_rhs, int mode, cudaStream_t s)
{
    switch (c->L) {
#define X(LL) case LL: return run_strip<LL>(c, in, out, n_rhs, mode, s);
        X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18)
#undef X
#define X(LL) case LL: return run_rows<LL>(c, in, out, n_rhs, mode, s);
        X(20) X(22) X(24) X(26) X(28) X(30) X(32)
#undef X
    }
    return set_error(HOL_EINVAL, "kpm strips: unsupported L=%d", c->L);
}

int kpm_pair(const hol_ctx* c, const double2* in, double2* out, int n_rhs, int mode, cudaStream_t s)
{
    switch (c->L) {
#define X(LL) case LL: return run_pair<LL>(c, in, out, n_rhs, mode, s);
        X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18) X(20) X(22) X(24) X(26) X(28) X(30) X(32)
#undef X
    }
    return set_error(HOL_EINVAL, "kpm pairs: unsupported L=%d", c->L);
}

}  // namespace hol
