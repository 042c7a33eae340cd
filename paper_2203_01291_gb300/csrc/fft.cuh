// Shared-memory mixed-radix FFT along tau (Stockham passes of radix 8, 4, 2, 3,
// 5, 7) over tiles of TS columns, plus complex helpers. Used by the
// preconditioner (twisted transforms), the Fourier-accelerated leapfrog (mass
// matrix along tau) and the measurements.
#pragma once

#include <cuda_runtime.h>

namespace hol {
namespace fft {

// ---------------------------------------------------------------- complex
template <typename R>
struct Cx;
template <>
struct Cx<float> {
    using T2 = float2;
    static __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
};
template <>
struct Cx<double> {
    using T2 = double2;
    static __device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
};
template <typename C>
__device__ __forceinline__ C cmul(C a, C b)
{
    C r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
template <typename C>
__device__ __forceinline__ C cadd(C a, C b)
{
    a.x += b.x;
    a.y += b.y;
    return a;
}

struct RadixPlan {
    int n;
    int r[16];
};

// Radix plan of a length: factors 4 first, then 2, 3, 5, 7; n = -1 if another
// prime factor remains. fp32: an odd power of two from 8 on takes one radix 8
// pass in place of a 4 and a 2 (a pass costs a barrier and a trip through shared
// memory, some 200 cycles). FP64 passes are bound by the FP64 pipe and spread over
// more warps with the smaller radices.
__host__ __device__ constexpr RadixPlan plan_of(int T, bool fp32 = false)
{
    RadixPlan p{0, {}};
    int t = T, e2 = 0;
    for (int u = T; u % 2 == 0; u /= 2) ++e2;
    if (fp32 && e2 >= 3 && e2 % 2 == 1) {
        p.r[p.n++] = 8;
        t /= 8;
    }
    const int rs[5] = {4, 2, 3, 5, 7};
    for (int k = 0; k < 5; ++k)
        while (t % rs[k] == 0 && p.n < 16) {
            p.r[p.n++] = rs[k];
            t /= rs[k];
        }
    if (t != 1) p.n = -1;
    return p;
}

// twiddle w2[k] = exp(-i pi k / T), 0 <= k < 2T (every caller's index is in
// range: 2 r k T / (Ns RAD) < 2T and 2 e T / RAD < 2T)
template <typename R>
__device__ __forceinline__ typename Cx<R>::T2 tw(const typename Cx<R>::T2* __restrict__ w2, long k,
                                                 int T)
{
    (void)T;
    return w2[k];
}

template <typename C>
__device__ __forceinline__ C csub(C a, C b)
{
    a.x -= b.x;
    a.y -= b.y;
    return a;
}
// multiply by -i
template <typename C>
__device__ __forceinline__ C cmi(C a)
{
    C r;
    r.x = a.y;
    r.y = -a.x;
    return r;
}

// Length-RAD DFT of a[] in place (root[e] = exp(-2 pi i e / RAD)). Odd lengths
// pair the inputs r and RAD - r: with s = a_r + a_{RAD-r}, d = a_r - a_{RAD-r}
// the outputs q and RAD - q are (a_0 + sum cos s) -/+ i (sum sin d), a third of
// the products of the plain sums (radix 5: 36 operations instead of 120).
template <typename R, int RAD>
__device__ __forceinline__ void dft_small(typename Cx<R>::T2 (&a)[RAD],
                                          const typename Cx<R>::T2 (&root)[RAD])
{
    using C2 = typename Cx<R>::T2;
    if constexpr (RAD == 2) {
        const C2 x = a[0], y = a[1];
        a[0] = cadd(x, y);
        a[1] = csub(x, y);
    } else if constexpr (RAD == 4) {
        const C2 s02 = cadd(a[0], a[2]), d02 = csub(a[0], a[2]);
        const C2 s13 = cadd(a[1], a[3]), d13 = cmi(csub(a[1], a[3]));
        a[0] = cadd(s02, s13);
        a[1] = cadd(d02, d13);
        a[2] = csub(s02, s13);
        a[3] = csub(d02, d13);
    } else if constexpr (RAD == 8) {   // two of length 4, the odd one turned by root^q
        C2 e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
        const C2 r4[4] = {root[0], root[2], root[4], root[6]};
        dft_small<R, 4>(e, r4);
        dft_small<R, 4>(o, r4);
        o[1] = cmul(o[1], root[1]);
        o[2] = cmi(o[2]);
        o[3] = cmul(o[3], root[3]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            a[q] = cadd(e[q], o[q]);
            a[q + 4] = csub(e[q], o[q]);
        }
    } else {
        constexpr int HF = (RAD - 1) / 2;
        C2 s[HF], d[HF];
#pragma unroll
        for (int r = 1; r <= HF; ++r) {
            s[r - 1] = cadd(a[r], a[RAD - r]);
            d[r - 1] = csub(a[r], a[RAD - r]);
        }
        const C2 a0 = a[0];
#pragma unroll
        for (int r = 0; r < HF; ++r) a[0] = cadd(a[0], s[r]);
#pragma unroll
        for (int q = 1; q <= HF; ++q) {
            C2 re = a0, im;
#pragma unroll
            for (int r = 1; r <= HF; ++r) {
                const C2 w = root[(r * q) % RAD];   // (cos, -sin)
                re.x = fma(w.x, s[r - 1].x, re.x);
                re.y = fma(w.x, s[r - 1].y, re.y);
                if (r == 1) {
                    im.x = w.y * d[0].x;
                    im.y = w.y * d[0].y;
                } else {
                    im.x = fma(w.y, d[r - 1].x, im.x);
                    im.y = fma(w.y, d[r - 1].y, im.y);
                }
            }
            // re + i im with im = -(sum sin d)
            a[q].x = re.x - im.y;
            a[q].y = re.y + im.x;
            a[RAD - q].x = re.x + im.y;
            a[RAD - q].y = re.y - im.x;
        }
    }
}

// One Stockham pass of radix RAD over TS columns: in[tau][c] -> out[.][c].
// Butterfly j (0 <= j < T/RAD) with k = j mod Ns reads in[j + r T/RAD],
// scales input r by exp(-2 pi i r k / (Ns RAD)), takes the length-RAD DFT
// and writes out[(j / Ns) Ns RAD + k + q Ns]. blockDim.x must be a multiple
// of TS; (k, j / Ns) are advanced incrementally instead of divided. TSC > 0: TS
// at compile time.
template <typename R, int RAD, int TSC>
__device__ __forceinline__ void stockham_pass(const typename Cx<R>::T2* __restrict__ in,
                                              typename Cx<R>::T2* __restrict__ out,
                                              const typename Cx<R>::T2* __restrict__ w2, int T, int TS_,
                                              int Ns)
{
    using C2 = typename Cx<R>::T2;
    const int TS = TSC > 0 ? TSC : TS_;
    const int nb = T / RAD;
    const int c = threadIdx.x % TS;
    const int sj = blockDim.x / TS;         // step of j per iteration
    int j = threadIdx.x / TS;
    int k = j % Ns, jb = j / Ns;
    const int sk = sj % Ns, sjb = sj / Ns;
    const int tstep = T / (Ns * RAD);       // twiddle index step per unit of k, halved
    C2 root[RAD];                           // exp(-2 pi i e / RAD)
#pragma unroll
    for (int e = 0; e < RAD; ++e) root[e] = w2[2 * e * (T / RAD)];
    for (; j < nb; j += sj) {
        C2 a[RAD];
        a[0] = in[j * TS + c];
        // twiddles from the table: powers of one cost two products each more
#pragma unroll
        for (int r = 1; r < RAD; ++r) {
            const C2 v = in[(j + r * nb) * TS + c];
            a[r] = k > 0 ? cmul(v, w2[2 * r * k * tstep]) : v;
        }
        dft_small<R, RAD>(a, root);
        const int ob = jb * Ns * RAD + k;
#pragma unroll
        for (int q = 0; q < RAD; ++q) out[(ob + q * Ns) * TS + c] = a[q];
        k += sk;
        jb += sjb;
        if (k >= Ns) {
            k -= Ns;
            jb += 1;
        }
    }
}

// Full forward DFT of length T along the first index of buf (TS columns);
// returns the buffer holding the result.
template <typename R, int TSC = 0>
__device__ typename Cx<R>::T2* fft_tau(typename Cx<R>::T2* a, typename Cx<R>::T2* b,
                                       const typename Cx<R>::T2* __restrict__ w2, int T, int TS,
                                       const RadixPlan& plan)
{
    int Ns = 1;
    for (int s = 0; s < plan.n; ++s) {
        __syncthreads();
        switch (plan.r[s]) {
        case 2: stockham_pass<R, 2, TSC>(a, b, w2, T, TS, Ns); break;
        case 3: stockham_pass<R, 3, TSC>(a, b, w2, T, TS, Ns); break;
        case 4: stockham_pass<R, 4, TSC>(a, b, w2, T, TS, Ns); break;
        case 5: stockham_pass<R, 5, TSC>(a, b, w2, T, TS, Ns); break;
        case 8:
            if constexpr (sizeof(R) == 4) stockham_pass<R, 8, TSC>(a, b, w2, T, TS, Ns);
            break;
        default: stockham_pass<R, 7, TSC>(a, b, w2, T, TS, Ns); break;
        }
        Ns *= plan.r[s];
        typename Cx<R>::T2* t = a;
        a = b;
        b = t;
    }
    __syncthreads();
    return a;
}


// ---------------------------------------------------------------------------
// The same transform with the length T, the tile width TS and the block size
// NT known at compile time (the lengths of the configured workloads): the
// plan, the butterfly loops and every index division are resolved by the
// compiler. The passes and twiddles are fft_tau's.
// ---------------------------------------------------------------------------
template <typename R, int RAD, int T, int TS, int NT, int Ns>
__device__ __forceinline__ void stockham_pass_ct(const typename Cx<R>::T2* __restrict__ in,
                                                 typename Cx<R>::T2* __restrict__ out,
                                                 const typename Cx<R>::T2* __restrict__ w2)
{
    using C2 = typename Cx<R>::T2;
    static_assert(NT % TS == 0, "block size must be a multiple of the tile width");
    constexpr int nb = T / RAD;
    constexpr int SJ = NT / TS;
    constexpr int tstep = T / (Ns * RAD);
    const int c = threadIdx.x % TS;
    const int j0 = threadIdx.x / TS;
    C2 root[RAD];
#pragma unroll
    for (int e = 0; e < RAD; ++e) root[e] = w2[2 * e * (T / RAD)];
#pragma unroll
    for (int jj = 0; jj < (nb + SJ - 1) / SJ; ++jj) {
        const int j = j0 + jj * SJ;
        if (nb % SJ != 0 && j >= nb) break;
        const int k = j % Ns, jb = j / Ns;
        C2 a[RAD];
        a[0] = in[j * TS + c];
#pragma unroll
        for (int r = 1; r < RAD; ++r) {
            const C2 v = in[(j + r * nb) * TS + c];
            a[r] = (Ns > 1 && k > 0) ? cmul(v, w2[2 * r * k * tstep]) : v;
        }
        dft_small<R, RAD>(a, root);
        const int ob = jb * Ns * RAD + k;
#pragma unroll
        for (int q = 0; q < RAD; ++q) out[(ob + q * Ns) * TS + c] = a[q];
    }
}

template <typename R, int T, int TS, int NT, int S = 0, int Ns = 1>
__device__ __forceinline__ typename Cx<R>::T2* fft_tau_ct(typename Cx<R>::T2* a,
                                                          typename Cx<R>::T2* b,
                                                          const typename Cx<R>::T2* __restrict__ w2)
{
    constexpr RadixPlan P = plan_of(T, sizeof(R) == 4);
    static_assert(P.n > 0, "length with a prime factor above 7");
    if constexpr (S < P.n) {
        constexpr int RAD = P.r[S];
        __syncthreads();
        stockham_pass_ct<R, RAD, T, TS, NT, Ns>(a, b, w2);
        return fft_tau_ct<R, T, TS, NT, S + 1, Ns * RAD>(b, a, w2);
    } else {
        __syncthreads();
        return a;
    }
}

}  // namespace fft
}  // namespace hol
