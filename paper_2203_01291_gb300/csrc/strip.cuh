// Strip layout of one L x L slice (any even L <= 32): every lane holds two
// adjacent columns of a chunk of rows. Against the one-column layout (cb.cuh) an
// even x-bond is a register pair and an odd one costs a shuffle per value
// instead of two, and the column pair of a row is one operand of the packed
// FP32 pair instructions.
#pragma once

#include "cb.cuh"

namespace hol {
namespace {

// Lane geometry of side L: LP = L / 2 lanes cover a row (two columns each), H
// chunks of RT or RT - 2 rows (the first NL are long; an unused row pair of a
// short chunk stays zero), G slices per warp. Every chunk starts on an even
// row, so the even y-bonds are register pairs.
template <int L>
struct RGeo {
    static constexpr int LP = L / 2;
    static constexpr int H = (L == 4 || L == 12 || L >= 22) ? 2
                           : (L == 6 || L == 10 || L == 18 || L == 20) ? 3 : 4;
    static constexpr int RT = ((L / 2 + H - 1) / H) * 2;
    static constexpr int NL = (L - H * (RT - 2)) / 2;     // long chunks
    static constexpr int E = 2 * RT;                      // values per lane
    static constexpr int LS = LP * H;                     // lanes per slice
    static constexpr int G = 32 / LS;
    static constexpr int SL = LS * E;                     // stored values per slice
    static_assert(LS <= 32 && NL >= 1 && NL <= H, "lane geometry");
    int g, ll, cx, h, left, right, up, down, row0;
    bool ok, shortc;
    __device__ __forceinline__ RGeo()
    {
        const int lane = threadIdx.x & 31;
        g = lane / LS;
        ok = g < G;
        if (!ok) g = 0;
        ll = ok ? lane - g * LS : (lane - G * LS) % LS;
        cx = ll % LP;
        h = ll / LP;
        const int base = g * LS;
        left = base + h * LP + (cx == 0 ? LP - 1 : cx - 1);
        right = base + h * LP + (cx + 1 == LP ? 0 : cx + 1);
        up = base + (h == 0 ? H - 1 : h - 1) * LP + cx;
        down = base + (h + 1 == H ? 0 : h + 1) * LP + cx;
        shortc = h >= NL;
        row0 = h * RT - (h > NL ? 2 * (h - NL) : 0);
    }
    __device__ __forceinline__ bool has(int rr) const { return NL == H || rr < RT - 2 || !shortc; }
    // site offset of the lane's row rr, first column
    __device__ __forceinline__ int site(int rr) const { return (row0 + rr) * L + 2 * cx; }
};

template <typename R>
struct Vec2;
template <>
struct Vec2<float> {
    using T = float2;
};
template <>
struct Vec2<double> {
    using T = double2;
};

// the four bond colours on a lane's strip (see cb.cuh for the factors)
template <typename R, int L>
__device__ __forceinline__ void rx_even(R (&v)[RGeo<L>::E], R th)
{
#pragma unroll
    for (int e = 0; e < RGeo<L>::E; e += 2) {
        const R a = v[e], b = v[e + 1];
        v[e] = fma(th, b, a);
        v[e + 1] = fma(th, a, b);
    }
}
template <typename R, int L>
__device__ __forceinline__ void rx_odd(R (&v)[RGeo<L>::E], const RGeo<L>& g, R th)
{
#pragma unroll
    for (int e = 0; e < RGeo<L>::E; e += 2) {
        const R rt = __shfl_sync(kFull, v[e], g.right);
        const R lf = __shfl_sync(kFull, v[e + 1], g.left);
        v[e] = fma(th, lf, v[e]);
        v[e + 1] = fma(th, rt, v[e + 1]);
    }
}
template <typename R, int L>
__device__ __forceinline__ void ry_even(R (&v)[RGeo<L>::E], R th)
{
#pragma unroll
    for (int e = 0; e < RGeo<L>::E; e += 4)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const R a = v[e + q], b = v[e + 2 + q];
            v[e + q] = fma(th, b, a);
            v[e + 2 + q] = fma(th, a, b);
        }
}
template <typename R, int L>
__device__ __forceinline__ void ry_odd(R (&v)[RGeo<L>::E], const RGeo<L>& g, R th)
{
    using K = RGeo<L>;
    constexpr int E = K::E;
    R dn[2], upv[2], last[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if constexpr (K::NL < K::H)
            last[q] = g.shortc ? v[E - 6 + q] : v[E - 2 + q];
        else
            last[q] = v[E - 2 + q];
        dn[q] = K::H == 1 ? v[q] : __shfl_sync(kFull, v[q], g.down);
        upv[q] = K::H == 1 ? last[q] : __shfl_sync(kFull, last[q], g.up);
    }
#pragma unroll
    for (int e = 2; e + 2 < E; e += 4)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const R a = v[e + q], b = v[e + 2 + q];
            v[e + q] = fma(th, b, a);
            v[e + 2 + q] = fma(th, a, b);
        }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        v[q] = fma(th, upv[q], v[q]);
        if constexpr (K::NL < K::H) {
            // the short chunk's last row (its pair above met a zero row)
            if (g.shortc)
                v[E - 6 + q] = fma(th, dn[q], v[E - 6 + q]);
            else
                v[E - 2 + q] = fma(th, dn[q], v[E - 2 + q]);
        } else {
            v[E - 2 + q] = fma(th, dn[q], v[E - 2 + q]);
        }
    }
}
template <typename R, int L>
__device__ __forceinline__ void rc_apply(R (&v)[RGeo<L>::E], const RGeo<L>& g, R th)
{
    rx_even<R, L>(v, th);
    rx_odd<R, L>(v, g, th);
    ry_even<R, L>(v, th);
    ry_odd<R, L>(v, g, th);
}
template <typename R, int L>
__device__ __forceinline__ void rc_apply_t(R (&v)[RGeo<L>::E], const RGeo<L>& g, R th)
{
    ry_odd<R, L>(v, g, th);
    ry_even<R, L>(v, th);
    rx_odd<R, L>(v, g, th);
    rx_even<R, L>(v, th);
}

// ---------------------------------------------------------------- FP32 pairs
// The two columns of a row as one 64-bit operand: one issue slot per pair.
typedef unsigned long long f32p;
__device__ __forceinline__ f32p pk(float a, float b)
{
    f32p r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f32p v, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32p fma2(f32p a, f32p b, f32p c)
{
    f32p r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32p mul2(f32p a, f32p b)
{
    f32p r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32p add2(f32p a, f32p b)
{
    f32p r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// the bond colours on a strip of pairs (th2 = (th, th))
template <int L>
__device__ __forceinline__ void px_even(f32p (&v)[RGeo<L>::RT], float th)
{
#pragma unroll
    for (int q = 0; q < RGeo<L>::RT; ++q) {
        float a, b;
        upk(v[q], a, b);
        v[q] = pk(fmaf(th, b, a), fmaf(th, a, b));
    }
}
template <int L>
__device__ __forceinline__ void px_odd(f32p (&v)[RGeo<L>::RT], const RGeo<L>& g, f32p th2)
{
#pragma unroll
    for (int q = 0; q < RGeo<L>::RT; ++q) {
        float a, b;
        upk(v[q], a, b);
        const float rt = __shfl_sync(kFull, a, g.right);
        const float lf = __shfl_sync(kFull, b, g.left);
        v[q] = fma2(pk(lf, rt), th2, v[q]);
    }
}
template <int L>
__device__ __forceinline__ void py_even(f32p (&v)[RGeo<L>::RT], f32p th2)
{
#pragma unroll
    for (int q = 0; q < RGeo<L>::RT; q += 2) {
        const f32p a = v[q], b = v[q + 1];
        v[q] = fma2(b, th2, a);
        v[q + 1] = fma2(a, th2, b);
    }
}
template <int L>
__device__ __forceinline__ void py_odd(f32p (&v)[RGeo<L>::RT], const RGeo<L>& g, f32p th2)
{
    using K = RGeo<L>;
    constexpr int RT = K::RT;
    f32p last = v[RT - 1];
    if constexpr (K::NL < K::H) last = g.shortc ? v[RT >= 3 ? RT - 3 : 0] : last;
    float a0, a1, b0, b1;
    upk(v[0], a0, a1);
    upk(last, b0, b1);
    const f32p dn = pk(__shfl_sync(kFull, a0, g.down), __shfl_sync(kFull, a1, g.down));
    const f32p up = pk(__shfl_sync(kFull, b0, g.up), __shfl_sync(kFull, b1, g.up));
#pragma unroll
    for (int q = 1; q + 1 < RT; q += 2) {
        const f32p a = v[q], b = v[q + 1];
        v[q] = fma2(b, th2, a);
        v[q + 1] = fma2(a, th2, b);
    }
    v[0] = fma2(up, th2, v[0]);
    if constexpr (K::NL < K::H) {   // a short chunk's last row met a zero row above
        const f32p t = fma2(dn, th2, g.shortc ? v[RT >= 3 ? RT - 3 : 0] : v[RT - 1]);
        v[RT - 1] = g.shortc ? v[RT - 1] : t;
        if constexpr (RT >= 3) v[RT - 3] = g.shortc ? t : v[RT - 3];
    } else {
        v[RT - 1] = fma2(dn, th2, v[RT - 1]);
    }
}

}  // namespace
}  // namespace hol
