// FP64 out = M^T M v in one launch for small systems: each lane group (strip.cuh)
// computes one slice of the result from v_{t-1}, v_t and v_{t+1},
//   w_t = v_t + s_t D_t C v_{t-1},  w_{t+1} = v_{t+1} + s_{t+1} D_{t+1} C v_t,
//   out_t = w_t + C^T s_{t+1} D_{t+1} w_{t+1},
// applying C once more per slice than M and M^T in turn. While every warp has a
// quarter multiprocessor to itself the extra arithmetic (an FP64 instruction
// holds it for sixty cycles, some 17 per value) costs less than a second launch
// and its trip through L2: L = 8, Ltau = 120, 2 rhs 11.7 -> 8.2 us.
#include "internal.cuh"
#include "strip.cuh"

namespace hol {
namespace {

template <int L>
__global__ void __launch_bounds__(32) k_MTM64(const double* __restrict__ v, double* __restrict__ out,
                                              const double* __restrict__ ev, int T, int n_rhs, double th)
{
    pdl_wait();      // the input comes from the previous kernel of the stream
    const PdlTriggerAtExit pdl_at_exit;
    using K = RGeo<L>;
    constexpr int N = L * L, E = K::E, RT = K::RT;
    const K geo;
    const long u_raw = (long)blockIdx.x * K::G + geo.g;      // slice of a right-hand side
    const bool live = geo.ok && u_raw < (long)T * n_rhs;
    const long u = live ? u_raw : 0;
    const int t = (int)(u % T);
    const long base = (u / T) * T * N;
    const int tm = t == 0 ? T - 1 : t - 1, tp = t + 1 == T ? 0 : t + 1;
    double a[E], b[E], w[E], d[E], d2[E];
#pragma unroll
    for (int q = 0; q < RT; ++q) {
        const double2 z = make_double2(0.0, 0.0);
        const bool h = geo.has(q);
        const int so = geo.site(q);
        auto ld = [&](const double* p) { return h ? *reinterpret_cast<const double2*>(p + so) : z; };
        const double2 vm = ld(v + base + (long)tm * N), v0 = ld(v + base + (long)t * N),
                      vp = ld(v + base + (long)tp * N), e0 = ld(ev + (long)t * N),
                      ep = ld(ev + (long)tp * N);
        a[2 * q] = vm.x; a[2 * q + 1] = vm.y;
        b[2 * q] = v0.x; b[2 * q + 1] = v0.y;
        w[2 * q] = vp.x; w[2 * q + 1] = vp.y;
        d[2 * q] = t == 0 ? e0.x : -e0.x; d[2 * q + 1] = t == 0 ? e0.y : -e0.y;
        d2[2 * q] = tp == 0 ? ep.x : -ep.x; d2[2 * q + 1] = tp == 0 ? ep.y : -ep.y;
    }
    rc_apply<double, L>(a, geo, th);
#pragma unroll
    for (int e = 0; e < E; ++e) a[e] = fma(d[e], a[e], b[e]);      // w_t
    rc_apply<double, L>(b, geo, th);
#pragma unroll
    for (int e = 0; e < E; ++e) b[e] = d2[e] * fma(d2[e], b[e], w[e]);
    rc_apply_t<double, L>(b, geo, th);
    if (live)
#pragma unroll
        for (int q = 0; q < RT; ++q)
            if (geo.has(q))
                *reinterpret_cast<double2*>(out + base + (long)t * N + geo.site(q)) =
                    make_double2(a[2 * q] + b[2 * q], a[2 * q + 1] + b[2 * q + 1]);
}

template <int L>
int run_mtm64(const hol_ctx* c, const double* v, double* out, int n_rhs, cudaStream_t s)
{
    const long units = (long)c->T * n_rhs, warps = (units + RGeo<L>::G - 1) / RGeo<L>::G;
    // one warp per quarter multiprocessor (and at most 12 values per lane: L <= 18): beyond
    // either, M and M^T in turn take less FP64 time than is saved
    if (warps > 4L * c->sms) return kNotTaken;
    HOL_CUDA(launch_pdl(c, k_MTM64<L>, (int)warps, 32, 0, s, v, out, c->ev64, c->T, n_rhs, c->th));
    HOL_CHECK_LAUNCH("k_MTM64");
    return HOL_OK;
}

}  // namespace

int launch_MTM64(const hol_ctx* c, const double* v, double* out, int n_rhs, cudaStream_t s)
{
    if (c->exact) return kNotTaken;
    switch (c->L) {
#define X(LL) case LL: return run_mtm64<LL>(c, v, out, n_rhs, s);
        X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18)
#undef X
    }
    return kNotTaken;
}

}  // namespace hol
