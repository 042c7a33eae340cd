// Plan and launch of the on-chip conjugate gradients (resident.cuh).
#include <algorithm>

#include "resident.cuh"

namespace hol {
namespace {

constexpr int kMaxCluster = 16;
constexpr size_t kResSmem = 220 * 1024;   // dynamic part; the reductions' static part beside it
// Shared memory that keeps a second block off the multiprocessor. A block that
// allocates tensor memory waits until it is free, and two clusters that held
// one multiprocessor's each and waited for the other's would never end: the
// instances that allocate it never share a multiprocessor.
constexpr size_t kOneBlock = 117 * 1024;

ResKernel res_kernel(int prec, int L, int K, bool tm)
{
    if (prec == HOL_F64) return tm ? ResKernel{} : resident_kernel_f64(L, K);
    return L >= 24 ? resident_kernel_f32_large(L, K, tm)
         : L >= 14 ? resident_kernel_f32_mid(L, K, tm) : resident_kernel_f32_small(L, K, tm);
}

int launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&at)[1], const ResPlan& p, int clusters,
                  cudaStream_t s)
{
    cfg = {};
    cfg.gridDim = dim3(p.cs * clusters);
    cfg.blockDim = dim3(32 * p.warps);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return HOL_OK;
}

}  // namespace

// Every cluster size and register set that fits, with the clusters the device
// holds at once: asked of the driver once per context and precision, since a
// program may solve for another number of right-hand sides at every call (the
// questions, ten to thirty of each kind, took as long as a small solve).
static void build_table(hol_ctx* c, int prec)
{
    ResTable& tab = c->res_table[prec == HOL_F64 ? 1 : 0];
    tab.n = 0;
    tab.built = 1;
    if (c->exact) return;
    const size_t w = prec == HOL_F64 ? 8 : 4;
    for (int cs = 1; cs <= kMaxCluster && cs <= c->T; ++cs)
        for (int tm = 0; tm < 2; ++tm) {
            ResPlan p{};
            p.cs = cs;
            p.slots = (c->T + cs - 1) / cs;
            ResKernel k{};
            for (int K : {1, 2, 4}) {
                k = res_kernel(prec, c->L, K, tm != 0);
                if (!k.fn) continue;
                p.k = K;
                p.warps = (p.slots + 2 + K * k.g - 1) / (K * k.g);   // the own slices and two copies
                if (p.warps <= 16) break;
                k.fn = nullptr;
            }
            if (!k.fn) continue;
            p.fn = k.fn;
            p.smem = (size_t)((tm ? 2 : 4) * p.slots + 11) * k.sl * w;
            if (tm) {
                // p, x and s D: three windows of K E columns, four warps side by side
                int cols = 32;
                while (cols < (p.warps + 3) / 4 * 3 * p.k * k.e) cols *= 2;
                p.tm_cols = cols;
                p.smem = std::max(p.smem, kOneBlock);
            }
            if (p.smem > kResSmem) continue;
            if (cs > 8 && cudaFuncSetAttribute((const void*)k.fn,
                                               cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                              cudaSuccess) {
                cudaGetLastError();
                continue;
            }
            if (smem_raise((const void*)k.fn, p.smem) != HOL_OK) continue;
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute at[1];
            launch_config(cfg, at, p, 1, nullptr);
            if (cudaOccupancyMaxActiveClusters(&p.clusters, (const void*)k.fn, &cfg) != cudaSuccess ||
                p.clusters < 1) {
                cudaGetLastError();
                continue;
            }
            // measured (us): the block barriers and the scalar chain; the
            // exchange across blocks; a lane's own chain; the block's bandwidth
            const double vals = (double)(p.slots + 2) * c->N, ke = p.k * k.e;
            p.us = prec == HOL_F64 ? 3.5 + (cs > 1 ? 0.5 : 0.0) + 0.4 * ke + vals * 0.0035
                                   : 1.3 + (cs > 1 ? 0.3 : 0.0) + ke * (tm ? 0.06 : 0.13) + vals * 0.00025;
            tab.p[tab.n++] = p;
        }
}

// The plan for n_rhs right-hand sides: the smallest modelled time of one
// iteration of all of them,
//   max(1, n_rhs / resident clusters) * (latency + values per block * rate).
ResPlan resident_plan(hol_ctx* c, int prec, int n_rhs)
{
    const ResTable& tab = c->res_table[prec == HOL_F64 ? 1 : 0];
    if (!tab.built) build_table(c, prec);
    ResPlan best{};
    best.us = 1e30;
    for (int k = 0; k < tab.n; ++k) {
        const ResPlan& p = tab.p[k];
        const double us = std::max(1.0, (double)n_rhs / p.clusters) * p.us;
        if (us < best.us) {
            best = p;
            best.us = us;
        }
    }
    best.clusters = std::min(best.clusters, n_rhs);
    return best;
}

bool resident_ok(hol_ctx* c, const hol_cg_opts* o, int n_rhs)
{
    if (!c->resident || c->exact || o->precond || c->fused || c->merged || c->persist) return false;
    const ResPlan p = resident_plan(c, o->prec, n_rhs);
    if (!p.fn) return false;
    if (o->prec == HOL_F64) {
        // bound by the FP64 pipes of the clusters' multiprocessors, where the
        // two-kernel iteration uses all of them: taken while the modelled time
        // stays below the latter's (measured: 13 us at n = 640, 23 us at two
        // right-hand sides of 40,960 values, where this one would take 22)
        return p.us < 9.0 + 1.0e-5 * (double)n_rhs * c->n;
    }
    return true;
}

// Enqueue one solve (results in dcg_state(c): it, done, tres; g[DCG_ERR],
// g[DCG_STICKY]).
int resident_enqueue(hol_ctx* c, const double* b, double* v, int n_rhs, const hol_cg_opts* o,
                     cudaStream_t s)
{
    const ResPlan p = resident_plan(c, o->prec, n_rhs);
    const bool f64 = o->prec == HOL_F64;
    ResArgs a;
    a.b = b;
    a.v = v;
    a.r = f64 ? (void*)c->v64a : (void*)c->v32a;
    a.p = f64 ? (void*)c->v64b : (void*)c->v32b;
    a.t64 = c->v64c;
    a.ev = f64 ? (const void*)c->ev64 : (const void*)c->ev32;
    a.ev64 = c->ev64;
    a.T = c->T;
    a.n_rhs = n_rhs;
    a.max_iter = o->max_iter;
    a.chk = o->check_every > 0 ? o->check_every : 10;
    a.rel_every = (!f64 && o->reliable_every > 0) ? o->reliable_every : 1 << 30;
    a.slots = p.slots;
    a.tm_cols = p.tm_cols;
    a.wait_tries = (int)((long)c->resident_wait * 1000000L / kMbTryNs);
    a.tol = o->tol;
    a.th = c->th;
    a.d = dcg_state(c);
    // iteration counts, flags, states and the solve's counters (not the
    // sticky failure flag) start at zero
    HOL_CUDA(cudaMemsetAsync(a.d.it, 0, (size_t)((a.d.g + DCG_STICKY) - a.d.it) * sizeof(int), s));
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    launch_config(cfg, at, p, p.clusters, s);
    HOL_CUDA(cudaLaunchKernelEx(&cfg, p.fn, a));
    HOL_CHECK_LAUNCH("k_cg_resident");
    return HOL_OK;
}

}  // namespace hol
