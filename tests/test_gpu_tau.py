"""Tau transforms of the preconditioner and the CG update joined to the forward one.

The FP32 transforms of the compile-time lengths use another radix plan than the
FP64 ones (one radix 8 pass where the power of two is odd): the FP32 application
is compared with the FP64 one, at both tile widths and at lengths without a
compile-time plan. Bound: that of the FP32 oracle comparison, 2e-5 of the largest
result. The joined update loads a thread's first elements ahead of the step
length: solves with fewer, exactly as many and more elements than that, certified by
the FP64 residual that the solver itself must report (it recomputes it, so the two
agree to the rounding of one FP64 operator). Marked gpu.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

hg = pytest.importorskip("paper_2203_01291_gb300")

DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    hg.build.build()
    torch.cuda.set_device(0)


def _field(ctx, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    ctx.set_field(torch.randn(ctx.Ltau, ctx.N, dtype=torch.float64, device=DEV, generator=g))
    return g


# (L, Ltau, right-hand sides): 40, 120, 160, 200 have compile-time plans; tiles are
# twice as wide when N n_rhs > 64 multiprocessors' worth of sites (10240 is above)
@pytest.mark.parametrize("L,T,nr", [(4, 40, 1), (16, 40, 40), (6, 120, 3), (32, 120, 10), (10, 160, 1),
                                    (32, 160, 10), (12, 200, 2), (16, 200, 40), (8, 80, 2), (4, 14, 3)])
def test_fp32_application_against_fp64(L, T, nr):
    with hg.Context(L=L, Ltau=T, alpha=1.1, max_rhs=max(2, nr)) as ctx:
        g = _field(ctx, 7 * L + T)
        v = torch.randn(nr, T, L * L, dtype=torch.float64, device=DEV, generator=g)
        for which in (hg.HOL_PINV, hg.HOL_PINVT, hg.HOL_PINV_PINVT):
            w64, w32 = torch.empty_like(v), torch.empty_like(v, dtype=torch.float32)
            ctx.precond_apply(which, v, w64)
            ctx.precond_apply(which, v.float(), w32)
            err = (w32.double() - w64).abs().max() / w64.abs().max()
            assert float(err) < 2e-5, (which, float(err))


@pytest.mark.parametrize("prec", [hg.HOL_F32, hg.HOL_F64])
@pytest.mark.parametrize("L,T,nr", [(4, 40, 1), (16, 128, 40), (8, 160, 160), (8, 200, 160), (6, 126, 2),
                                    (6, 256, 2), (6, 300, 2)])
def test_preconditioned_solve_is_certified(L, T, nr, prec):
    tol = 1e-9
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=max(2, nr)) as ctx:
        g = _field(ctx, 3 * L + T)
        R = torch.randn(nr, T, L * L, dtype=torch.float64, device=DEV, generator=g)
        b, v, q = torch.empty_like(R), torch.empty_like(R), torch.empty_like(R)
        ctx.fermion_matvec(hg.HOL_OP_MT, R, b)
        it, res = ctx.cg_solve(b, v, tol=tol, prec=prec, precond=True)
        ctx.fermion_matvec(hg.HOL_OP_MTM, v, q)
        true = ((b - q).flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)).cpu().numpy()
        assert np.all(it > 0) and np.all(res < tol)
        assert np.all(true < tol + 1e-12) and np.allclose(true, res, rtol=1e-2, atol=1e-12)
