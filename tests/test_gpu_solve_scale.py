"""Plain CG does not depend on the scale of the right-hand side: a power of two in
front of b is the same power of two in front of v, bit for bit, with the same
iterations and residuals, over the range in which |b| itself can be formed
(about 1e-154 ... 1e154); other factors are certified as well. Marked gpu."""
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


def _inputs(ctx, nr, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    ctx.set_field(torch.randn(ctx.Ltau, ctx.N, dtype=torch.float64, device=DEV, generator=g))
    R = torch.randn(nr, ctx.Ltau, ctx.N, dtype=torch.float64, device=DEV, generator=g)
    b = torch.empty_like(R)
    ctx.fermion_matvec(hg.HOL_OP_MT, R, b)
    return b


# clusters of one and of several blocks, with and without tensor memory; FP64 on chip
@pytest.mark.parametrize("L,T,prec", [(4, 40, hg.HOL_F32), (8, 120, hg.HOL_F32), (16, 160, hg.HOL_F32),
                                      (32, 100, hg.HOL_F32), (4, 40, hg.HOL_F64), (8, 24, hg.HOL_F64)])
def test_powers_of_two(L, T, prec):
    kw = dict(tol=1e-10, max_iter=20000, prec=prec)
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=4) as ctx:
        b = _inputs(ctx, 4, L + T)
        v0, v1 = torch.empty_like(b), torch.empty_like(b)
        it0, r0 = ctx.cg_solve(b, v0, **kw)
        # a different power for every right-hand side of one solve
        for ks in ((-60, 60, -90, 100), (-120, 126, 1, -1), (-400, 400, -280, 310)):
            f = torch.tensor([2.0 ** k for k in ks], dtype=torch.float64, device=DEV)[:, None, None]
            it1, r1 = ctx.cg_solve(b * f, v1, **kw)
            assert np.array_equal(it0, it1) and np.array_equal(r0, r1), ks
            assert torch.equal(v0 * f, v1), ks


@pytest.mark.parametrize("scale", [1e-30, 1e-20, 3e-10, 1e12, 1e20, 1e30])
def test_other_factors(scale):
    with hg.Context(L=8, Ltau=60, alpha=1.0, max_rhs=2) as ctx:
        b = _inputs(ctx, 2, 3) * scale
        v, q = torch.empty_like(b), torch.empty_like(b)
        it, res = ctx.cg_solve(b, v, tol=1e-10, max_iter=20000, prec=hg.HOL_F32)
        ctx.fermion_matvec(hg.HOL_OP_MTM, v, q)
        true = ((b - q).flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)).cpu().numpy()
        assert np.all(res < 1e-10) and np.all(true < 1e-10 + 1e-13)


@pytest.mark.parametrize("prec", [hg.HOL_F32, hg.HOL_F64])
def test_tolerance_below_what_a_residual_can_reach(prec):
    """tol far below the FP64 rounding of b: the cap ends the solve, and the solution is as
    good as FP64 allows (a residual of some rounding errors of |M^T M| |v|)."""
    with hg.Context(L=4, Ltau=40, alpha=1.0, max_rhs=1) as ctx:
        b = _inputs(ctx, 1, 9)
        v = torch.empty_like(b)
        it, res = ctx.cg_solve(b, v, tol=1e-30, max_iter=3000, prec=prec, reliable_every=100000,
                               raise_on_nonconv=False)
        assert it[0] == 3000 and res[0] < 1e-12
