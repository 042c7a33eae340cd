"""Which solves run on chip, by the launches they take: one for a whole solve on chip,
two or three per iteration otherwise. Marked gpu.

FP32 at every lattice size while the state fits, FP64 for the small systems its rule
takes; not above L = 20 in FP64 (no kernel), nor where the state does not fit (L = 32,
Ltau = 400) or the rule finds the two-kernel iteration faster (16 right-hand sides of
L = 20 in FP64), nor with the option off, a preconditioner or the exact propagator."""
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


def _launches(ctx, nr, prec, **kw):
    g = torch.Generator(device=DEV)
    g.manual_seed(2)
    ctx.set_field(torch.randn(ctx.Ltau, ctx.N, dtype=torch.float64, device=DEV, generator=g))
    b = torch.randn(nr, ctx.Ltau, ctx.N, dtype=torch.float64, device=DEV, generator=g)
    v = torch.empty_like(b)
    n0 = hg.hol_launch_count()
    ctx.cg_solve(b, v, tol=1e-9, max_iter=20, prec=prec, raise_on_nonconv=False, **kw)
    return hg.hol_launch_count() - n0


F32 = [(4, 2, 1), (4, 40, 1), (6, 28, 3), (8, 120, 2), (10, 50, 7), (12, 34, 2), (14, 60, 4), (16, 160, 2),
       (18, 30, 2), (20, 40, 3), (22, 18, 2), (24, 26, 2), (26, 46, 2), (28, 120, 2), (30, 38, 2), (32, 200, 16),
       (8, 24, 700)]


@pytest.mark.parametrize("L,T,nr,prec,on", [(*s, hg.HOL_F32, True) for s in F32] +
                         [(4, 40, 1, hg.HOL_F64, True), (8, 24, 1, hg.HOL_F64, True),
                          (32, 400, 1, hg.HOL_F32, False), (22, 18, 2, hg.HOL_F64, False),
                          (32, 4, 1, hg.HOL_F64, False), (20, 120, 16, hg.HOL_F64, False)])
def test_path(L, T, nr, prec, on):
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=nr) as ctx:
        assert (_launches(ctx, nr, prec) == 1) == on
        ctx.set_option("resident_cg", 0)
        assert _launches(ctx, nr, prec) > 20


def test_other_solves_keep_the_iteration_kernels():
    with hg.Context(L=8, Ltau=24, alpha=1.0, max_rhs=1) as ctx:
        assert _launches(ctx, 1, hg.HOL_F32, precond=True) > 20
    with hg.Context(L=8, Ltau=24, alpha=1.0, max_rhs=1, kinetic=hg.HOL_KINETIC_EXACT) as ctx:
        assert ctx.get_option("resident_cg") == 0
        assert _launches(ctx, 1, hg.HOL_F32) > 20
