"""How a solve on chip fails: a wait between the blocks of a cluster that runs out
(option resident_wait_ms 0: at once, the copies on their way are still awaited), and
several right-hand sides that fail in different ways. Marked gpu."""
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


# with and without tensor memory; more right-hand sides than clusters; FP64
@pytest.mark.parametrize("L,T,nr,prec", [(16, 160, 1, hg.HOL_F32), (8, 120, 3, hg.HOL_F32),
                                         (32, 200, 20, hg.HOL_F32), (8, 120, 1, hg.HOL_F64)])
def test_wait_that_runs_out(L, T, nr, prec):
    kw = dict(tol=1e-8, prec=prec)
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=nr) as ctx:
        b = _inputs(ctx, nr, L)
        v0, v1 = torch.empty_like(b), torch.empty_like(b)
        it0, _ = ctx.cg_solve(b, v0, **kw)
        assert ctx.get_option("resident_wait_ms") == 1000
        ctx.set_option("resident_wait_ms", 0)
        for solve in (ctx.cg_solve, ctx.cg_solve_graph):
            with pytest.raises(hg.HolError) as e:
                solve(b, v1, **kw)
            assert e.value.code == hg._abi.HOL_ETIMEOUT
        ctx.set_option("resident_wait_ms", 1000)
        it1, _ = ctx.cg_solve(b, v1, **kw)      # the context goes on
        assert torch.equal(v0, v1) and list(it0) == list(it1)
        for bad in (-1, 10001):
            with pytest.raises(hg.HolError):
                ctx.set_option("resident_wait_ms", bad)


def test_a_number_that_is_not_finite_counts_over_a_missed_tolerance():
    """One NaN among right-hand sides that later run into the iteration cap: the captured
    batch reports the former, whichever is recorded last."""
    with hg.Context(L=8, Ltau=40, alpha=1.0, max_rhs=16) as ctx:
        xi = _inputs(ctx, 16, 1)
        xi[3, 5, 7] = float("nan")
        out = torch.empty_like(xi)
        G2 = torch.empty(80, 8, 8, dtype=torch.float64, device=DEV)
        opts = hg.hol_cg_opts(1e-12, 40, 0, hg.HOL_F32, 50, 10)
        with pytest.raises(hg.HolError) as e:
            hg.measure_batch_graph([ctx], [xi], [out], [G2], opts)
        assert e.value.code == hg._abi.HOL_ENUMERIC
