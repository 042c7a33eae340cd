"""How a solve on chip fails: several right-hand sides that fail in different ways.
Marked gpu."""
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
