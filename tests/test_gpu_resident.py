"""Plain CG with its state on chip (option resident_cg, the default): the same
certified solutions as the two-kernel iteration over every lattice size, uneven
and tiny slice counts, more right-hand sides than clusters (segments handed
between clusters), zero and non-finite right-hand sides and the iteration cap.
Marked gpu.

Bounds. A solve certifies |b - M^T M v| / |b| < tol in FP64, so the residual
recomputed here with the FP64 operator may exceed tol by that operator's own
rounding only (1e-13 of |b|, the operator's test bound times |M^T M v| ~ |b|).
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


def _inputs(ctx, nr, seed, zero=None):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    x = torch.randn(ctx.Ltau, ctx.N, dtype=torch.float64, device=DEV, generator=g)
    R = torch.randn(nr, ctx.Ltau, ctx.N, dtype=torch.float64, device=DEV, generator=g)
    if zero is not None:
        R[zero] = 0.0
    ctx.set_field(x)
    b = torch.empty_like(R)
    ctx.fermion_matvec(hg.HOL_OP_MT, R, b)
    return b


def _residual(ctx, b, v):
    q = torch.empty_like(b)
    ctx.fermion_matvec(hg.HOL_OP_MTM, v, q)
    return ((b - q).flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)).cpu().numpy()


SHAPES = [(L, T, nr) for L, T, nr in [
    (4, 2, 1), (4, 40, 1), (4, 14, 3), (6, 28, 3), (8, 120, 2), (8, 6, 5), (10, 50, 7), (12, 34, 2),
    (14, 60, 4), (16, 160, 2), (16, 22, 9), (18, 30, 2), (20, 40, 3), (22, 18, 2), (24, 26, 2),
    (26, 46, 2), (28, 120, 2), (30, 38, 2), (32, 200, 2), (32, 4, 1)]]


@pytest.mark.parametrize("prec", [hg.HOL_F32, hg.HOL_F64])
@pytest.mark.parametrize("L,T,nr", SHAPES)
def test_certified_and_equal_to_the_two_kernel_solve(L, T, nr, prec):
    tol = 1e-10
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=max(2, nr)) as ctx:
        b = _inputs(ctx, nr, 100 * L + T)
        sols = []
        for on in (1, 0):
            ctx.set_option("resident_cg", on)
            assert ctx.get_option("resident_cg") == on
            v = torch.full_like(b, float("nan"))
            it, res = ctx.cg_solve(b, v, tol=tol, prec=prec)
            assert np.all(res < tol) and np.all(it > 0)
            true = _residual(ctx, b, v)
            assert np.all(true < tol + 1e-13) and np.allclose(true, res, rtol=1e-2, atol=1e-13)
            sols.append(v)
        # both certified: their difference has a residual of at most 2 tol
        d = sols[0] - sols[1]
        q = torch.empty_like(d)
        ctx.fermion_matvec(hg.HOL_OP_MTM, d, q)
        rel = (q.flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)).max().item()
        assert rel < 2 * tol + 1e-13


@pytest.mark.parametrize("L,T,nr,chk,rel", [(8, 24, 700, 10, 50), (16, 40, 200, 4, 20),
                                            (32, 60, 40, 10, 50), (20, 30, 170, 7, 11)])
def test_more_right_hand_sides_than_clusters(L, T, nr, chk, rel):
    """Unfinished right-hand sides pass between clusters after every segment;
    a solve of the same right-hand side alone certifies the same residual."""
    tol = 1e-9
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=nr) as ctx:
        b = _inputs(ctx, nr, 7 * L, zero=nr // 2)
        v = torch.full_like(b, float("nan"))
        it, res = ctx.cg_solve(b, v, tol=tol, prec=hg.HOL_F32, check_every=chk, reliable_every=rel)
        assert np.all(res < tol)
        assert res[nr // 2] == 0.0 and it[nr // 2] == 0 and float(v[nr // 2].abs().max()) == 0.0
        live = np.arange(nr) != nr // 2
        true = _residual(ctx, b, v)
        assert np.all(true[live] < tol + 1e-13)
        # repeatable, whichever cluster ran which segment
        v2 = torch.full_like(b, float("nan"))
        it2, res2 = ctx.cg_solve(b, v2, tol=tol, prec=hg.HOL_F32, check_every=chk, reliable_every=rel)
        assert np.array_equal(it, it2) and np.array_equal(res, res2) and torch.equal(v, v2)


@pytest.mark.parametrize("prec", [hg.HOL_F32, hg.HOL_F64])
def test_iteration_cap_and_bad_input(prec):
    with hg.Context(L=8, Ltau=24, alpha=1.0, max_rhs=3) as ctx:
        b = _inputs(ctx, 3, 5)
        v = torch.empty_like(b)
        it, res = ctx.cg_solve(b, v, tol=1e-30, max_iter=12, prec=prec, check_every=5,
                               raise_on_nonconv=False)
        assert np.all(it == 12) and np.all(res > 0)
        assert np.allclose(_residual(ctx, b, v), res, rtol=1e-6)
        with pytest.raises(hg.HolError) as e:
            ctx.cg_solve(b, v, tol=1e-30, max_iter=12, prec=prec)
        assert e.value.code == hg._abi.HOL_ENOTCONV
        bad = b.clone()
        bad[1, 3, 5] = float("nan")
        with pytest.raises(hg.HolError) as e:
            ctx.cg_solve(bad, v, tol=1e-8, prec=prec)
        assert e.value.code == hg._abi.HOL_ENUMERIC
        it, res = ctx.cg_solve(b, v, tol=1e-8, prec=prec)   # the context goes on
        assert np.all(res < 1e-8)


def test_graph_and_host_solves_are_the_same():
    with hg.Context(L=12, Ltau=40, alpha=1.1, max_rhs=5) as ctx:
        b = _inputs(ctx, 5, 11)
        v0, v1 = torch.empty_like(b), torch.empty_like(b)
        it0, r0 = ctx.cg_solve(b, v0, tol=1e-10, prec=hg.HOL_F32)
        it1, r1 = ctx.cg_solve_graph(b, v1, tol=1e-10, prec=hg.HOL_F32)
        assert np.array_equal(it0, it1) and np.array_equal(r0, r1) and torch.equal(v0, v1)
