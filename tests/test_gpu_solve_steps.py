"""Step lengths of the plain mixed CG, on chip and as two kernels. Marked gpu."""
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


@pytest.mark.parametrize("on", [1, 0])
@pytest.mark.parametrize("L,T,every", [(8, 40, 8), (16, 60, 16), (24, 30, 12), (28, 20, 14), (32, 40, 16)])
def test_first_step_length(L, T, every, on):
    """The first step from b is alpha = |b|^2 / |M b|^2, read off a component of b that is
    one. b has a row of ones every `every` sites and s = 0.7 ... 1 times 2^-12.1 elsewhere, and
    the field is such that every component of M b is of order one at random. An FP32
    chain of squares that starts with a one loses every s^2 after it (less than half
    an ulp): a chain down the rows 11 to 15 of them for every one, with s^2 3.8e-8 on
    average 4.2e-7 to 5.7e-7 of |b|^2. Summed by groups of four, with the groups' sums in
    compensated pairs, at most three are lost for every one, 1.1e-7. alpha is rounded to
    FP32, 6e-8. In |M b|^2 rounding is random (1e-8 of the sum at most) but for the hopping
    constant's own, 3e-8 of tanh(0.1) in each of four bonds, twice: 2.4e-8. Bound: 2.1e-7."""
    g = torch.Generator(device=DEV)
    g.manual_seed(L)
    row = torch.arange(L, device=DEV)[:, None] % every == 0
    s = 2.0 ** -12.1 * (0.7 + 0.3 * torch.rand(T, L, L, dtype=torch.float64, device=DEV, generator=g))
    b = torch.where(row, 1.0, s).to(torch.float32).to(torch.float64).reshape(1, T, L * L)
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=1) as ctx:
        ctx.set_option("resident_cg", on)
        w, v = torch.empty_like(b), torch.empty_like(b)
        ctx.set_field(torch.zeros(T, L * L, dtype=torch.float64, device=DEV))
        ctx.fermion_matvec(hg.HOL_OP_M, b, w)
        cb = (w - b).abs()[0]                                    # C b
        u = 0.5 + torch.rand(T, L * L, dtype=torch.float64, device=DEV, generator=g)
        ctx.set_field(-torch.log(u / cb) / 0.1)                  # D C b = u
        ctx.fermion_matvec(hg.HOL_OP_M, b, w)
        alpha = float((b * b).sum() / (w * w).sum())
        ctx.cg_solve(b, v, tol=1e-12, max_iter=1, prec=hg.HOL_F32, raise_on_nonconv=False)
        got = v.reshape(T, L, L)[:, ::every]
        assert float((got / alpha - 1.0).abs().max()) < 2.1e-7


@pytest.mark.parametrize("on", [1, 0])
@pytest.mark.parametrize("prec,tol,rel", [(hg.HOL_F64, 1e-10, 50), (hg.HOL_F32, 1e-5, 100000)])
@pytest.mark.parametrize("L,T", [(4, 40), (6, 30), (8, 24)])
def test_check_after_the_first_one_below_tol(L, T, prec, tol, rel, on):
    """A solve ends at the check after the first one whose residual is below tol: capped one
    interval earlier, where the cap forces the true residual, it is certified already.
    In FP32 a single segment (tol above its drift from the true residual), so the
    recursive residual decides there too; it is the true one but for its drift, 1e-7 of |b|
    at most, so it may be above tol by that."""
    g = torch.Generator(device=DEV)
    g.manual_seed(100 + L)
    with hg.Context(L=L, Ltau=T, alpha=1.0, max_rhs=1) as ctx:
        ctx.set_option("resident_cg", on)
        ctx.set_field(torch.randn(T, L * L, dtype=torch.float64, device=DEV, generator=g))
        for _ in range(5):
            R = torch.randn(1, T, L * L, dtype=torch.float64, device=DEV, generator=g)
            b, v = torch.empty_like(R), torch.empty_like(R)
            ctx.fermion_matvec(hg.HOL_OP_MT, R, b)
            kw = dict(tol=tol, prec=prec, check_every=10, reliable_every=rel)
            it, _ = ctx.cg_solve(b, v, **kw)
            drift = 1e-7 if prec == hg.HOL_F32 else 1e-13
            _, res = ctx.cg_solve(b, v, max_iter=int(it[0]) - 10, raise_on_nonconv=False, **kw)
            assert res[0] < tol + drift
            _, res = ctx.cg_solve(b, v, max_iter=int(it[0]) - 20, raise_on_nonconv=False, **kw)
            assert res[0] > tol - drift
