"""The one-launch field set-up, the banded force and the one-launch FP64 M^T M on
both sides of their size rules, against plain torch FP64 values of the same
definitions (the bond products written out by rolls). Marked gpu.

Bounds: a result is a sum of a few dozen products; 1e-13 of the largest value
for the operator, 1e-12 for the force (the oracle tests' bounds), 1e-11 for the
action (a sum of n_pf N Ltau terms of both signs).
"""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

hg = pytest.importorskip("paper_2203_01291_gb300")

DEV = "cuda"
DTAU, ALPHA, W0 = 0.1, 1.1, 0.8


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    hg.build.build()
    torch.cuda.set_device(0)


def _bond(v, dim, odd):
    ch, sh = math.cosh(DTAU), math.sinh(DTAU)
    L = v.shape[dim]
    even = torch.arange(L, device=v.device) % 2 == (1 if odd else 0)
    shape = [1] * v.dim()
    shape[dim] = L
    partner = torch.where(even.view(shape), v.roll(-1, dim), v.roll(1, dim))
    return ch * v + sh * partner


def _C(v, trans=False):
    order = [(-1, 0), (-1, 1), (-2, 0), (-2, 1)]
    for dim, odd in reversed(order) if trans else order:
        v = _bond(v, dim, odd)
    return v


def _signs(T):
    s = -torch.ones(T, 1, 1, dtype=torch.float64, device=DEV)
    s[0] = 1.0
    return s


def _gen(L, T, nr, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    x = torch.randn(T, L, L, dtype=torch.float64, device=DEV, generator=g)
    v = torch.randn(nr, T, L, L, dtype=torch.float64, device=DEV, generator=g)
    return g, x, v


SHAPES = [(4, 2, 1), (4, 40, 3), (6, 30, 2), (8, 120, 2), (8, 120, 40), (10, 14, 5), (12, 60, 1),
          (14, 50, 2), (16, 160, 2), (16, 160, 16), (18, 22, 4), (20, 120, 2), (22, 10, 2),
          (24, 160, 2), (26, 16, 1), (28, 120, 2), (30, 24, 3), (32, 200, 2), (32, 200, 16)]


@pytest.mark.parametrize("L,T,nr", SHAPES)
def test_operator_and_force(L, T, nr):
    g, x, v = _gen(L, T, nr, 31 * L + T)
    b = torch.randn(nr, T, L, L, dtype=torch.float64, device=DEV, generator=g)
    s = _signs(T)
    D = torch.exp(-DTAU * ALPHA * x)
    with hg.Context(L=L, Ltau=T, alpha=ALPHA, omega0=W0, max_rhs=max(2, nr)) as ctx:
        ctx.set_field(x)
        # spectral bounds of the field set-up
        dbar = D.mean(0)
        lo, hi = ctx.bounds()
        e4 = math.exp(4 * DTAU)
        assert abs(lo - float(dbar.min()) / e4) < 1e-13 * lo and abs(hi - float(dbar.max()) * e4) < 1e-13 * hi
        # M^T M
        w = v + s * D * _C(v).roll(1, 1)
        ref = w + _C(s * D * w, True).roll(-1, 1)
        out = torch.full_like(v, float("nan"))
        ctx.fermion_matvec(hg.HOL_OP_MTM, v, out)
        assert float((out - ref).abs().max()) < 1e-13 * float(ref.abs().max())
        # force and action, with and without the bosonic part, twice (the block counts return to zero)
        y = D * _C(v).roll(1, 1)
        Ff = (DTAU * ALPHA) * (s * (v + s * y) * y - 0.5 * (b * v).roll(1, 1)).sum(0)
        lap = x.roll(-1, 0) - 2 * x + x.roll(1, 0)
        Fb = DTAU * W0 ** 2 * x - lap / DTAU
        S = 0.5 * float((b * v).sum())
        scale = 0.5 * float((b * v).abs().sum())
        F = torch.empty_like(x)
        SF = torch.empty(1, dtype=torch.float64, device=DEV)
        for bos in (True, False, True):
            F.fill_(float("nan"))
            SF.fill_(float("nan"))
            ctx.force(v, b, F, with_bosonic=bos, S_F=SF)
            want = Ff + Fb if bos else Ff
            assert float((F - want).abs().max()) < 1e-12 * float(want.abs().max())
            assert abs(float(SF) - S) < 1e-11 * scale
        F.fill_(float("nan"))
        ctx.force(v, b, F, with_bosonic=True)
        assert float((F - Ff - Fb).abs().max()) < 1e-12 * float((Ff + Fb).abs().max())
