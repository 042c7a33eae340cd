"""Imaginary-time axes at and beyond the length up to which a block of the Chebyshev
plan holds all its sums and its whole cosine table (Ltau = 1206): the field, the
operator, the plain solve and the preconditioner against the oracle, on both sides
of that length and up to the longest ones. Marked gpu.

Bounds. Operator: one product of five factors per value, 1e-13 of the largest. Solve:
certified in FP64, so the oracle's residual is below tol up to one operator's rounding.
Preconditioner: the bounds of the oracle comparison on short axes, 1e-11 (FP64) and
2e-5 (FP32) of the largest value at series of up to 125 terms; the longest here has
about 700, so five times that in FP32 (FP64: 700 steps of a few 1e-16 stay below
1e-11 as they are).
"""
import numpy as np
import pytest
import torch

import holstein_inputs as hi
from oracle import dense as D

pytestmark = pytest.mark.gpu

hg = pytest.importorskip("paper_2203_01291_gb300")

DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    hg.build.build()
    torch.cuda.set_device(0)


def _setup(L, T, exact=False):
    w = hi.Workload("p", L=L, Ltau=T, alpha=1.0, omega0=1.0, x_std=1.0, seed=T)
    x = hi.phonon_field(w)
    ctx = hg.Context(L=L, Ltau=T, alpha=1.0, omega0=1.0, max_rhs=2,
                     kinetic=hg.HOL_KINETIC_EXACT if exact else hg.HOL_KINETIC_CHECKERBOARD)
    return w, D.model_of(w, "exact" if exact else "checkerboard"), x, ctx


def _err(a, ref):
    return float(np.abs(a.double().cpu().numpy() - ref).max() / np.abs(ref).max())


@pytest.mark.parametrize("L,T", [(4, 1206), (4, 1208), (6, 1500), (4, 1812)])
def test_field_operator_and_solve(L, T):
    w, m, x, ctx = _setup(L, T)
    C = D.kinetic_propagator(m)
    v = hi.gaussian_vectors(w, 1, seed=5)
    with ctx:
        ctx.set_field(torch.tensor(x, device=DEV))
        vt = torch.tensor(v, device=DEV)
        out = torch.empty_like(vt)
        ctx.fermion_matvec(hg.HOL_OP_M, vt, out)
        assert _err(out[0], D.M_apply_blocks(m, x, v[0], C)) < 1e-13
        b = torch.empty_like(vt)
        ctx.fermion_matvec(hg.HOL_OP_MT, vt, b)
        for prec in (hg.HOL_F32, hg.HOL_F64):
            _, res = ctx.cg_solve(b, out, tol=1e-9, prec=prec, max_iter=60000)
            bh = b[0].cpu().numpy()
            q = D.MT_apply_blocks(m, x, D.M_apply_blocks(m, x, out[0].cpu().numpy(), C), C)
            assert res[0] < 1e-9 and np.linalg.norm(bh - q) < (1e-9 + 1e-13) * np.linalg.norm(bh)


def test_exact_propagator_field():
    w, m, x, ctx = _setup(4, 1210, exact=True)
    v = hi.gaussian_vectors(w, 1, seed=6)
    with ctx:
        ctx.set_field(torch.tensor(x, device=DEV))
        vt = torch.tensor(v, device=DEV)
        out = torch.empty_like(vt)
        ctx.fermion_matvec(hg.HOL_OP_MT, vt, out)
        assert _err(out[0], D.MT_apply_blocks(m, x, v[0])) < 1e-13


@pytest.mark.parametrize("L,T", [(4, 1200), (4, 1250), (6, 1568), (4, 1750)])
def test_preconditioner(L, T):
    w, m, x, ctx = _setup(L, T)
    v = hi.gaussian_vectors(w, 1, seed=7)
    refs = {hg.HOL_PINV: D.precond_inverse_apply(m, x, v[0]),
            hg.HOL_PINVT: D.precond_inverse_apply(m, x, v[0], trans=True)}
    with ctx:
        ctx.set_field(torch.tensor(x, device=DEV))
        for which, ref in refs.items():
            for dt, tol in ((torch.float64, 1e-11), (torch.float32, 1e-4)):
                vt = torch.tensor(v, device=DEV, dtype=dt)
                out = torch.empty_like(vt)
                ctx.precond_apply(which, vt, out)
                assert _err(out[0], ref) < tol, (which, dt, _err(out[0], ref))
