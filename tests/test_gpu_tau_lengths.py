"""Tau transforms without a compile-time length, against the oracle: lengths with an odd
power of two (one radix 8 pass in FP32), without one and with none, both tile widths,
and lengths whose twiddles no longer fit in shared memory beside the tile (FP64 above
1408, FP32 above 1564). Marked gpu.

Bounds: those of the oracle comparison, 1e-11 (FP64) and 2e-5 (FP32) of the largest value;
five times that in FP32 for series of up to 700 terms (the two long lengths).
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


# 24 = 8 3, 56 = 8 7, 96 = 32 3, 168 = 8 21, 512 = 2^9; 48, 144, 180: even power; 50, 126, 150: one 2
@pytest.mark.parametrize("T", [8, 24, 48, 50, 56, 96, 126, 144, 150, 168, 180, 512, 1400, 1440, 1568])
def test_against_the_oracle(T):
    # narrow tiles, then wide ones: N n_rhs beyond 64 sites per multiprocessor (of at most 160)
    w = hi.Workload("p", L=4, Ltau=T, alpha=1.0, omega0=1.0, x_std=1.0, seed=T)
    x, m = hi.phonon_field(w), D.model_of(w)
    v = hi.gaussian_vectors(w, 1, seed=7)
    refs = {hg.HOL_PINV: D.precond_inverse_apply(m, x, v[0]),
            hg.HOL_PINVT: D.precond_inverse_apply(m, x, v[0], trans=True)}
    for nr in (1, 641):
        if nr > 1 and T > 600:
            continue
        with hg.Context(L=4, Ltau=T, alpha=1.0, omega0=1.0, max_rhs=nr) as ctx:
            ctx.set_field(torch.tensor(x, device=DEV))
            for which, ref in refs.items():
                for dt, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5 if T < 600 else 1e-4)):
                    vt = torch.tensor(v, device=DEV, dtype=dt).expand(nr, T, 16).contiguous()
                    out = torch.empty_like(vt)
                    ctx.precond_apply(which, vt, out)
                    r = torch.tensor(ref, device=DEV)
                    err = float((out.double() - r).abs().max() / r.abs().max())
                    assert err < tol, (which, dt, nr, err)
