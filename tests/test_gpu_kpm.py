"""Chebyshev kernels of the preconditioner (kpm_registers 4, the default) against
the general shared-memory kernel (0) on the same inputs: every lattice size, both
precisions, P^-1, P^-T and both, right-hand side counts on either side of the
launch rules (lane groups left idle, one or two multiprocessors per problem, both
transform tiles) and even Ltau of every radix mix. Marked gpu.

Both evaluate the same series of at most a few hundred steps; a step's rounding
is a few units in the last place of vectors no larger than the input, so the
bounds are those of the oracle comparison: 1e-11 (FP64) and 2e-5 (FP32) of the
largest result.
"""
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


CASES = [(4, 40, 1), (4, 14, 9), (6, 30, 4), (8, 120, 3), (10, 50, 5), (12, 84, 2), (14, 196, 3),
         (16, 160, 2), (16, 2, 1), (18, 90, 2), (20, 120, 2), (20, 42, 40), (22, 168, 3), (24, 70, 2),
         (26, 60, 3), (28, 120, 2), (28, 36, 70), (30, 112, 2), (32, 200, 2), (32, 200, 16), (32, 10, 3)]


@pytest.mark.parametrize("dt,tol", [(torch.float64, 1e-11), (torch.float32, 2e-5)])
@pytest.mark.parametrize("L,T,nr", CASES)
def test_strip_kernels_equal_the_shared_memory_kernel(L, T, nr, dt, tol):
    g = torch.Generator(device=DEV)
    g.manual_seed(L * 1000 + T)
    with hg.Context(L=L, Ltau=T, alpha=1.2, max_rhs=max(2, nr)) as ctx:
        ctx.set_field(torch.randn(T, L * L, dtype=torch.float64, device=DEV, generator=g))
        v = torch.randn(nr, T, L * L, dtype=dt, device=DEV, generator=g)
        for which in (hg.HOL_PINV, hg.HOL_PINVT, hg.HOL_PINV_PINVT):
            out = {}
            for kpm in (4, 0):
                ctx.set_option("kpm_registers", kpm)
                out[kpm] = torch.full_like(v, float("nan"))
                ctx.precond_apply(which, v, out[kpm])
            err = (out[4] - out[0]).abs().max() / out[0].abs().max()
            assert float(err) < tol, (which, float(err))
