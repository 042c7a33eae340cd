"""Performance cases: what a user of the library runs, through its public calls.

Each case is one pass of a public entry point on device-resident inputs, with
the context (the handle a program keeps) and the input buffers prepared before.
Shapes are those of the repository's workloads: the L = 4, Ltau = 40 parity
lattice, the L = 16, Ltau = 160 trajectory, the L = 32, Ltau = 200 benchmark,
the L = 24, Ltau = 160 force and the chains of L = 8 ... 28 at Ltau = 120.

Kinds
  matvec   fermion_matvec (M, M^T or M^T M; FP64 or FP32)
  precond  precond_apply (P^-1, P^-T or both; FP64 or FP32)
  force    hol_set_field and force, as every force evaluation of a trajectory
           calls them: the field, then dS/dx and S_F from the solved pairs
  cg       cg_solve to a certified residual (FP64 or mixed, with or without P)
  hmc      fourier_accel_leapfrog: one whole trajectory
  chains   hmc_batch_graph: one trajectory of uneven independent chains
  measure  stochastic_measure: the Green-function estimates of a probe set

Solves run to a residual of 1e-12 (inside trajectories 1e-9 for the forces and
1e-10 for the action), the tight end of what this repository's configurations
and tests ask for: the result is then fixed to about 1e-10, whatever rounding
path reaches it. Iteration counts are statistics of the way there, not
results, and are not returned.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2203_01291_gb300 as hg

DTAU, HOP, MU = 0.1, 1.0, 0.0
OPS = {"M": hg.HOL_OP_M, "MT": hg.HOL_OP_MT, "MTM": hg.HOL_OP_MTM}
PCS = {"PINV": hg.HOL_PINV, "PINVT": hg.HOL_PINVT, "PINV_PINVT": hg.HOL_PINV_PINVT}
CHAIN_SIZES = "8,12,16,20,24,28"
# even, prime factors 2, 3, 5, 7 only (what the tau transforms take)
TAUS = [40, 48, 56, 60, 70, 80, 84, 90, 96, 100, 112, 120, 126, 140, 144, 150, 160, 168, 180, 192,
        196, 200]


def listed():
    big = dict(L=32, T=200, omega0=0.5, alpha=1.0, shift=0.0)
    hmc = dict(L=16, T=160, omega0=1.0, alpha=1.5, shift=0.5)
    grad = dict(L=24, T=160, omega0=1.0, alpha=1.2, shift=0.0)
    tiny = dict(L=4, T=40, omega0=1.0, alpha=1.0, shift=0.0)

    def chain(L):
        return dict(L=L, T=120, omega0=1.0, alpha=1.0, shift=0.0)

    return [
        # the smallest calls: the FP64 operator on a small chain's two
        # pseudofermions, and the parity lattice's FP64 solve
        dict(name="matvec64_chain8", kind="matvec", prec=64, op="MTM", rhs=2, tune=False, **chain(8)),
        dict(name="cg64_tiny", kind="cg", prec=64, pc=False, rhs=1, tune=False, **tiny),
        # the operator of the benchmark's solve, 16 right-hand sides in FP32
        dict(name="matvec32_big32", kind="matvec", prec=32, op="MTM", rhs=16, tune=True, **big),
        # the preconditioner inside an HMC trajectory (two pseudofermions), on
        # the benchmark's 16 right-hand sides, and in FP64 on a size that is
        # no power of two
        dict(name="precond32_hmc16", kind="precond", prec=32, op="PINV_PINVT", rhs=2, **hmc),
        dict(name="precond32_big32", kind="precond", prec=32, op="PINV_PINVT", rhs=16, **big),
        dict(name="precond64_chain20", kind="precond", prec=64, op="PINV_PINVT", rhs=2, **chain(20)),
        # one force evaluation (new field, two pseudofermions)
        dict(name="force_grad24", kind="force", rhs=2, **grad),
        # the benchmark: 16 mixed-precision solves in one call
        dict(name="cg32_big32", kind="cg", prec=32, pc=False, rhs=16, tune=True, **big),
        # the FP64 preconditioned solve of a trajectory's two pseudofermions
        dict(name="pcg64_hmc16", kind="cg", prec=64, pc=True, rhs=2, tune=False, **hmc),
        # one trajectory of 20 steps with 4 bosonic sub-steps, mixed precision
        dict(name="hmc16", kind="hmc", prec=32, rhs=2, steps=20, sub=4, tune=True, **hmc),
        # one chain of every lattice size, in one captured graph per step
        dict(name="chains", kind="chains", prec=32, rhs=2, steps=4, sub=4, tune=True,
             sizes=CHAIN_SIZES, T=120, omega0=1.0, alpha=1.0, shift=0.0),
        # a 128-probe measurement of the largest chain
        dict(name="measure_chain28", kind="measure", prec=32, rhs=128, tune=True, **chain(28)),
    ]


def draw(rng):
    """One more case of the same ranges (sizes up to the listed ones)."""
    kind = rng.choice(["matvec", "matvec", "precond", "precond", "force", "cg", "cg", "hmc",
                       "measure"])
    omega0 = rng.choice([0.5, 0.75, 1.0])
    # the field's effect on the operator grows with alpha / omega0: at most the benchmark's 2
    case = dict(kind=kind, L=2 * rng.randint(2, 16), T=rng.choice(TAUS), omega0=omega0,
                alpha=round(rng.uniform(0.7, min(1.5, 2.0 * omega0)), 2),
                shift=rng.choice([0.0, 0.5]), prec=rng.choice([32, 32, 64]))

    def many(most):   # right-hand sides, log-uniform; at most `most` and the largest call's size
        cap = max(1, min(most, int(1.3e7 / (case["L"] ** 2 * case["T"]))))
        return max(1, min(cap, int(round(math.exp(rng.uniform(0.0, math.log(cap + 1)))))))

    if kind == "matvec":
        case.update(op=rng.choice(["M", "MT", "MTM", "MTM"]), rhs=many(64),
                    tune=rng.choice([False, True]))
    elif kind == "precond":
        case.update(op=rng.choice(["PINV", "PINVT", "PINV_PINVT", "PINV_PINVT"]), rhs=many(32))
    elif kind == "force":
        case.update(rhs=many(16))
    elif kind == "cg":
        pc = rng.choice([False, True])
        case.update(pc=pc, tune=rng.choice([False, True]),
                    rhs=many(4 if case["prec"] == 64 or pc else 32))
    elif kind == "hmc":
        case.update(prec=32, rhs=2, steps=rng.randint(1, 4), sub=rng.choice([1, 2, 4]), tune=False,
                    L=2 * rng.randint(2, 12))
    else:   # the lattice transforms take the same prime factors as the tau ones
        case.update(prec=32, tune=True, L=rng.choice([4, 6, 8, 10, 12, 14, 16, 18, 20, 24, 28]),
                    T=rng.choice([40, 60, 80, 96, 100, 120]))
        case.update(rhs=max(2, many(128)))
    return case


# ---------------------------------------------------------------- inputs
def _gauss(seed, stream, shape):
    g = np.random.Generator(np.random.PCG64([int(seed), stream]))
    return g.standard_normal(shape)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _field(case, seed, L=None, k=0):
    """x[tau][i] of the free phonon's width 1 / omega0 around a shift, i.i.d."""
    L = L or case["L"]
    return _dev(_gauss(seed, 100 + k, (case["T"], L * L)) / case["omega0"] + case["shift"])


def _vectors(case, seed, stream, rhs, L=None):
    L = L or case["L"]
    return _dev(_gauss(seed, stream, (rhs, case["T"], L * L)))


def _probes(case, seed):
    g = np.random.Generator(np.random.PCG64([int(seed), 7]))
    z = g.integers(0, 2, size=(case["rhs"], case["T"], case["L"] ** 2), dtype=np.int8)
    return _dev(z).to(torch.float64) * 2.0 - 1.0


class _State:
    pass


def _ctx(case, L=None):
    return hg.Context(L=L or case["L"], Ltau=case["T"], dtau=DTAU, t=HOP, mu=MU,
                      alpha=case["alpha"], omega0=case["omega0"], max_rhs=max(2, case["rhs"]))


def _md(case):
    return hg.md_opts(0.01, case["steps"], case["sub"], case["omega0"], force_tol=1e-9,
                      action_tol=1e-10, prec=hg.HOL_F32 if case["prec"] == 32 else hg.HOL_F64,
                      precond=True)


def prepare(case, seed):
    s = _State()
    s.case = case
    kind = case["kind"]
    if kind == "chains":
        sizes = [int(v) for v in case["sizes"].split(",")]
        s.ctx = [_ctx(case, L) for L in sizes]
        s.x0 = [_field(case, seed, L, k) for k, L in enumerate(sizes)]
        s.x = [x.clone() for x in s.x0]
        s.Rpf = [_vectors(case, seed, 200 + k, case["rhs"], L) for k, L in enumerate(sizes)]
        s.Rp = [_vectors(case, seed, 300 + k, 1, L)[0].contiguous() for k, L in enumerate(sizes)]
        for c, x in zip(s.ctx, s.x0):
            c.set_field(x)
            c.tune(case["rhs"])
        s.opts = _md(case)
        torch.cuda.synchronize()
        return s
    rhs = case["rhs"]
    s.ctx = _ctx(case)
    s.x0 = _field(case, seed)
    s.ctx.set_field(s.x0)
    if case.get("tune"):
        s.ctx.tune(rhs)
    if kind in ("matvec", "precond"):
        dt = torch.float64 if case["prec"] == 64 else torch.float32
        s.v = _vectors(case, seed, 1, rhs).to(dt)
        s.out = torch.empty_like(s.v)
    elif kind == "force":   # a solved pair (v, b = M^T M v), b in plain torch
        s.v = _vectors(case, seed, 1, rhs)
        s.b = _Ref(case, s.x0).MTM(s.v).contiguous()
        s.F = torch.empty_like(s.x0)
        s.S = torch.empty(1, dtype=torch.float64, device="cuda")
    elif kind == "cg":      # b = M^T R, the pseudofermion right-hand side
        s.b = _Ref(case, s.x0).MT(_vectors(case, seed, 1, rhs)).contiguous()
        s.v = torch.empty_like(s.b)
    elif kind == "hmc":
        s.x = s.x0.clone()
        s.Rpf = _vectors(case, seed, 1, rhs)
        s.Rp = _vectors(case, seed, 2, 1)[0].contiguous()
        s.opts = _md(case)
    elif kind == "measure":
        s.xi = _probes(case, seed)
        s.Gxi = torch.empty_like(s.xi)
        s.G2 = torch.empty(2 * case["T"], case["L"], case["L"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "matvec":
        s.ctx.fermion_matvec(OPS[case["op"]], s.v, s.out)
        return s.out
    if kind == "precond":
        s.ctx.precond_apply(PCS[case["op"]], s.v, s.out)
        return s.out
    if kind == "force":
        s.ctx.set_field(s.x0)
        s.ctx.force(s.v, s.b, s.F, with_bosonic=True, S_F=s.S)
        return {"dSdx": s.F, "S_F": s.S}
    if kind == "cg":
        s.ctx.cg_solve(s.b, s.v, tol=1e-12, max_iter=100000, precond=case["pc"],
                       prec=hg.HOL_F32 if case["prec"] == 32 else hg.HOL_F64)
        return s.v
    if kind == "hmc":
        s.x.copy_(s.x0)
        acc, _, terms = s.ctx.fourier_accel_leapfrog(s.x, s.Rpf, s.Rp, s.opts, 0.0)
        return {"x": s.x, "accepted": acc, "terms": terms}
    if kind == "chains":
        for x, x0 in zip(s.x, s.x0):
            x.copy_(x0)
        acc, _ = hg.hmc_batch_graph(s.ctx, s.x, s.Rpf, s.Rp, s.opts, [0.0] * len(s.ctx))
        return {"x": s.x, "accepted": acc}
    s.ctx.stochastic_measure(s.xi, s.Gxi, s.G2, tol=1e-12,
                             prec=hg.HOL_F32 if case["prec"] == 32 else hg.HOL_F64)
    return {"Gxi": s.Gxi, "G2": s.G2}


# ---------------------------------------------------------------- work
def _iterations(case):
    """Rough CG iterations of a solve to 1e-12 on these fields."""
    its = {4: 130, 6: 250, 8: 420, 10: 600}.get(case["L"], 900 + 60 * max(0, case["L"] - 12))
    return its * case["T"] / 120.0 * (0.4 if case.get("pc") else 1.0)


def work(case):
    kind, T = case["kind"], case["T"]
    if kind == "chains":
        per = [work(dict(case, kind="hmc", L=int(L))) for L in case["sizes"].split(",")]
        return {k: sum(p[k] for p in per) for k in ("bytes", "flops")}
    n, rhs = case["L"] ** 2 * T, case["rhs"]
    w = 4 if case.get("prec") == 32 else 8
    apply = 10.0 * n * rhs              # four bond colours and the diagonal, 2 flops each
    if kind == "matvec":
        return {"bytes": 2 * n * rhs * w + n * w, "flops": apply * (2 if case["op"] == "MTM" else 1)}
    db = 0.85 if case["omega0"] == 1.0 else 1.0   # about the width of the Bbar spectrum
    orders = sum(max(1, int(db * (T / (2 * math.pi * (k + 0.5)) + 1))) for k in range(T // 2))
    series = orders * case["L"] ** 2 * rhs * 2 * 16.0   # complex vectors, 16 flops per part and step
    fft = 2 * 2.5 * n * rhs * math.log2(T)
    pinv = fft + series * (2 if case.get("op", "PINV_PINVT") == "PINV_PINVT" else 1)
    if kind == "precond":
        return {"bytes": 2 * n * rhs * w, "flops": pinv}
    if kind == "force":
        return {"bytes": 2 * n * rhs * 8 + 2 * n * 8, "flops": (apply + 8.0 * n * rhs)}
    its = _iterations(dict(case, pc=case.get("pc", kind == "hmc")))
    per_it = 2 * apply + 10.0 * n * rhs + (pinv if case.get("pc", kind == "hmc") else 0.0)
    if kind == "cg":
        return {"bytes": 2 * n * rhs * 8 + n * 8, "flops": its * per_it}
    if kind == "hmc":
        return {"bytes": n * 8 * (2 + rhs + 1), "flops": (case["steps"] + 2) * its * per_it}
    return {"bytes": 2 * n * rhs * 8 + 3 * n * 8,
            "flops": its * per_it + 2 * 5.0 * n * rhs * math.log2(n)}


# ---------------------------------------------------------------- 64-bit values
class _Ref:
    """M, M^T and the force in plain FP64 torch, from the definitions:
    (M v)_tau = v_tau + s_tau D_tau C v_{tau-1}, s_0 = 1, s_{tau>0} = -1,
    D = exp(-dtau (alpha x - mu)), C the four bond colours (x even, x odd,
    y even, y odd), each bond [[cosh, sinh], [sinh, cosh]](dtau t)."""

    def __init__(self, case, x):
        self.L, self.T = case["L"], case["T"]
        self.alpha, self.omega0 = case["alpha"], case["omega0"]
        self.x = x.reshape(self.T, self.L, self.L)
        self.D = torch.exp(-DTAU * (self.alpha * self.x - MU))
        sg = -torch.ones(self.T, dtype=torch.float64, device=x.device)
        sg[0] = 1.0
        self.sD = self.D * sg[:, None, None]
        self.s = sg[:, None, None]
        self.ch, self.sh = math.cosh(DTAU * HOP), math.sinh(DTAU * HOP)

    def _bond(self, v, colour):
        dim = -1 if colour < 2 else -2
        off = colour & 1
        if off:
            v = v.roll(-1, dim)
        shp = v.shape
        w = v.reshape(shp[:-1] + (self.L // 2, 2)) if dim == -1 else \
            v.reshape(shp[:-2] + (self.L // 2, 2, self.L))
        w = (self.ch * w + self.sh * w.flip(dim)).reshape(shp)
        return w.roll(1, dim) if off else w

    def C(self, v, trans=False):
        for colour in (3, 2, 1, 0) if trans else (0, 1, 2, 3):
            v = self._bond(v, colour)
        return v

    def _grid(self, v):
        return v.reshape(-1, self.T, self.L, self.L)

    def M(self, v):
        g = self._grid(v)
        return (g + self.sD * self.C(g).roll(1, 1)).reshape(v.shape)

    def MT(self, u):
        g = self._grid(u)
        return (g + self.C(self.sD * g, True).roll(-1, 1)).reshape(u.shape)

    def MTM(self, v):
        return self.MT(self.M(v))

    def force(self, v, b):
        gv, gb = self._grid(v), self._grid(b)
        y = self.D * self.C(gv).roll(1, 1)
        u = gv + self.s * y
        F = (DTAU * self.alpha) * (self.s * u * y - 0.5 * (gb * gv).roll(1, 1)).sum(0)
        x = self.x
        lap = x.roll(-1, 0) - 2.0 * x + x.roll(1, 0)
        F = F + DTAU * self.omega0 ** 2 * x - lap / DTAU
        return F.reshape(self.T, -1), 0.5 * (gv * gb).sum()

    def pinv(self, v, which):
        """The preconditioner: the twisted tau transform, the Chebyshev series
        of (I - exp(-i phi) Bbar)^-1 per frequency, and back."""
        L, T = self.L, self.T
        dbar = self.D.mean(0)
        g = math.exp(4.0 * DTAU * HOP)
        lo, hi = float(dbar.min()) / g, float(dbar.max()) * g
        db = hi - lo
        tau = torch.arange(T, dtype=torch.float64, device=v.device)
        tw = torch.exp(-1j * math.pi * tau / T)[:, None, None]
        vh = torch.fft.fft(self._grid(v) * tw, dim=1, norm="ortho")[:, : T // 2]
        phi = [2.0 * math.pi * (w + 0.5) / T for w in range(T // 2)]
        order = [max(1, int(math.floor(db * (1.0 / p + 1.0)))) for p in phi]
        coef = torch.zeros(T // 2, max(order), dtype=torch.complex128)
        for w, (p, nP) in enumerate(zip(phi, order)):
            nq = 2 * nP
            th = math.pi * (torch.arange(nq, dtype=torch.float64) + 0.5) / nq
            f = 1.0 / (1.0 - complex(math.cos(p), -math.sin(p)) *
                       (lo + (torch.cos(th) + 1.0) * db / 2).to(torch.complex128))
            m = torch.arange(nP, dtype=torch.float64)
            c = torch.cos(m[:, None] * th[None, :]).to(torch.complex128) @ f * (2.0 / nq)
            c[0] /= 2.0
            coef[w, :nP] = c
        coef = coef.to(v.device)[None, :, :, None, None]

        def series(u, trans):
            cf = coef.conj() if trans else coef

            def A(z):
                bz = self.C(dbar * z, True) if trans else dbar * self.C(z)
                return 2.0 * (bz - lo * z) / db - z

            prev, cur = u, A(u)
            acc = cf[:, :, 0] * u
            for m in range(1, coef.shape[2]):
                acc = acc + cf[:, :, m] * cur
                prev, cur = cur, 2.0 * A(cur) - prev
            return acc

        if which != "PINV":
            vh = series(vh, True)
        if which != "PINVT":
            vh = series(vh, False)
        full = torch.cat([vh, vh.flip(1).conj()], dim=1)
        return (torch.fft.ifft(full, dim=1, norm="ortho") * tw.conj()).real.reshape(v.shape)

    def solve(self, b):
        """Conjugate gradients on M^T M to the rounding of the residual."""
        g = b.reshape(-1, self.T * self.L ** 2)
        x = torch.zeros_like(g)
        bn = (g * g).sum(1, keepdim=True)
        for _ in range(2):              # one restart from the true residual
            r = g - self.MTM(x)
            p, rr = r, (r * r).sum(1, keepdim=True)
            for it in range(40000):
                q = self.MTM(p)
                al = rr / (p * q).sum(1, keepdim=True)
                x = x + al * p
                r = r - al * q
                rn = (r * r).sum(1, keepdim=True)
                if it % 25 == 24 and bool((rn <= 1e-29 * bn).all()):
                    break
                p = r + rn / rr * p
                rr = rn
        return x.reshape(b.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("hmc", "chains"):       # thousands of solves deep: no independent value
        return None
    if kind in ("cg", "measure") and case["L"] ** 2 * case["T"] * case["rhs"] > 1.3e7:
        return None
    ref = _Ref(case, _field(case, seed))
    rhs = case["rhs"]
    if kind in ("matvec", "precond"):
        v = _vectors(case, seed, 1, rhs)
        if case["prec"] == 32:
            v = v.to(torch.float32).to(torch.float64)
        if kind == "precond":
            return ref.pinv(v, case["op"])
        return {"M": ref.M, "MT": ref.MT, "MTM": ref.MTM}[case["op"]](v)
    if kind == "force":
        v = _vectors(case, seed, 1, rhs)
        F, S = ref.force(v, ref.MTM(v))
        return {"dSdx": F, "S_F": S.reshape(1)}
    if kind == "cg":
        return ref.solve(ref.MT(_vectors(case, seed, 1, rhs)))
    xi = _probes(case, seed)
    Gxi = ref.solve(ref.MT(xi))
    L, T = case["L"], case["T"]
    G2 = torch.zeros(2 * T, L, L, dtype=torch.complex128, device=xi.device)
    for a, b in zip(xi, Gxi):           # circular cross-correlation of the antiperiodic extensions
        a, b = a.reshape(T, L, L), b.reshape(T, L, L)
        fa = torch.fft.fftn(torch.cat([a, -a]))
        G2 += fa.conj() * torch.fft.fftn(torch.cat([b, -b]))
    G2 = torch.fft.ifftn(G2).real / (2.0 * T * L * L * rhs)
    return {"Gxi": Gxi, "G2": G2}
