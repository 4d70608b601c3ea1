"""Performance cases: what a program that propagates the 3D time-dependent Dirac equation with this
package has it do, each through the public entry points of ``paper_2512_21697_gb300.binding``.

A case is a dict of plain values: ``kind`` says which call is made, the other keys give the
discretised system (N radial B-splines of order ``order``, |kappa| <= ``kmax``, every mu or |mu| = 1/2,
multipoles l <= ``lmax``, box R), the pulse and the solver setting.  The sizes are those of
``workloads.py`` (small, slice, medium, production, batch) and of the tests; ``draw`` spreads them over
the same ranges.

  run       advance a state by a few Crank-Nicolson steps: dirac_run (``graph``) or dirac_step
  batch     advance several instances with their own radial size and pulse: dirac_solve_batch
  residual  the refinement residual A_- psi - A_+ x: dirac_residual
  apply     y = A_+- x in the solve's accurate precision: dirac_apply
  apply32   the complex64 operator of the mixed solve: dirac_apply32
  precond   z = M^-1 r: dirac_precond_apply (complex128) or dirac_precond_apply32
  forward   the initial-guess network on M positions: dirac_guess_forward
  grad      loss and gradient of a training batch: dirac_guess_loss_grad
  spectrum  observables and the photoelectron spectrum of a state: dirac_observables, dirac_spectrum

``exact`` evaluates the same quantities in 64 bits from the discretisation's definition (knots,
splines, dual-kinetic-balance components, Clebsch-Gordan and Gaunt integrals, all formed here) with
numpy and torch.
"""
import functools
import json
import math

import numpy as np
import torch

from paper_2512_21697_gb300 import binding as B
from paper_2512_21697_gb300 import workloads as W

DEV = "cuda"


# ---- cases ---------------------------------------------------------------------------------------

def _system(N, kmax, lmax, R=300.0, order=7, grid=1, two_mu_max=0, E0=0.1, nm=800.0, cycles=3.0, dt=0.005):
    return dict(N=N, kmax=kmax, lmax=lmax, R=R, order=order, grid=grid, two_mu_max=two_mu_max, E0=E0, nm=nm,
                cycles=cycles, dt=dt)


SMALL = _system(60, 4, 2, R=50.0, grid=0, two_mu_max=1, E0=0.05, cycles=1.0, dt=0.01)
SLICE = _system(157, 5, 6)
MEDIUM = _system(600, 14, 6)
PRODUCTION = _system(1000, 30, 6)


def listed():
    return [
        # the smallest propagation: a radial test problem with |mu| = 1/2 and a short pulse, plain FP64,
        # ten steps; launches and the latency of the dependent kernels count
        dict(SMALL, name="run small fp64", kind="run", precision=0, fact=0, driver="graph", steps=10, tol=1e-12,
             phase=0.5),
        # the main use: the production basis at peak field, mixed precision with double-float refinement
        # and the factorised inner operator, two steps of the captured driver
        dict(PRODUCTION, name="run production mixed", kind="run", precision=2, fact=1, driver="graph", steps=2,
             tol=1e-10, phase=0.5),
        # a mid-sized propagation with the library's default options on the host-driven loop, near the
        # pulse start
        dict(MEDIUM, name="step medium mixed", kind="run", precision=2, fact=0, driver="host", steps=2, tol=1e-10,
             phase=0.05),
        # the same system in plain FP64, the setting a user checks the mixed one against
        dict(MEDIUM, name="run medium fp64", kind="run", precision=0, fact=0, driver="graph", steps=2, tol=1e-10,
             phase=0.5),
        # a pulse-parameter scan: eight instances of different radial size and pulse side by side
        dict(name="batch 8 mixed", kind="batch", first=0, count=8, kmax=20, lmax=2, precision=2, fact=1, steps=2,
             tol=1e-10, window=8),
        # the accurate residual alone (a user's check of a state), production size
        dict(PRODUCTION, name="residual production", kind="residual", precision=2, tol=1e-10, phase=0.57),
        # the inner solve's operator alone, factorised, production size
        dict(PRODUCTION, name="apply32 production", kind="apply32", precision=2, fact=1, sign=1, phase=0.43),
        # the same with the default (stored) coupling on a small ragged slice of the production system
        dict(SLICE, name="apply32 slice", kind="apply32", precision=2, fact=0, sign=-1, phase=0.3),
        # the inner solve's preconditioner, production size
        dict(PRODUCTION, name="precond32 production", kind="precond", precision=2, complex64=True),
        # the initial-guess network on every position of the production system (inference of one step)
        dict(name="forward production", kind="forward", M=1861860, tensor_cores=1),
        # one training batch of the initial-guess network (loss and gradient)
        dict(name="grad 4096", kind="grad", B=4096),
        # what is read off a final state: observables with the bound population and dP/dE on a grid
        dict(_system(301, 8, 4), name="spectrum 301", kind="spectrum", e_hi=2.0, n_grid=2000, phase=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "residual", "residual", "apply", "apply32", "apply32", "precond",
                       "forward", "grad", "spectrum"])
    if kind == "forward":
        return dict(kind=kind, M=_log(rng, 100, 1861860), tensor_cores=rng.choice([1, 1, 2]))
    if kind == "grad":
        return dict(kind=kind, B=_log(rng, 64, 8192))
    if kind == "batch":
        return dict(kind=kind, first=rng.randrange(100, 200), count=rng.randrange(2, 8), kmax=_log(rng, 4, 20),
                    lmax=rng.choice([1, 2, 2, 3]), precision=2, fact=rng.choice([0, 1, 1]), steps=1, tol=1e-10,
                    window=rng.choice([0, 4]))
    kmax = _log(rng, 2, 28)
    N = _log(rng, 40, 1000)
    order = 7 if rng.random() < 0.85 else rng.choice([5, 6, 8])
    lmax = rng.choice([1, 2, 3, 4, 5, 6, 6, 8])
    if kind == "spectrum":
        kmax, N = min(kmax, 8), min(N, 301)
    if order != 7 or lmax > 6:   # the general forms: mid-sized at most
        kmax, N = min(kmax, 14), min(N, 600)
    # box and field as the workloads have them: the small box for short grids
    c = _system(N, kmax, lmax, R=rng.choice([50.0, 100.0]) if N < 150 else 300.0, order=order,
                two_mu_max=rng.choice([0, 0, 0, 1]), E0=round(math.exp(rng.uniform(math.log(0.02), math.log(0.2))), 4),
                nm=round(rng.uniform(400, 1600), 1), cycles=float(rng.randrange(2, 7)))
    c.update(kind=kind, phase=round(rng.uniform(0.05, 0.95), 3))
    if kind == "run":
        p = rng.choice([0, 1, 2, 2, 2])
        c.update(precision=p, fact=rng.choice([0, 1]) if p == 2 and order == 7 else 0,
                 driver=rng.choice(["graph", "host"]), steps=rng.choice([1, 2, 3]), tol=rng.choice([1e-10, 1e-12]))
        if p < 2 and kmax > 20:
            c["steps"] = 1
    elif kind == "residual":
        c.update(precision=rng.choice([0, 2, 2, 2]), tol=rng.choice([1e-10, 1e-12]))
    elif kind == "apply":
        c.update(precision=rng.choice([0, 0, 2]), sign=rng.choice([1, -1]))
    elif kind == "apply32":
        p = rng.choice([1, 2, 2, 2])
        c.update(precision=p, fact=rng.choice([0, 1]) if p == 2 and order == 7 else 0, sign=rng.choice([1, -1]))
    elif kind == "precond":
        c.update(precision=2, complex64=rng.random() < 0.7)
    else:
        c.update(e_hi=2.0, n_grid=_log(rng, 100, 4000))
    return c


# ---- the program's handles and inputs --------------------------------------------------------------

def _cfg(case):
    m = case["N"] + 5 - case["order"]   # knot intervals, half of them linear up to R / 5
    return dict(Z=1.0, c=W.C_AU, R=case["R"], N=case["N"], order=case["order"], grid=case["grid"],
                r_lin=case["R"] / 5 if case["grid"] else 0.0, n_lin=m // 2 if case["grid"] else 0,
                kappa_max=case["kmax"], two_mu_max=case["two_mu_max"], l_max=case["lmax"], quad=14, E0=case["E0"],
                omega=W.omega_from_nm(case["nm"]), n_cycles=case["cycles"], dt=case["dt"], time_eval=0, t0=0.0)


def _duration(cfg):
    return cfg["n_cycles"] * 2 * math.pi / cfg["omega"]


class _Handle:
    """A basis with its operator, as a program keeps them over a run."""

    def __init__(self, case, cfg, stream=None):
        self.cfg = cfg
        self.bas = B.Basis(cfg)
        self.op = B.Operator(self.bas, cfg, stream=stream, tol=case.get("tol", 1e-10), precision=case.get("precision", 0),
                             max_iter=1000, tol_inner=1e-5, max_outer=30, guess=1)
        if case.get("fact"):
            self.op.set_factorised(case["fact"])
        self.psi0 = torch.from_numpy(self.bas.initial_state()[0]).to(DEV)
        if case["kind"] in ("run", "batch"):   # the buffers its driver runs on
            self.psi = torch.empty_like(self.psi0)
            self.hist = torch.empty(2 * self.bas.n, dtype=torch.complex128, device=DEV)
        n1 = cfg["N"] + 1
        # entries that the boundary condition leaves unused (slot 0), as the library's layout has them
        used = np.ones((self.bas.nch, n1, 2), bool)
        used[:, 0, 0] = self.bas.kappa == -1
        used[:, 0, 1] = self.bas.kappa == 1
        decay = 0.7 ** np.abs(self.bas.kappa)[:, None, None] * np.exp(-3.0 * np.arange(n1) / n1)[None, :, None]
        self.envelope = torch.from_numpy((used * decay).reshape(-1)).to(DEV)

    def wave(self, seed):
        """A seeded random state with the amplitudes of a wave packet: falling off with |kappa| and r."""
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        z = torch.randn(2, self.bas.n, dtype=torch.float64, device=DEV, generator=g)
        z = torch.complex(z[0], z[1]) * self.envelope
        return z / torch.linalg.norm(z)


_KEPT = {}   # the handles of the case at hand, as a program keeps them


def _handle(case):
    key = json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)
    if key not in _KEPT:
        _KEPT.clear()   # the previous case's operators go before the next are set up
        if case["kind"] in ("forward", "grad"):
            _KEPT[key] = B.GuessNet(max(64, case.get("B", 64)), W.guess_net_init(7))
        elif case["kind"] == "batch":
            _KEPT[key] = [_Handle(case, c, torch.cuda.Stream()) for c in _batch_cfgs(case)]
        else:
            _KEPT[key] = [_Handle(case, _cfg(case))]
    return _KEPT[key]


def _batch_cfgs(case):
    return W.batch_instances(case["count"], seed0=case["first"], kappa_max=case["kmax"], l_max=case["lmax"])


def _start_time(case, cfg, seed):
    """A start time near the case's phase of the pulse, another for each seed."""
    return (case.get("phase", 0.5) + 0.02 * (np.random.default_rng(seed).random() - 0.5)) * _duration(cfg)


def _normal(seed, *shape):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn(*shape, device=DEV, generator=g)


def _net_batch(n, seed):
    x = _normal(seed, n, 32)
    x[:, 27:] = 0   # the unused features
    return x, x[:, 12:16] + 0.3 * _normal(seed + 1, n, 4)


def prepare(case, seed):
    kind = case["kind"]
    h = _handle(case)
    if kind == "forward":
        x, _ = _net_batch(case["M"], seed)
        return dict(kind=kind, net=h, x=x, out=torch.empty(case["M"], 4, device=DEV), tc=case["tensor_cores"])
    if kind == "grad":
        x, t = _net_batch(case["B"], seed)
        return dict(kind=kind, net=h, x=x, t=t)
    if kind in ("run", "batch"):
        # the ground state (with a small seeded wave) taken three steps into the pulse, so that the
        # history is what a run has at that point
        insts = []
        for k, i in enumerate(h):
            t = _start_time(case, i.cfg, seed + 1000 * k)
            psi = i.psi0 + 1e-3 * i.wave(seed + 1000 * k)
            hist = torch.zeros(2 * i.bas.n, dtype=torch.complex128, device=DEV)
            torch.cuda.synchronize()
            nh = i.op.step(psi, 3, t, hist=hist)[2]
            insts.append(dict(h=i, psi=psi, hist=hist, n_hist=nh, t=t + 3 * i.cfg["dt"]))
        return dict(kind=kind, insts=insts, steps=case["steps"], driver=case.get("driver"), window=case.get("window"))
    h = h[0]
    psi = h.wave(seed)
    s = dict(kind=kind, op=h.op, t=_start_time(case, h.cfg, seed))
    if kind == "residual":
        s.update(psi=psi, x=psi + 0.01 * h.wave(seed + 1), r=torch.empty_like(psi))
    elif kind == "apply":
        s.update(sign=case["sign"], x=psi, y=torch.empty_like(psi))
    elif kind == "apply32":
        x = psi.to(torch.complex64)
        s.update(sign=case["sign"], x=x, y=torch.empty_like(x))
    elif kind == "precond":
        r = psi.to(torch.complex64) if case["complex64"] else psi
        s.update(r=r, z=torch.empty_like(r), complex64=case["complex64"])
    else:
        s.update(psi=psi + h.psi0, grid=np.linspace(0.0, case["e_hi"], case["n_grid"]), e_hi=case["e_hi"])
        h.op.observables(s["psi"], bound=True)   # the eigenvectors are computed once per operator and window
        h.op.spectrum(s["psi"], 0.0, case["e_hi"], s["grid"])
    return s


# ---- one pass ------------------------------------------------------------------------------------

def _load(inst):
    """The instance's state and history into the buffers the handle's driver runs on."""
    h = inst["h"]
    with torch.cuda.stream(h.op.stream):
        h.psi.copy_(inst["psi"])
        h.hist.copy_(inst["hist"])
    return h


def run(s):
    kind = s["kind"]
    if kind == "run":
        i = s["insts"][0]
        h = _load(i)
        f = h.op.run if s["driver"] == "graph" else h.op.step
        f(h.psi, s["steps"], i["t"], hist=h.hist, n_hist=i["n_hist"])
        return {"psi": h.psi, "hist": h.hist}
    if kind == "batch":
        hs = [_load(i) for i in s["insts"]]
        B.solve_batch([h.op for h in hs], [h.psi for h in hs], [h.hist for h in hs], s["steps"],
                      [i["t"] for i in s["insts"]], n_hist=[i["n_hist"] for i in s["insts"]], window=s["window"])
        return {"psi": [h.psi for h in hs], "hist": [h.hist for h in hs]}
    if kind == "residual":
        return {"bnorm": s["op"].residual(s["t"], s["psi"], s["x"], s["r"]), "r": s["r"]}
    if kind == "apply":
        s["op"].apply(s["sign"], s["t"], s["x"], s["y"])
        return s["y"]
    if kind == "apply32":
        s["op"].apply32(s["sign"], s["t"], s["x"], s["y"])
        return s["y"]
    if kind == "precond":
        (s["op"].precond32 if s["complex64"] else s["op"].precond)(s["r"], s["z"])
        return s["z"]
    if kind == "forward":
        s["net"].forward(s["x"], s["out"], tensor_cores=s["tc"])
        return s["out"]
    if kind == "grad":
        loss, grad = s["net"].loss_grad(s["x"], s["t"])
        return {"loss": loss, "grad": grad}
    obs = s["op"].observables(s["psi"], bound=True)
    return {"obs": obs, "dpde": s["op"].spectrum(s["psi"], 0.0, s["e_hi"], s["grid"])[0]}


# ---- what a pass cannot do without ------------------------------------------------------------------

def _channels(kmax, two_mu_max):
    """Channels (kappa, 2 mu) in the library's order."""
    return [(sg * ak, tm) for tm in range(1 - 2 * kmax, 2 * kmax, 2) if two_mu_max <= 0 or abs(tm) <= two_mu_max
            for ak in range(1, kmax + 1) for sg in (-1, 1) if 2 * ak - 1 >= abs(tm)]


def _orbital(k):
    return k if k > 0 else -k - 1


def _n_terms(kmax, two_mu_max, lmax):
    """(pair, multipole) terms of the coupling: mu and mu +- 1, l within the triangle of the orbital
    momenta of one channel and the partner's opposite kappa, and of their parity."""
    by_mu = {}
    for k, m in _channels(kmax, two_mu_max):
        by_mu.setdefault(m, []).append(k)
    n = 0
    for m, ks in by_mu.items():
        for a in ks:
            for b in by_mu.get(m + 2, ()):
                l1, l2 = _orbital(a), _orbital(-b)
                l3, l4 = _orbital(-a), _orbital(b)
                lo = min(abs(l1 - l2), abs(l3 - l4))
                hi = max(l1 + l2, l3 + l4)
                n += sum(1 for l in range(lo, min(hi, lmax) + 1) if (l1 + l2 + l) % 2 == 0)
    return n


def _operator_work(c):
    """(unknowns, band entries, flops of one complex operator product).  The least known count: the
    coupling through its factors -- six angular sums per (channel, multipole) from the partners
    (12 real multiply-adds per directed term and slot), then two band rows from each of them -- and the
    diagonal blocks."""
    nch, n1, bd = len(_channels(c["kmax"], c["two_mu_max"])), c["N"] + 1, 2 * c["order"] - 1
    terms = _n_terms(c["kmax"], c["two_mu_max"], c["lmax"])
    angular = 2 * terms * n1 * 12
    radial = nch * (c["lmax"] + 1) * n1 * bd * 24
    diagonal = nch * n1 * bd * 4 * 4
    return nch * n1 * 2, 2 * c["kmax"] * n1 * bd * 4, 2 * (angular + radial + diagonal)


def work(case):
    kind = case["kind"]
    if kind == "forward":
        return {"bytes": case["M"] * 36 * 4, "flops": 2 * case["M"] * (32 * 256 + 2 * 256 * 256 + 256 * 4)}
    if kind == "grad":
        return {"bytes": case["B"] * 36 * 4 + 2 * 141060 * 4,
                "flops": 6 * case["B"] * (32 * 256 + 2 * 256 * 256 + 256 * 4)}
    if kind == "batch":
        parts = [work(dict(case, kind="run", N=c["N"], order=7, two_mu_max=0)) for c in _batch_cfgs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, band, flops = _operator_work(case)
    if kind == "spectrum":
        # projections on the levels of a kappa in the window, about pi / R apart in momentum
        levels = math.sqrt(2 * case["e_hi"]) * case["R"] / math.pi
        return {"bytes": n * 16 + 2 * band * 8 + 2 * case["kmax"] * levels * 2 * (case["N"] + 1) * 8,
                "flops": 4 * n * levels + 8 * n * (2 * case["order"] - 1) * 2}
    if kind == "precond":
        kb = 2 * case["order"] - 1
        el = 8 if case["complex64"] else 16
        return {"bytes": 2 * n * el + 2 * case["kmax"] * 2 * (case["N"] + 1) * 3 * kb * el, "flops": 8 * n * 3 * kb}
    pulse = (case["lmax"] + 1) * 3 * 9 * (case["N"] + 1) * (2 * case["order"] - 1) * 8   # the projected pulse matrices
    if kind == "run":   # per step: A_- psi, and A_+ on the guess, and twice per iteration (one at least)
        return {"bytes": case["steps"] * (6 * n * 16 + pulse), "flops": 4 * case["steps"] * flops}
    if kind == "residual":
        return {"bytes": 3 * n * 16 + 2 * band * 8 + pulse, "flops": 2 * flops}
    el = 8 if kind == "apply32" else 16
    return {"bytes": 2 * n * el + 2 * band * el // 2 + pulse, "flops": flops}


# ---- the same quantities in 64 bits ------------------------------------------------------------------

class _Exact:
    """The discretised problem from its definition: B-splines at Gauss-Legendre points, the
    dual-kinetic-balance components P = p0 + kappa p1, Q = q0 + kappa q1, S and H0 per kappa as bands,
    the pulse's multipoles F_l(r, t) and the angular coefficients."""

    def __init__(self, cfg):
        self.cfg = cfg
        k, N, R = cfg["order"], cfg["N"], cfg["R"]
        self.k, self.n1, self.half, m = k, N + 1, k - 1, N + 5 - k
        if cfg["grid"]:
            n_lin, h = cfg["n_lin"], cfg["r_lin"] / cfg["n_lin"]
            M = m - n_lin
            lo, hi = 1.0, 2.0
            for _ in range(300):   # growth factor with h (g + ... + g^M) = R - r_lin
                g = 0.5 * (lo + hi)
                lo, hi = (g, hi) if h * np.sum(g ** np.arange(1.0, M + 1)) < R - cfg["r_lin"] else (lo, g)
            brk = np.concatenate([h * np.arange(n_lin + 1), cfg["r_lin"] + h * np.cumsum(g ** np.arange(1.0, M + 1))])
            brk[m] = R
        else:
            brk = R * np.arange(m + 1) / m
        t = np.concatenate([np.zeros(k - 1), brk, np.full(k - 1, R)])
        gx, gw = np.polynomial.legendre.leggauss(cfg["quad"])
        r = 0.5 * (brk[:-1] + brk[1:])[:, None] + 0.5 * np.diff(brk)[:, None] * gx
        self.r, self.w = r, 0.5 * np.diff(brk)[:, None] * gw          # [interval][point]
        j = np.arange(m) + k - 1                                      # knot span of each interval

        def basis(o):   # order-o splines B_{j-o+1 .. j} at the points, [interval][point][o]
            b = np.ones((m, r.shape[1], 1))
            for q in range(1, o):
                nb = np.zeros((m, r.shape[1], q + 1))
                for i in range(q):
                    right, left = t[j + i + 1][:, None], t[j + i + 1 - q][:, None]
                    nb[..., i] += (right - r) / (right - left) * b[..., i]
                    nb[..., i + 1] += (r - left) / (right - left) * b[..., i]
                b = nb
            return b

        def derive(b, o):   # derivative of the order-o splines from values (or derivatives) of order o - 1
            out = np.zeros(b.shape[:2] + (o,))
            for i in range(o - 1):   # B_{s, o-1}, s = j - o + 2 + i, over t[s + o - 1] - t[s]
                s = j - o + 2 + i
                v = (o - 1) * b[..., i] / (t[s + o - 1] - t[s])[:, None]
                out[..., i + 1] += v
                out[..., i] -= v
            return out

        u, du = basis(k), derive(basis(k - 1), k)
        ddu = derive(derive(basis(k - 2), k - 1), k)
        c2, rr = 2 * cfg["c"], r[..., None]
        z = np.zeros_like(u)
        # [kappa power][type] of P, Q and their derivatives, each [interval][point][k]
        self.P = [[u, du / c2], [z, -u / rr / c2]]
        self.Q = [[du / c2, u], [u / rr / c2, z]]
        self.dP = [[du, ddu / c2], [z, -(du / rr - u / rr ** 2) / c2]]
        self.dQ = [[ddu / c2, du], [(du / rr - u / rr ** 2) / c2, z]]
        self.slot = np.arange(m)[:, None] + np.arange(k)[None, :] - 1   # slot of a local spline; outside: unused
        self.ch = _channels(cfg["kappa_max"], cfg["two_mu_max"])
        self.kappa = np.array([x[0] for x in self.ch])
        self.n = len(self.ch) * 2 * self.n1

    def component(self, F, kappa):
        """The functions of one kappa at the points, [interval][point][k][type]."""
        return np.stack([F[0][t] + kappa * F[1][t] for t in range(2)], axis=-1)

    def used(self, kappa):
        m = np.ones((self.n1, 2), bool)
        m[0] = (kappa == -1, kappa == 1)
        return m

    @functools.lru_cache(maxsize=None)
    def blocks(self, kappa):
        """S and H0 of one kappa, dense (2 n1)^2, on the GPU."""
        cfg, c = self.cfg, self.cfg["c"]
        P, Q, dP, dQ = (self.component(F, kappa) for F in (self.P, self.Q, self.dP, self.dQ))
        w, rr = self.w[..., None, None], self.r[..., None, None]
        U = -cfg["Z"] / rr
        local = []
        for left, right in (((P, P), (Q, Q)),
                            ((P, U * P - c * (dQ - kappa * Q / rr)),
                             (Q, (U - 2 * c * c) * Q + c * (dP + kappa * P / rr)))):
            local.append(sum(np.einsum("iqat,iqbu->iatbu", w * a, b) for a, b in (left, right)))
        out = []
        for L, unit in zip(local, (1.0, 0.0)):
            D = np.zeros((self.n1 + 2 * self.k, 2, self.n1 + 2 * self.k, 2))   # margins for the dropped splines
            for a in range(self.k):
                for b in range(self.k):
                    D[self.slot[:, a], :, self.slot[:, b], :] += L[:, a, :, b, :]
            D = D[:self.n1, :, :self.n1, :]
            off = ~self.used(kappa)
            D[off], D[:, :, off] = 0.0, 0.0
            D[0, off[0], 0, off[0]] = unit
            out.append(torch.from_numpy(D.reshape(2 * self.n1, 2 * self.n1)).to(DEV))
        return out

    def field(self, t):
        """F_l at the points: sum over the carriers of the sin^2 pulse, [l][interval][point]."""
        cfg, T = self.cfg, _duration(self.cfg)
        s, amp = t - cfg["t0"], cfg["E0"] / cfg["omega"]
        F = np.zeros((cfg["l_max"] + 1,) + self.r.shape)
        if not 0 <= s <= T:
            return F
        for w, wt in ((cfg["omega"], 0.5), (cfg["omega"] + 2 * math.pi / T, -0.25),
                      (cfg["omega"] - 2 * math.pi / T, -0.25)):
            x = w * self.r / cfg["c"]
            for l in range(cfg["l_max"] + 1):
                lead = np.prod(x[None] / (2.0 * np.arange(1, l + 1).reshape(-1, 1, 1) + 1), axis=0)
                term, jl = np.ones_like(x), np.ones_like(x)
                for q in range(1, 40):
                    term = term * (-x * x) / (2.0 * q * (2.0 * l + 2 * q + 1))
                    jl = jl + term
                f = math.sin(w * s) * (-1) ** (l // 2) if l % 2 == 0 else -math.cos(w * s) * (-1) ** ((l - 1) // 2)
                F[l] += amp * wt * f * lead * jl
        return F

    @functools.lru_cache(maxsize=None)
    def angular(self):
        """A1[l][a][b] = 4 pi Y_l0 matrix element of sigma_x between (kappa_a, mu_a) and (-kappa_b, mu_b)."""
        x, wx = np.polynomial.legendre.leggauss(4 * self.cfg["kappa_max"] + self.cfg["l_max"] + 8)
        lm = self.cfg["kappa_max"] + 1

        def theta(l_hi, m):   # normalised associated Legendre functions l = m .. l_hi at x
            p = np.full_like(x, math.sqrt(0.5))
            for i in range(1, m + 1):
                p = -p * np.sqrt(1 - x * x) * math.sqrt((2 * i + 1) / (2 * i))
            rows, prev = {m: p}, 0.0
            for l in range(m + 1, l_hi + 1):
                a = math.sqrt((4 * l * l - 1) / (l * l - m * m))
                b = math.sqrt(((l - 1) ** 2 - m * m) / (4 * (l - 1) ** 2 - 1)) if l > m + 1 else 0.0
                rows[l], prev = a * (x * rows[l - 1] - b * prev), rows[l - 1]
            return rows

        def spin(k, tm):   # Clebsch-Gordan factors of the upper and the lower spinor row
            l, mu = _orbital(k), tm / 2
            p, q = math.sqrt(max(0.0, l + mu + 0.5) / (2 * l + 1)), math.sqrt(max(0.0, l - mu + 0.5) / (2 * l + 1))
            return (p, q) if k < 0 else (-q, p)

        ylm0 = theta(self.cfg["l_max"], 0)
        tab = [theta(lm + 1, m) for m in range(lm + 1)]
        A = np.zeros((self.cfg["l_max"] + 1, len(self.ch), len(self.ch)))
        where = {}
        for i, (k, tm) in enumerate(self.ch):
            where.setdefault(tm, []).append(i)
        for l in range(self.cfg["l_max"] + 1):
            pref = math.sqrt(4 * math.pi * (2 * l + 1)) / math.sqrt(2 * math.pi)
            for tm, rows in where.items():
                for other, m, up in ((tm - 2, (tm - 1) // 2, True), (tm + 2, (tm + 1) // 2, False)):
                    if other not in where or abs(m) > lm:
                        continue
                    T = np.zeros((lm + 2, len(x)))
                    for q, v in tab[abs(m)].items():
                        T[q] = v
                    G = pref * (T * (wx * ylm0[l])) @ T.T
                    cols = where[other]
                    la = [_orbital(self.ch[a][0]) for a in rows]
                    lb = [_orbital(-self.ch[b][0]) for b in cols]
                    ca = np.array([spin(self.ch[a][0], tm)[0 if up else 1] for a in rows])
                    cb = np.array([spin(-self.ch[b][0], other)[1 if up else 0] for b in cols])
                    A[l][np.ix_(rows, cols)] += ca[:, None] * G[np.ix_(la, lb)] * cb[None, :]
        A[np.abs(A) < 1e-13] = 0.0
        return torch.from_numpy(A).to(DEV)

    def groups(self):
        """Channels of each kappa."""
        return [(int(k), np.flatnonzero(self.kappa == k)) for k in np.unique(self.kappa)]

    def per_kappa(self, f, x):
        """f(kappa, columns) on the channels of each kappa; x [channel][2 n1]."""
        y = torch.empty_like(x)
        for k, idx in self.groups():
            i = torch.from_numpy(idx).to(DEV)
            y[i] = f(k, x[i].T).T
        return y

    def points(self, F, x):
        """sum over the functions of x at the points: [channel][interval point] complex."""
        out = torch.empty(x.shape[0], self.r.size, dtype=x.dtype, device=DEV)
        slot = torch.from_numpy(self.slot).to(DEV) + self.k
        for k, idx in self.groups():
            i = torch.from_numpy(idx).to(DEV)
            pad = torch.zeros(len(idx), self.n1 + 2 * self.k, 2, dtype=x.dtype, device=DEV)
            pad[:, self.k:self.k + self.n1] = x[i].reshape(len(idx), self.n1, 2)
            f = torch.from_numpy(self.component(F, k)).to(DEV)
            loc = torch.view_as_real(pad[:, slot])                                   # [c][interval][k][type][2]
            out[i] = torch.view_as_complex(torch.einsum("iqat,ciatz->ciqz", f, loc).contiguous()).reshape(len(idx), -1)
        return out

    def project(self, F, g):
        """Integrals of the functions with g (already weighted): the transpose of points()."""
        out = torch.empty(g.shape[0], 2 * self.n1, dtype=g.dtype, device=DEV)
        m = self.slot.shape[0]
        for k, idx in self.groups():
            i = torch.from_numpy(idx).to(DEV)
            f = torch.from_numpy(self.component(F, k)).to(DEV)
            loc = torch.einsum("iqat,ciqz->ciatz", f, torch.view_as_real(g[i].reshape(len(idx), m, -1)))
            acc = torch.zeros(len(idx), self.n1 + 2 * self.k, 2, 2, dtype=torch.float64, device=DEV)
            for a in range(self.k):   # a local spline's slots are distinct over the intervals
                acc[:, torch.from_numpy(self.slot[:, a]).to(DEV) + self.k] += loc[:, :, a]
            v = torch.view_as_complex(acc[:, self.k:self.k + self.n1].contiguous())
            v[:, ~torch.from_numpy(self.used(k)).to(DEV)] = 0
            out[i] = v.reshape(len(idx), -1)
        return out

    def coupling(self, t, x):
        """X(t) x with H = H0 + i X: -c sum_l [A1 P . F_l Q_b - A2 Q . F_l P_b]."""
        A, F = self.angular(), self.field(t)
        Pb, Qb = self.points(self.P, x), self.points(self.Q, x)
        gP, gQ = torch.zeros_like(Pb), torch.zeros_like(Qb)
        mm = lambda M, z: torch.complex(M @ z.real, M @ z.imag)  # noqa: E731
        for l in range(A.shape[0]):
            f = torch.from_numpy((F[l] * self.w).reshape(-1)).to(DEV)
            gP += f * mm(A[l], Qb)
            gQ += f * mm(A[l].T, Pb)
        return -self.cfg["c"] * (self.project(self.P, gP) - self.project(self.Q, gQ))

    def apply(self, sign, t, x, couple=True):
        """A_sign(t) x = (S + sign i tau H0) x - sign tau X x."""
        tau = 0.5 * self.cfg["dt"]
        v = x.reshape(len(self.ch), -1)

        def diagonal(k, z):
            S, H = self.blocks(k)
            return torch.complex(S @ z.real - sign * tau * (H @ z.imag), S @ z.imag + sign * tau * (H @ z.real))

        y = self.per_kappa(diagonal, v)
        if couple:
            y -= sign * tau * self.coupling(t, v)
        return y.reshape(-1)

    def precond(self, r):
        tau = 0.5 * self.cfg["dt"]

        def solve(k, z):
            S, H = self.blocks(k)
            return torch.linalg.solve(torch.complex(S, tau * H), z)

        return self.per_kappa(solve, r.reshape(len(self.ch), -1)).reshape(-1)

    def step(self, psi, t):
        """One Crank-Nicolson step, A_+ x = A_- psi at the midpoint, by preconditioned minimal
        residuals on the error until the residual is at rounding."""
        t = t + 0.5 * self.cfg["dt"]
        b = self.apply(-1, t, psi)
        x = psi.clone()
        for _ in range(60):
            r = b - self.apply(+1, t, x)
            if torch.linalg.norm(r) <= 2e-15 * torch.linalg.norm(b):
                break
            # GMRES(6) on the correction
            Z, Y = [], []
            q = r
            for _ in range(6):
                z = self.precond(q)
                y = self.apply(+1, t, z)
                for zp, yp in zip(Z, Y):
                    a = torch.vdot(yp, y)
                    y, z = y - a * yp, z - a * zp
                nrm = torch.linalg.norm(y)
                y, z = y / nrm, z / nrm
                a = torch.vdot(y, r)
                x, r = x + a * z, r - a * y
                Z.append(z)
                Y.append(y)
                q = r
                if torch.linalg.norm(r) <= 1e-16 * torch.linalg.norm(b):
                    break
        return x


def _exact_net(case, seed):
    """The network with its weights rounded to bfloat16, in 64 bits."""
    w = torch.from_numpy(W.guess_net_init(7)).to(DEV)
    shapes = [(32, 256), (256,), (256, 256), (256,), (256, 256), (256,), (256, 4), (4,)]
    parts, o = [], 0
    for s in shapes:
        v = w[o:o + math.prod(s)].reshape(s)
        o += math.prod(s)
        parts.append((v.bfloat16() if len(s) == 2 else v).double().requires_grad_(case["kind"] == "grad"))
    x, t = _net_batch(case["M"] if case["kind"] == "forward" else case["B"], seed)

    def net(z):
        for i in (0, 2, 4):
            z = torch.tanh(z @ parts[i] + parts[i + 1])
        return z @ parts[6] + parts[7]

    if case["kind"] == "forward":
        return torch.cat([net(z.double()) for z in x.split(1 << 17)])
    loss = (net(x.double()) - t.double()).square().sum() / case["B"]
    grad = torch.autograd.grad(loss, parts)
    return {"loss": loss.item(), "grad": torch.cat([g.reshape(-1) for g in grad])}


def _exact_spectrum(case, E, psi):
    v = psi.reshape(len(E.ch), -1)
    c2 = E.cfg["c"] ** 2
    grid = np.linspace(0.0, case["e_hi"], case["n_grid"])
    obs, dpde = dict(norm=0.0, energy=0.0, p_ground=0.0, p_bound=0.0), np.zeros_like(grid)
    for k, idx in E.groups():
        S, H = E.blocks(k)
        use = torch.from_numpy(E.used(k).reshape(-1)).to(DEV)
        S, H, z = S[use][:, use], H[use][:, use], v[torch.from_numpy(idx).to(DEV)][:, use].T
        # shift and invert, so that the levels near the shift (the bound and the low continuum states, out
        # of a spectrum that reaches 1e7) come out to rounding: L^T (H - sigma S)^-1 L y = y / (e - sigma)
        sigma = -0.0137
        L = torch.linalg.cholesky(S)
        M = L.T @ torch.linalg.solve(H - sigma * S, L)
        mu, y = torch.linalg.eigh(0.5 * (M + M.T))
        e, order = torch.sort(sigma + 1.0 / mu)
        q = (y[:, order].T.to(z.dtype) @ (L.T.to(z.dtype) @ z)).abs().square()   # |v_j^T S psi|^2, [level][channel]
        obs["norm"] += (z.conj() * (S.to(z.dtype) @ z)).sum().real.item()
        obs["energy"] += (z.conj() * (H.to(z.dtype) @ z)).sum().real.item()
        bound = (e > -c2) & (e < 0)
        obs["p_bound"] += q[bound].sum().item()
        if k == -1:
            obs["p_ground"] = q[bound][0, [E.ch[i][1] for i in idx].index(1)].item()
        sel = (e > 0) & (e <= case["e_hi"])
        lev, p = e[sel].cpu().numpy(), q[sel].sum(1).cpu().numpy()
        if len(lev) < 2:
            continue
        d = np.empty_like(lev)
        d[0], d[-1], d[1:-1] = lev[1] - lev[0], lev[-1] - lev[-2], 0.5 * (lev[2:] - lev[:-2])
        dpde += np.interp(grid, lev, p / d, left=0.0, right=0.0)
    return {"obs": obs, "dpde": dpde}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "grad"):
        return _exact_net(case, seed)
    if kind == "batch":
        return None
    nch, n1 = len(_channels(case["kmax"], case["two_mu_max"])), case["N"] + 1
    if kind == "run" and nch * n1 * case["steps"] > 40000:
        return None   # minutes
    s = prepare(case, seed)
    E = _Exact(_cfg(case))
    if kind == "run":
        i = s["insts"][0]
        psi, hist = i["psi"].clone(), [i["hist"][:E.n].clone(), i["hist"][E.n:].clone()]
        for q in range(case["steps"]):
            new = E.step(psi, i["t"] + q * E.cfg["dt"])
            psi, hist = new, [psi, hist[0]]
        return {"psi": psi, "hist": torch.cat(hist)}
    if kind == "residual":
        b = E.apply(-1, s["t"], s["psi"])
        return {"bnorm": torch.linalg.norm(b).item(), "r": b - E.apply(+1, s["t"], s["x"])}
    if kind in ("apply", "apply32"):
        return E.apply(s["sign"], s["t"], s["x"].to(torch.complex128))
    if kind == "precond":
        return E.precond(s["r"].to(torch.complex128))
    return _exact_spectrum(case, E, s["psi"])
