"""The preconditioner at every spline order beside the production order 7, against the oracle: orders up to 8
run the rotated-lane kernel, orders from 9 on, whose factors store more superdiagonals than a warp has lanes,
the shifting-window one.

Bars: complex128 1e-10, as test_gpu_parity.py states (a NumPy restatement of the sweeps on the library's own
blocks is within 2e-12 of a dense solve at every order).  complex64: the backward error of test_gpu_parity32.py
with kb = 2 order - 1.  Step: solved to 1e-12, the residual formed by the oracle's operator below 1e-11 (its own
and the apply's rounding, 1e-12 of the largest entry, beside the tolerance), at most twice the oracle's
iterations to 1e-14 plus 8."""
import math

import numpy as np
import pytest

from paper_2512_21697_gb300 import binding as B, layout, workloads as W

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


def _case(oracle_mod, order, **opt):
    cfg = dict(W.SMALL, order=order, N=40)
    bas = B.Basis(cfg)
    orc = oracle_mod.Oracle(**W.oracle_params(cfg))
    perm = layout.lib_to_paper_perm(bas.kappa, bas.two_mu, cfg["kappa_max"], cfg["two_mu_max"], cfg["N"])
    inv = np.empty_like(perm)
    inv[perm] = np.arange(len(perm))
    return cfg, bas, orc, perm, inv, B.Operator(bas, cfg, tol=1e-12, max_iter=300, **opt)


def _random(orc, seed):
    x = W.random_state(orc.n, seed)
    x[~orc.active_mask()] = 0
    return x / np.linalg.norm(x)


@pytest.mark.parametrize("order", [3, 4, 5, 6, 8, 9, 10, 11, 12])
def test_precond_at_every_order(oracle_mod, order):
    import torch
    cfg, bas, orc, perm, inv, op = _case(oracle_mod, order, precision=2, tol_inner=1e-5, max_outer=30)
    r = _random(orc, order)
    rd = torch.from_numpy(r[inv].copy()).cuda()
    zd = torch.empty_like(rd)
    op.precond(rd, zd)
    ref = orc.precond(r)
    assert np.linalg.norm(zd.cpu().numpy()[perm] - ref) <= 1e-10 * np.linalg.norm(ref)
    r32 = rd.to(torch.complex64)
    z32 = torch.empty_like(r32)
    op.precond32(r32, z32)
    z = z32.cpu().numpy().astype(np.complex128)[perm]
    r = r32.cpu().numpy().astype(np.complex128)[perm]
    size = lambda v: np.abs(v.real) + np.abs(v.imag)   # noqa: E731
    for c, kappa in enumerate(orc.kappa):
        S, H = orc.radial(int(kappa))
        s = slice(c * orc.nb, (c + 1) * orc.nb)
        on = orc.active_mask()[s]
        M, zc, rc = (S + 0.5j * cfg["dt"] * H)[np.ix_(on, on)], z[s][on], r[s][on]
        bound = 8 * (2 * (2 * order - 1) + 1) * U32 * (size(M) @ size(zc) + size(rc)).max()
        assert np.abs(M @ zc - rc).max() <= bound, int(kappa)


@pytest.mark.parametrize("order", [4, 8, 9, 12])
def test_fp64_step_at_other_orders(oracle_mod, order):
    import torch
    cfg, bas, orc, perm, inv, op = _case(oracle_mod, order)
    psi = _random(orc, 40 + order)
    t0 = 0.5 * cfg["n_cycles"] * 2 * math.pi / cfg["omega"]
    pd = torch.from_numpy(psi[inv].copy()).cuda()
    its, res, _ = op.step(pd, 1, t0)
    assert res[0] <= 1e-12
    x, tm = pd.cpu().numpy()[perm], t0 + 0.5 * cfg["dt"]
    b = orc.apply(tm, -1, psi)
    assert np.linalg.norm(orc.apply(tm, +1, x) - b) <= 1e-11 * np.linalg.norm(b)
    assert its[0] <= 2 * orc.step(psi, t0, tol=1e-14)[1] + 8
