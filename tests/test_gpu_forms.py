"""Each form of the products at production size against sampled rows of the oracle, the form that ran read
back from the library: the kernels that the steps run (owner and gather passes, subgroup form) as well as the
angular sums first, which single calls take by default.

Bars: as test_gpu_parity32.py states for its production rows -- complex64 (2 m + 8) u 4 max|y| for the stored
coupling, 64 times that for the factorised forms; double-float 1e-11 of the largest entry."""
import math

import numpy as np
import pytest

from paper_2512_21697_gb300 import binding as B, workloads as W
from test_gpu_parity32 import U32, _production

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def prod(oracle_mod):
    cfg, bas, orc, perm, inv, rows, T, torch = _production(oracle_mod)
    op = B.Operator(bas, cfg, tol=cfg["tol"], precision=2, tol_inner=1e-5, max_outer=20)
    t = 0.43 * T
    ch, idx = rows // orc.nb, rows % orc.nb
    psi, x = W.random_state(orc.n, 44), W.random_state(orc.n, 45)
    x = psi + 0.01 * x
    psi[~orc.active_mask()] = 0
    x[~orc.active_mask()] = 0
    x32 = x.astype(np.complex64)
    ref = {"b": orc.apply_rows(t, -1, psi, ch, idx), "ax": orc.apply_rows(t, +1, x, ch, idx)}
    for sign in (+1, -1):
        ref["y32", sign] = orc.apply_rows(t, sign, x32.astype(np.complex128), ch, idx)
    dev = {"psi": torch.from_numpy(psi[inv]).cuda(), "x": torch.from_numpy(x[inv]).cuda(),
           "x32": torch.from_numpy(x32[inv]).cuda()}
    m = 2 * 13 * (1 + int(np.bincount(orc.edges()[0]).max()))
    yield op, t, perm, rows, ref, dev, m
    op.set_call_form(False)
    op.set_factorised(0)


@pytest.mark.parametrize("as_steps,mode,form", [(True, 0, "owner"), (True, 1, "subgroup"), (False, 0, "angular"),
                                                (False, 1, "angular")])
def test_production_apply32_rows_in_each_form(prod, as_steps, mode, form):
    import torch
    op, t, perm, rows, ref, dev, m = prod
    op.set_call_form(as_steps)
    op.set_factorised(mode)
    bar = (1 if form == "owner" else 64) * (2 * m + 8) * U32 * 4
    for sign in (+1, -1):
        y = torch.empty_like(dev["x32"])
        op.apply32(sign, t, dev["x32"], y)
        assert op.form("apply32") == form
        yn = y.cpu().numpy().astype(np.complex128)[perm]
        assert np.abs(yn[rows] - ref["y32", sign]).max() <= bar * np.abs(yn).max(), sign


@pytest.mark.parametrize("as_steps,form", [(True, "owner"), (False, "angular")])
def test_production_residual_rows_in_each_form(prod, as_steps, form):
    import torch
    op, t, perm, rows, ref, dev, m = prod
    op.set_call_form(as_steps)
    scale = max(np.abs(ref["b"]).max(), np.abs(ref["ax"]).max())
    for mode in (0, 1, 2):   # automatic (the offsets at this tolerance), Dot2, offsets
        op.set_residual_mode(mode)
        r = torch.empty_like(dev["psi"])
        op.residual(t, dev["psi"], dev["x"], r)
        assert op.form("residual") == form
        assert np.abs(r.cpu().numpy()[perm][rows] - (ref["b"] - ref["ax"])).max() <= 1e-11 * scale, mode
    op.set_residual_mode(0)
    y = torch.empty_like(dev["psi"])
    op.apply(+1, t, dev["x"], y)
    assert op.form("apply") == ("rows" if as_steps else "angular")
    assert np.abs(y.cpu().numpy()[perm][rows] - ref["ax"]).max() <= 1e-11 * np.abs(ref["ax"]).max()


@pytest.mark.parametrize("precision,tol,resid,inner", [(0, 1e-10, "angular", None), (1, 1e-10, "split", "owner"),
                                                       (2, 1e-10, "owner", "owner"), (2, 1e-12, "angular", "angular")])
def test_steps_report_their_forms(precision, tol, resid, inner):
    # a system from which on the products are factorised; a single call in between changes nothing for the steps
    import torch
    cfg = dict(W.PRODUCTION, N=255, n_lin=126, kappa_max=20, l_max=2, E0=0.2)
    bas = B.Basis(cfg)
    op = B.Operator(bas, cfg, tol=tol, precision=precision, max_iter=500, tol_inner=1e-5, max_outer=20)
    psi = torch.from_numpy(bas.initial_state()[0]).cuda()
    y, hist = torch.empty_like(psi), torch.zeros(2 * bas.n, dtype=torch.complex128, device="cuda")
    t = 0.4 * cfg["n_cycles"] * 2 * math.pi / cfg["omega"]
    for drive in (lambda: op.step(psi, 1, t, hist=hist), lambda: op.run(psi, 1, t, hist)):
        op.apply(+1, t, psi, y)
        if precision != 1:
            assert op.form("apply") == "angular"
        drive()
        assert op.form("residual") == resid and op.form("apply32") == inner
    op.set_call_form(True)
    op.residual(t, psi, psi, y)
    assert op.form("residual") == resid and op.form("apply32") == inner
    with pytest.raises(B.DiracError):
        op.set_call_form(2)
