"""The workspace of the products with the angular sums first, where the steps keep the stored coupling values:
an operator that only steps holds none of it, the first single product sets it up, and a captured stream or a
device without room leaves the product in the steps' form, with the steps' results."""
import math

import numpy as np
import pytest

from paper_2512_21697_gb300 import binding as B, workloads as W

pytestmark = pytest.mark.gpu

# 840 channels, 256 slots, three multipoles: the angular sums alone take 66 MB
CFG = dict(W.PRODUCTION, N=255, n_lin=126, kappa_max=20, l_max=2, E0=0.2)
SUMS = 840 * 18 * 256 * 16


def _op(stream=None):
    bas = B.Basis(CFG)
    return bas, B.Operator(bas, CFG, stream=stream, tol=1e-10, precision=2, tol_inner=1e-5, max_outer=20)


def _vectors(bas, seed):
    import torch
    psi = torch.from_numpy(W.random_state(bas.n, seed)).cuda()
    t = 0.4 * CFG["n_cycles"] * 2 * math.pi / CFG["omega"]
    torch.cuda.synchronize()
    return t, psi, torch.empty_like(psi)


def test_only_single_products_take_the_workspace():
    import torch
    bas, op = _op()
    t, psi, y = _vectors(bas, 71)
    held = op.device_bytes()
    hist = torch.zeros(2 * bas.n, dtype=torch.complex128, device="cuda")
    state = torch.from_numpy(bas.initial_state()[0]).cuda()
    op.set_overlap(True)   # the second set of coupling values
    two_sets = op.device_bytes()
    op.step(state, 2, t, hist=hist)
    op.run(state, 1, t, hist)
    op.set_call_form(True)
    op.residual(t, psi, psi, y)
    assert op.device_bytes() == two_sets and op.form("residual") == "owner"
    op.set_call_form(False)
    for call in (lambda: op.residual(t, psi, psi, y), lambda: op.apply(+1, t, psi, y),
                 lambda: op.step(state, 2, t, hist=hist), lambda: op.residual(t, psi, psi, y)):
        call()   # in either buffer set
    assert op.form("residual") == "angular"
    assert SUMS <= op.device_bytes() - two_sets <= 0.25 * held


def test_captured_product_allocates_nothing():
    import torch
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    bas, op = _op(s)
    t, psi, y = _vectors(bas, 72)
    held = op.device_bytes()
    op.set_call_form(True)
    op.apply(+1, t, psi, y)
    torch.cuda.synchronize()
    ref, z = y.clone(), torch.zeros_like(y)
    op.set_call_form(False)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        op.apply(+1, t, psi, z)
    assert op.device_bytes() == held and op.form("apply") == "rows"
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(z, ref)
    # set up while another stream is captured: that capture stays valid
    g2, w = torch.cuda.CUDAGraph(), torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.graph(g2, stream=other):
        w.add_(1.0)
        op.apply(+1, t, psi, z)
    g2.replay()
    torch.cuda.synchronize()
    assert torch.equal(w, torch.ones_like(w))
    assert op.form("apply") == "angular" and op.device_bytes() - held >= SUMS
    assert torch.linalg.norm(z - ref) <= 1e-11 * torch.linalg.norm(ref)


def test_without_room_the_product_keeps_the_steps_form():
    import torch
    bas, op = _op()
    t, psi, y = _vectors(bas, 73)
    x32 = psi.to(torch.complex64)
    y32 = torch.empty_like(x32)
    op.set_call_form(True)
    op.residual(t, psi, 0.5 * psi, y)
    op.apply32(+1, t, x32, y32)
    ref, ref32, half = y.clone(), y32.clone(), 0.5 * psi
    op.set_call_form(False)
    held = op.device_bytes()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - SUMS // 2, dtype=torch.uint8, device="cuda")
    try:
        op.residual(t, psi, half, y)
        assert op.form("residual") == "owner" and op.device_bytes() == held
        op.apply32(+1, t, x32, y32)
        assert op.form("apply32") == "owner" and op.device_bytes() == held
    finally:
        del filler
        torch.cuda.empty_cache()
    assert torch.equal(y, ref) and torch.equal(y32, ref32)
    op.residual(t, psi, half, y)   # one form for the op's life
    assert torch.equal(y, ref) and np.isfinite(y.abs().max().item())
