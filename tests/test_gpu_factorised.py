"""The factorised products (angular sums first, csrc/kernels_ang.cu) at system sizes where the library
takes them, with radial sizes at the edges of the row tiles (32 and 64 slots of the radial pass, 128
positions of the angular pass) and one to four multipoles, against rows of the oracle's FP64 operator.

Bars: as test_gpu_parity32.py states for the production rows -- complex64 normwise
64 (2 m + 8) u 4 max|y| with m = 2 x 13 x (1 + partners); double-float residual and apply 1e-11 of the
largest entry; FP64 1e-12 of max|y| (sums of about 10^3 terms in another order)."""
import math

import numpy as np
import pytest

from paper_2512_21697_gb300 import binding as B, layout, workloads as W

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


def _case(oracle_mod, kmax, N, lmax, seed):
    m = N + 5 - 7
    cfg = dict(W.PRODUCTION, N=N, n_lin=m // 2, kappa_max=kmax, l_max=lmax, E0=0.2)
    bas = B.Basis(cfg)
    orc = oracle_mod.Oracle(**W.oracle_params(cfg))
    perm = layout.lib_to_paper_perm(bas.kappa, bas.two_mu, kmax, 0, N)
    inv = np.empty_like(perm)
    inv[perm] = np.arange(len(perm))
    g = np.random.default_rng(seed)
    # the paper's order within a channel: type 0 slots, then type 1 slots; slots at the tile edges and the ends
    slots = np.unique(np.clip([0, 1, 5, 6, 31, 32, 63, 64, 119, 120, 127, 128, N - 6, N - 1, N], 0, N))
    ch = g.choice(orc.nch, 6, replace=False)
    rows = np.concatenate([[c * orc.nb + s, c * orc.nb + N + 1 + s] for c in ch for s in slots])
    psi = W.random_state(orc.n, seed)
    psi[~orc.active_mask()] = 0
    return cfg, bas, orc, perm, inv, rows, psi / np.linalg.norm(psi)


# (kappa_max, N, l_max): radial slots N + 1 = 50 (one ragged 64-slot tile, two of 32), 128 (whole tiles),
# 129 (one slot over), 256 + 1
@pytest.mark.parametrize("kmax,N,lmax", [(30, 49, 2), (20, 127, 3), (20, 128, 1), (14, 256, 2)])
def test_mixed_products_match_oracle_rows(oracle_mod, kmax, N, lmax):
    import torch
    cfg, bas, orc, perm, inv, rows, psi = _case(oracle_mod, kmax, N, lmax, 61)
    x = psi + 0.01 * _case(oracle_mod, kmax, N, lmax, 62)[6]
    T = cfg["n_cycles"] * 2 * math.pi / cfg["omega"]
    t = 0.43 * T
    ch, idx = rows // orc.nb, rows % orc.nb
    op = B.Operator(bas, cfg, tol=1e-10, precision=2, tol_inner=1e-5, max_outer=20)
    pd, xd = torch.from_numpy(psi[inv]).cuda(), torch.from_numpy(x[inv]).cuda()
    m = 2 * 13 * (1 + int(np.bincount(orc.edges()[0]).max()))
    x32 = xd.to(torch.complex64)
    xr = x32.cpu().numpy().astype(np.complex128)[perm]
    y32 = {}
    for mode in (0, 1):
        op.set_factorised(mode)
        for sign in (+1, -1):
            y = torch.empty_like(x32)
            op.apply32(sign, t, x32, y)
            y32[mode, sign] = y
            yn = y.cpu().numpy().astype(np.complex128)[perm]
            ref = orc.apply_rows(t, sign, xr, ch, idx)
            assert np.abs(yn[rows] - ref).max() <= 64 * (2 * m + 8) * U32 * 4 * np.abs(yn).max()
            assert np.all(yn[~orc.active_mask()] == 0)
    assert torch.equal(y32[0, 1], y32[1, 1]) and torch.equal(y32[0, -1], y32[1, -1])
    b, ax = orc.apply_rows(t, -1, psi, ch, idx), orc.apply_rows(t, +1, x, ch, idx)
    scale = max(np.abs(b).max(), np.abs(ax).max())
    for mode in (1, 2):
        op.set_residual_mode(mode)
        r = torch.empty_like(pd)
        bn = op.residual(t, pd, xd, r)
        assert np.abs(r.cpu().numpy()[perm][rows] - (b - ax)).max() <= 1e-11 * scale, mode
        y = torch.empty_like(pd)
        op.apply_assembled(-1, pd, y)   # the band entries of the residual's time
        assert np.abs(y.cpu().numpy()[perm][rows] - b).max() <= 1e-11 * np.abs(b).max()
        assert abs(bn - torch.linalg.norm(y).item()) <= 1e-6 * bn


# ||b|| of the factorised residual: psi rounded to nearest.  Truncated words are low by 2^-24 of a word's leading
# bit, uniform, so by 2^-25 / mean leading fraction = 4.3e-8 on average, which is all of the bar.
@pytest.mark.parametrize("kmax,N,lmax", [(20, 128, 1), (14, 256, 2)])
def test_mixed_bnorm_has_no_truncation_bias(oracle_mod, kmax, N, lmax):
    import torch
    cfg, bas, orc, perm, inv, rows, psi = _case(oracle_mod, kmax, N, lmax, 65)
    op = B.Operator(bas, cfg, tol=1e-10, precision=2, tol_inner=1e-5, max_outer=20)
    pd = torch.from_numpy(psi[inv]).cuda()
    t = 0.43 * cfg["n_cycles"] * 2 * math.pi / cfg["omega"]
    r, y = torch.empty_like(pd), torch.empty_like(pd)
    bn = op.residual(t, pd, pd, r)
    op.apply(-1, t, pd, y)
    assert abs(bn - torch.linalg.norm(y).item()) <= 4.3e-8 * bn


# sizes where the FP64 products are factorised too (precision 0), beside the stored ones of precision 1
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kmax,N,lmax", [(30, 96, 2), (20, 255, 2)])
def test_fp64_products_match_oracle_rows(oracle_mod, kmax, N, lmax, precision):
    import torch
    cfg, bas, orc, perm, inv, rows, psi = _case(oracle_mod, kmax, N, lmax, 63)
    t = 0.57 * cfg["n_cycles"] * 2 * math.pi / cfg["omega"]
    ch, idx = rows // orc.nb, rows % orc.nb
    op = B.Operator(bas, cfg, tol=1e-10, precision=precision, tol_inner=1e-5, max_outer=20)
    xd = torch.from_numpy(psi[inv]).cuda()
    y = torch.empty_like(xd)
    for sign in (+1, -1):
        op.apply(sign, t, xd, y)
        yn = y.cpu().numpy()[perm]
        assert np.abs(yn[rows] - orc.apply_rows(t, sign, psi, ch, idx)).max() <= 1e-12 * np.abs(yn).max()
        assert np.all(yn[~orc.active_mask()] == 0)
    if precision == 1:
        m = 2 * 13 * (1 + int(np.bincount(orc.edges()[0]).max()))
        x32 = xd.to(torch.complex64)
        y32 = torch.empty_like(x32)
        op.apply32(+1, t, x32, y32)
        yn = y32.cpu().numpy().astype(np.complex128)[perm]
        ref = orc.apply_rows(t, +1, x32.cpu().numpy().astype(np.complex128)[perm], ch, idx)
        assert np.abs(yn[rows] - ref).max() <= 64 * (2 * m + 8) * U32 * 4 * np.abs(yn).max()


# stored FP64 products: the kernel split over the partners (radial slots at the edges of its 8-row blocks, the
# largest grid) and the row kernel above
@pytest.mark.parametrize("kmax,N,lmax", [(3, 40, 1), (4, 47, 2), (4, 48, 2), (30, 135, 1), (30, 143, 1)])
def test_stored_fp64_product_matches_oracle_rows(oracle_mod, kmax, N, lmax):
    import torch
    cfg, bas, orc, perm, inv, rows, psi = _case(oracle_mod, kmax, N, lmax, 64)
    t = 0.57 * cfg["n_cycles"] * 2 * math.pi / cfg["omega"]
    ch, idx = rows // orc.nb, rows % orc.nb
    op = B.Operator(bas, cfg, tol=1e-10, precision=1, tol_inner=1e-5, max_outer=20)
    xd = torch.from_numpy(psi[inv]).cuda()
    y = torch.empty_like(xd)
    ys = {}
    for sign in (+1, -1):
        op.apply(sign, t, xd, y)
        yn = ys[sign] = y.cpu().numpy()[perm]
        assert np.abs(yn[rows] - orc.apply_rows(t, sign, psi, ch, idx)).max() <= 1e-12 * np.abs(yn).max()
        assert np.all(yn[~orc.active_mask()] == 0)
    # the residual's epilogues: r = b - A_+ x and ||b||
    r = torch.empty_like(xd)
    bn = op.residual(t, xd, xd, r)
    scale = max(np.abs(ys[1]).max(), np.abs(ys[-1]).max())
    assert np.abs(r.cpu().numpy()[perm] - (ys[-1] - ys[1])).max() <= 1e-12 * scale
    assert abs(bn - np.linalg.norm(ys[-1])) <= 1e-12 * bn


@pytest.mark.parametrize("precision,tol", [(0, 1e-10), (1, 1e-10), (2, 1e-10), (2, 1e-12)])
def test_drivers_agree_and_modes_switch(precision, tol):
    # host loop, overlapped assembly, captured driver: the same arithmetic, bit for bit, with single
    # products (whose form may be another) in between; precision 2 also through the per-channel form and
    # back (captured graphs are rebuilt)
    import torch
    cfg = dict(W.PRODUCTION, N=255, n_lin=126, kappa_max=20, l_max=2, E0=0.2)
    bas = B.Basis(cfg)
    op = B.Operator(bas, cfg, tol=tol, precision=precision, max_iter=500, tol_inner=1e-5, max_outer=20)
    psi0 = torch.from_numpy(bas.initial_state()[0]).cuda()
    t0 = 0.5 * cfg["n_cycles"] * 2 * math.pi / cfg["omega"]
    y = torch.empty_like(psi0)

    def steps(f):
        psi, hist = psi0.clone(), torch.zeros(2 * bas.n, dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        _, res, _ = f(psi, 3, t0, hist=hist)
        assert max(res) <= tol
        op.apply(+1, t0, psi, y)
        z = torch.empty_like(y)
        op.apply_assembled(+1, psi, z)
        assert torch.equal(y, z)
        return psi

    a = steps(op.step)
    assert torch.equal(a, steps(op.run))
    if precision == 2:
        op.set_overlap(True)
        assert torch.equal(a, steps(op.step))
        op.set_overlap(False)
        op.set_factorised(2)
        c = steps(op.run)
        assert torch.linalg.norm(c - a) <= 1e-9 * torch.linalg.norm(a)
        op.set_factorised(1)
        d = steps(op.run)
        assert torch.linalg.norm(d - a) <= 1e-9 * torch.linalg.norm(a)
        op.set_factorised(0)
        assert torch.equal(a, steps(op.run))
