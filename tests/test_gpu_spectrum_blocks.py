"""The spectrum at kappa counts on both sides of the grid kernel's 16 kappas per block, with level counts that
are not multiples of the four vectors a warp projects on, and ragged grid sizes, against the oracle (bar: as
test_gpu_spectrum.py's random state)."""
import numpy as np
import pytest

from paper_2512_21697_gb300 import binding as B, workloads as W
from test_gpu_spectrum import _setup, _window_clear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kmax,n_grid", [(1, 1), (8, 15), (9, 17), (17, 333)])
def test_spectrum_at_block_edges(kmax, n_grid):
    import torch
    cfg = dict(W.SMALL, kappa_max=kmax, two_mu_max=1, N=40)
    bas, orc, perm, inv = _setup(cfg)
    x = W.random_state(orc.n, 22)
    x[~orc.active_mask()] = 0
    x /= np.linalg.norm(x)
    _window_clear(orc, 0.0, 50.0)
    grid = np.linspace(0.7, 45.0, n_grid)
    op = B.Operator(bas, cfg, tol=1e-12)
    got, _ = op.spectrum(torch.from_numpy(x[inv].copy()).cuda(), 0.0, 50.0, grid)
    ref = orc.spectrum(x, 0.0, 50.0, grid)
    assert np.max(np.abs(got - ref)) <= 1e-9 * np.max(np.abs(ref))
