"""The rotated-lane preconditioner (csrc/kernels_t.cu, k_precond_rot) against the shifting-window one at
radial sizes on both sides of its 16- and 32-row chunks, with 16 lanes per channel (interchanges of at most
two rows) and with 32 (a step size at which they reach four).  The operations and their order are the same:
bit for bit."""
import numpy as np
import pytest

from paper_2512_21697_gb300 import binding as B, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [0.005, 10.0])
@pytest.mark.parametrize("N,kmax,mu", [(23, 2, 0), (24, 3, 1), (31, 1, 0), (32, 4, 1), (47, 2, 0), (60, 5, 0)])
def test_rotated_lanes_equal_shifting_window(N, kmax, mu, dt):
    import torch
    cfg = dict(W.PRODUCTION, R=50.0, N=N, grid=0, r_lin=0.0, n_lin=0, kappa_max=kmax, two_mu_max=mu, l_max=2, dt=dt)
    bas = B.Basis(cfg)
    op = B.Operator(bas, cfg, tol=1e-10, precision=2, tol_inner=1e-5, max_outer=20)
    g = np.random.default_rng(N)
    r = torch.from_numpy(g.standard_normal(bas.n) + 1j * g.standard_normal(bas.n)).cuda()
    for single in (False, True):
        x = r.to(torch.complex64) if single else r
        z = {}
        for sched in (1, 3):
            op.set_schedule(single, sched)
            z[sched] = torch.empty_like(x)
            (op.precond32 if single else op.precond)(x, z[sched])
        torch.cuda.synchronize()
        assert torch.isfinite(torch.view_as_real(z[1])).all()
        assert torch.equal(z[1], z[3])
