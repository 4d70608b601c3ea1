"""Gradient of the initial-guess network at batches above 32768 samples, where the partials are 1024 samples long
and their number grows.  Bars: random samples as test_gpu_guess.py's test_loss_and_gradient_match_oracle states
for FP32 sums.  Equal samples, whose terms round the same way each time, give the gradient of one within the
roundings of 1024 + 1024 additions and of three layers' 256-term sums (32 partials of 32768 samples miss
it by 2.5e-4 on average)."""
import numpy as np
import pytest

from oracle import guess_net as G
from paper_2512_21697_gb300 import binding as B
from test_gpu_guess import _net_and_batch

pytestmark = pytest.mark.gpu


def _check(net, p, x, t, xd, td, bar):
    loss, grad = net.loss_grad(xd, td)
    ref, gr = G.loss_and_grads(p, x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - ref) <= 1e-5 * ref
    gflat = G.flatten(gr).astype(np.float64)
    o = 0
    for name, shp in G.SHAPES:
        n = int(np.prod(shp))
        a, b = grad[o:o + n], gflat[o:o + n]
        assert np.linalg.norm(a - b) <= bar * np.linalg.norm(b), name
        o += n


@pytest.mark.parametrize("n", [32768, 32769, 33793])
def test_random_samples_at_the_partials_limit(n):
    _, p, x, t, xd, td = _net_and_batch(n, 32)
    _check(B.GuessNet(n, G.flatten(p)), p, x, t, xd, td, 1e-4)


def test_equal_samples():
    n = 1 << 20
    _, p, x, t, xd, td = _net_and_batch(1, 33)
    _check(B.GuessNet(n, G.flatten(p)), p, x, t, xd.expand(n, 32).contiguous(), td.expand(n, 4).contiguous(),
           (2048 + 768) * 2.0 ** -24)
