"""Loss and gradient of the initial-guess network at batch sizes on both sides of the gradient kernel's
sample chunks (32 rows staged at a time, 32 partials of 32, 64, .. samples), against the NumPy oracle.  Bars: as
test_gpu_guess.py's test_loss_and_gradient_match_oracle states for FP32 sums."""
import numpy as np
import pytest

from oracle import guess_net as G
from test_gpu_guess import _net_and_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 32, 33, 63, 65, 1024, 1025, 2049])
def test_gradient_at_chunk_edges(B):
    net, p, x, t, xd, td = _net_and_batch(B, 31)
    loss, grad = net.loss_grad(xd, td)
    lr_, gr = G.loss_and_grads(p, x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - lr_) <= 1e-5 * lr_
    gflat = G.flatten(gr).astype(np.float64)
    o = 0
    for name, shp in G.SHAPES:
        n = int(np.prod(shp))
        a, b = grad[o:o + n], gflat[o:o + n]
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b) + 1e-9, name
        o += n
