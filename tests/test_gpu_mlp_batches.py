"""Gradients of the surrogate at batch sizes around its tiles (GPU): one 128-row tile, odd
numbers of them (odd splits of the weight-gradient products), a full training batch."""
import numpy as np
import pytest

from oracle import mlp as omlp
from test_gpu_surrogate import batch, net, rel  # noqa: F401  (net is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [128, 384, 1408, 4096])
def test_gradients_of_any_batch(net, B):  # noqa: F811
    import paper_2605_26347_gb300 as pkg
    s, p = net
    x, t = batch(B, B)
    ref_loss, ref = omlp.loss_and_grads(p, x.astype(np.float64), t.astype(np.float64), bf=True)
    for _ in range(2):  # the second call reuses the buffers of the first
        loss, g = s.gradients(x, t)
        assert abs(loss - ref_loss) < 1e-4 * ref_loss
        gd = pkg.unpack_params(g)
        for k in ("W3", "b3", "W2", "b2", "W1", "b1"):
            assert rel(gd[k], ref[k]) < 2e-3, (k, rel(gd[k], ref[k]))  # bf16 flips, as in test_gpu_surrogate
