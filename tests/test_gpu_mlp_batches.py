"""The surrogate at the batch sizes it takes, multiples of 128 (GPU): gradients and forward pass of
one 128-row tile, odd numbers of them (odd splits of the weight-gradient products), a full
training batch; smaller batches in the buffers of larger ones."""
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


@pytest.mark.parametrize("B", [128, 1408])
def test_weight_gradients_of_the_last_outputs(net, B):  # noqa: F811
    """dW3 has 450 rows, the product's last 128-row tile 512: one warp of it holds rows on both
    sides of the end.  Row by row, so that two wrong rows do not hide in the norm of 450; a row
    is a sum over B samples in which a bf16 flip moves one term by 2^-8, 2^-8 / sqrt(B) of the
    row each (4e-4 at B = 128), a few per row."""
    import paper_2605_26347_gb300 as pkg
    s, p = net
    x, t = batch(B, B + 1)
    _, ref = omlp.loss_and_grads(p, x.astype(np.float64), t.astype(np.float64), bf=True)
    g = pkg.unpack_params(s.gradients(x, t)[1])["W3"]
    for j in range(384, 450):
        assert rel(g[j], ref["W3"][j]) < 2e-3, (j, rel(g[j], ref["W3"][j]))


@pytest.mark.parametrize("sizes", [(128, 384, 1408), (4096, 128, 1408)])
def test_forward_of_any_batch(sizes):
    """The forward pass alone (no transposed activations), in growing buffers and in those of a larger
    batch and of its gradients; bf16 flips as in test_gpu_surrogate."""
    import paper_2605_26347_gb300 as pkg
    s = pkg.Surrogate(seed=0)
    p = {k: v.astype(np.float64) for k, v in pkg.unpack_params(s.get_params()).items()}
    for B in sizes:
        x, t = batch(B, B + 2)
        y = s.forward(x).cpu().numpy().astype(np.float64)
        assert rel(y, omlp.forward(p, x.astype(np.float64), bf=True)["y"]) < 1e-3, B
        s.gradients(x, t)
