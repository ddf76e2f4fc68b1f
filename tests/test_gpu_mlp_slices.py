"""The initializer's MLP at the sizes where its slices end: 16-point fragments of the forward pass, 64-point
slices of a training step (a lone point, ragged last slices, CTAs that take several slices), against the
initializer oracle.  Tolerances are the BF16 ones of test_gpu_init.py: activations may differ by one BF16
unit where FP32 sums differ in their last bits."""
import numpy as np
import pytest

import oracle
from tests._parity import rel_l2
from tests.test_gpu_init import _mlp_with_random_weights

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 200, 19457, 45007])
def test_forward_and_gradients(n):
    from paper_2601_17354_gb300 import initializer as I
    mlp, ws = _mlp_with_random_weights(I, I.Initializer(), n)
    rng = np.random.default_rng(n)
    x = rng.normal(size=(n, 16)).astype(np.float32)
    x[:: 7] *= 6.0  # activations into both saturated tails
    t = rng.normal(size=(n, 8)).astype(np.float32)
    t[:, 3:7] /= np.linalg.norm(t[:, 3:7], axis=1, keepdims=True)
    xb = torch.from_numpy(x).cuda().bfloat16()
    xr = xb.float().cpu().numpy()
    y = oracle.mlp_forward(xr, ws, mode=1)
    assert rel_l2(mlp.forward(xb).cpu().numpy(), y) < 5e-3
    mlp.loss_sum.zero_()
    mlp.grad.zero_()
    mlp.accumulate_grad(xb, torch.from_numpy(t).cuda())
    loss, dy = oracle.init_loss(y, t)
    assert abs(mlp.loss_sum.item() / n - loss) <= 1e-3 * loss
    got, off = mlp.grad.cpu().numpy(), 0
    for w in oracle.mlp_backward(xr, ws, dy, mode=1):
        assert rel_l2(got[off:off + w.size], w.reshape(-1)) < 2e-2, off
        off += w.size
