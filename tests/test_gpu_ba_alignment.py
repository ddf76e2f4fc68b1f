"""Bundle adjustment takes its arrays at any float's address: slices of a packed buffer that start at an odd
float give bit for bit what the same arrays give at the start of their own allocation."""
import pytest

from tests.test_gpu_ba import DELTA, SIGMA, _dev, _setup

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _packed(t):
    """t as a contiguous view one element into a buffer of its own."""
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    view = flat[1:].view(t.shape)
    view.copy_(t)
    assert view.is_contiguous() and view.data_ptr() % 8 == 4
    return view


@pytest.mark.parametrize("C,n", [(3, 40), (12, 700)])
def test_arrays_at_odd_floats(C, n):
    from paper_2601_17354_gb300 import ba as B
    p, obs, R, t, P = _setup(50 + C, C, n, False)
    ba = B.BundleAdjuster(C, n, len(obs[0]))
    dev = _dev(R, t, P, obs)
    odd = [_packed(x) for x in dev]
    for a, b in zip(ba.step(*dev, p.K, SIGMA, DELTA, 1e-3)[:2], ba.step(*odd, p.K, SIGMA, DELTA, 1e-3)[:2]):
        assert torch.equal(a, b)
    for args in (dev, odd):
        ba.solve(*args, p.K, SIGMA, DELTA, iters=2)
    for a, b in zip(dev[:3], odd[:3]):
        assert torch.equal(a, b)
