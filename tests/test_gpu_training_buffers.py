"""GPU: the training entry points on caller buffers that are aligned to their floats only (views that start one
element into an allocation): losses and gradients are those of aligned buffers, bit by bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _offset(t):
    """A copy of t that starts one float into its allocation."""
    buf = torch.empty(t.numel() + 1, device=t.device)
    buf[1:] = t.reshape(-1)
    return buf[1:]


@pytest.mark.parametrize("which", ["x", "target", "sigma"])
def test_gradients_from_buffers_at_odd_floats(which):
    from paper_2406_06640_gb300.binding import UNet

    dev, S, C, B = "cuda:0", 32, 16, 8
    gen = torch.Generator(device=dev).manual_seed(5)
    bufs = dict(x=torch.rand(B, S, S, generator=gen, device=dev),
                target=torch.rand(B, S // 2, S // 2, 2, generator=gen, device=dev),
                sigma=torch.rand(B, generator=gen, device=dev))
    results = []
    for case in (bufs, dict(bufs, **{which: _offset(bufs[which])})):
        net = UNet(S, C, B, seed=1)
        grads = np.empty(net.param_count(), np.float32)
        loss = net.gradients(case["x"].data_ptr(), case["target"].data_ptr(), case["sigma"].data_ptr(), 0.1, grads)
        results.append((loss, grads))
        net.close()
    assert results[0][0] == results[1][0] and np.isfinite(results[0][0])
    assert np.array_equal(results[0][1], results[1][1])
