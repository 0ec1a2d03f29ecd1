"""Bias gradients are sums over all voxels held in no fewer bits than FP64: output gradients whose sums FP64
adds without rounding (partial sums of 53 bits) have to come out exactly, after cancelling almost entirely."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cout", [64, 27, 6])
def test_head_bias_gradient_is_exact(cout):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda as D

    dims, nvox = (32, 32, 16), 32 * 32 * 16
    net = D.UNet(0, None, 9, cout, (8, 8, 8, 8), seed=1)
    rng = np.random.default_rng(cout)
    # in units of 2^-46: a sixteenth of the voxels near 1 with either sign, the rest near 2^-25
    big = (rng.integers(1 << 23, 1 << 24, (nvox, cout)) << 23) * rng.choice([-1, 1], (nvox, cout))
    first = np.where(rng.random((nvox, cout)) < 1 / 16, big, rng.integers(1 << 21, 1 << 22, (nvox, cout)))
    second = -rng.permuted(first, axis=0)
    small = np.argmin(np.abs(second), axis=0)
    second[small, np.arange(cout)] += 1 + 5 * np.arange(cout)
    g = np.stack([first, second])
    want = g.sum(axis=(0, 1)) * 2.0 ** -46
    assert np.array_equal(want, (1 + 5 * np.arange(cout)) * 2.0 ** -46)
    gy = torch.from_numpy((g * 2.0 ** -46).astype(np.float32)).cuda()
    assert np.array_equal(gy.cpu().numpy().astype(float), g * 2.0 ** -46)
    x = torch.randn((2, nvox, 9), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    y = torch.empty((2, nvox, cout), device="cuda")
    net.dda_unet_forward_train(x, y, dims)
    net.dda_unet_backward(gy, dims)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(np.asarray(net.dda_unet_get_params(1))[-cout:], want.astype(np.float32))
