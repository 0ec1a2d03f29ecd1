"""Tiles of the network's convolutions and weight gradients at their edges: rows longer than one x tile,
rows that the tiles do not divide, the deepest level down to one voxel, one and several samples; forward pass and every layer's weight and bias gradient against the oracle (oracle/unet.py,
with the kernels' bfloat16 rounding points)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import unet as OU  # noqa: E402


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda
    return dda


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# dims x, y, z; batch; channels
CASES = [((40, 8, 8), 1, (6, 10, 12, 16)), ((72, 16, 8), 1, (6, 10, 12, 16)), ((8, 8, 8), 3, (6, 10, 12, 16)),
         ((16, 8, 24), 2, (12, 24, 32, 48))]


@pytest.mark.parametrize("dims,batch,ch", CASES)
def test_forward_and_gradients(D, dims, batch, ch):
    cin, cout = 9, 6
    net = D.UNet(0, None, cin, cout, ch, seed=sum(dims))
    theta = net.dda_unet_get_params().astype(np.float64)
    rng = np.random.default_rng(dims[0] + batch)
    shape = (batch, dims[2], dims[1], dims[0])
    x = rng.standard_normal(shape + (cin,)).astype(np.float32)
    t = rng.standard_normal(shape + (cout,)).astype(np.float32)
    mask = (rng.random(shape) > 0.3).astype(np.float32)
    y = torch.empty(shape + (cout,), device="cuda")
    net.dda_unet_forward(torch.from_numpy(x).cuda(), y, dims)
    ref = OU.forward(theta, x.astype(np.float64), cin, cout, ch, quant=True)
    # bfloat16 rounding decisions on FP32 against FP64 activations: the bars of the network's other tests
    assert _rel(y.cpu().numpy(), ref) <= 5e-3
    loss = net.dda_unet_loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(),
                                  torch.from_numpy(mask).cuda(), dims)
    g = net.dda_unet_get_params(which=1).astype(np.float64)
    lr, gr = OU.loss_and_grad(theta, x.astype(np.float64), t.astype(np.float64), mask.astype(np.float64), cin, cout,
                              ch, quant=True)
    assert loss == pytest.approx(lr, rel=1e-4)
    o = 0
    for taps, a, b in OU.layer_shapes(cin, cout, ch):
        nw = taps * a * b
        assert _rel(g[o:o + nw], gr[o:o + nw]) <= 2e-2, ("W", o)
        assert _rel(g[o + nw:o + nw + b], gr[o + nw:o + nw + b]) <= 2e-2, ("b", o)
        o += nw + b
