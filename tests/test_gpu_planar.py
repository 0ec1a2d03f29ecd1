"""Boxes of one layer: the off-diagonal components between the layer and its normal vanish, so dipoles along
the normal give no field in the layer, and dipoles in the layer none along the normal, exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("box", [(9, 7, 1), (20, 33, 1), (15, 1, 12), (1, 14, 9), (1, 1, 40)])
def test_layer_and_normal_decouple(box):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda as D

    z, y, x = np.meshgrid(*(np.arange(b) for b in box[::-1]), indexing="ij")
    ctx = D.Context(0)
    ctx.dda_setup_target(np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.int32))
    ctx.dda_set_incident(0.7, [(0.3, 1.1, 2.0)])
    ctx.dda_build_green_fft()
    ctx.dda_set_polarizability("GKDLDR", 1.5 + 0.1j)
    gen = torch.Generator(device="cuda").manual_seed(sum(box))
    for dt in (torch.complex64, torch.complex128):
        for along in range(3):
            p = torch.zeros((ctx.nrhs, 3, ctx.n), dtype=dt, device="cuda")
            p[:, along] = torch.randn((ctx.nrhs, ctx.n), dtype=dt, device="cuda", generator=gen)
            ap = torch.empty_like(p)
            ctx.dda_matvec(p, ap)
            for a in range(3):
                # every offset has n_a n_along = 0 where one of the two axes has a single layer
                if a != along and 1 in (box[a], box[along]):
                    assert (ap[:, a] == 0).all(), (dt, along, a)
