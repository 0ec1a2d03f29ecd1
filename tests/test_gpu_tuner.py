"""What the first product of a grid costs: a configuration is tried with at most one warm-up product, four
timed ones and three more when it is close to the best, of which a grid has about ten."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("box,pad", [((64, 48, 32), (128, 96, 64)), ((40, 40, 40), (80, 80, 80))])
def test_first_product_makes_few_products(box, pad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda as D

    z, y, x = np.meshgrid(*(np.arange(b) for b in box[::-1]), indexing="ij")
    ctx = D.Context(0)
    ctx.dda_setup_target(np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.int32))
    ctx.dda_set_incident(0.3, [(0.3, 1.1, 2.0)])
    ctx.dda_build_green_fft(pad)
    ctx.dda_set_polarizability("GKDLDR", 1.5 + 0.1j)
    p = torch.randn((ctx.nrhs, 3, ctx.n), dtype=torch.complex64, device="cuda")
    ap = torch.empty_like(p)
    before = D.LIB.dda_kernel_launches()
    ctx.dda_matvec(p, ap)
    first = D.LIB.dda_kernel_launches() - before
    before = D.LIB.dda_kernel_launches()
    ctx.dda_matvec(p, ap)
    each = D.LIB.dda_kernel_launches() - before
    assert each in (3, 5)
    # twelve configurations, eight products each, most of them of three launches
    assert first <= 300, first
