"""The interaction tensor built from paired parities against the oracle's direct sum: lengths of one to four
radices in different orders (frequency -k then lies elsewhere in the storage order), axes of a single
layer, lengths far beyond twice the box, and a y axis near the longest the library takes, whose rows
need the pack's shared memory opt-in; complex128 and complex64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import dda as odda  # noqa: E402
from paper_1002_1505_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda
    return dda


@pytest.mark.parametrize("box,pad", [
    ((5, 4, 3), (10, 8, 6)),
    ((4, 5, 3), (18, 30, 6)),
    ((3, 3, 8), (6, 6, 30)),
    ((1, 7, 6), (2, 16, 12)),
    ((7, 1, 6), (16, 2, 12)),
    ((7, 6, 1), (16, 12, 2)),
    ((2, 9, 2), (4, 18, 50)),
    ((8, 8, 8), (64, 32, 16)),
    ((2, 400, 1), (4, 800, 2)),
])
def test_product_matches_direct_sum(D, box, pad):
    w = W.Workload("green", "RCTGLPRSM", box, 1.5 + 0.05j, 2.0, "GKDLDR", W.uniform_orientations(1, 3), pad=pad)
    ctx = D.Context(0)
    D.setup_workload(ctx, w)
    prob = odda.build_problem(w.shape, w.shpar, w.m, w.x, w.prescription, w.orientations, e01_lf=w.e01,
                              iorth=w.iorth, pad=w.pad)
    rng = np.random.default_rng(sum(pad))
    p = rng.standard_normal((2, 3, ctx.n)) + 1j * rng.standard_normal((2, 3, ctx.n))
    for dt, tol in ((torch.complex64, 1e-5), (torch.complex128, 1e-12)):  # the bars of every product
        pd = torch.from_numpy(p).to(dt).cuda()
        ap = torch.empty_like(pd)
        ctx.dda_matvec(pd, ap)
        for b in range(2):
            ref = odda.apply_a(prob, b, pd[b].cpu().numpy().astype(complex), "direct")
            got = ap[b].cpu().numpy().astype(complex)
            assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= tol, (dt, b)
