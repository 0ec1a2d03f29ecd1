"""The complex64 plane pass worked off in two halves of ky (DDA_SCHEDULE half256 / half384) against the
oracle's direct sum: every plane pair that has the kernel, boxes that fill the pruned half exactly and
boxes with odd ragged ends, one row or column short of a thread's tile."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import dda as odda  # noqa: E402
from oracle import interaction as oint  # noqa: E402
from paper_1002_1505_gb300 import workloads as W  # noqa: E402

PAIRS = [(64, 96), (80, 80), (96, 64), (96, 96), (128, 128), (128, 64), (64, 128), (128, 96), (96, 128)]


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda
    return dda


@pytest.mark.parametrize("threads", [256, 384])
@pytest.mark.parametrize("short", [(0, 0), (3, 5)])
@pytest.mark.parametrize("py,pz", PAIRS)
def test_half_planes_match_direct_sum(D, monkeypatch, py, pz, short, threads):
    monkeypatch.setenv("DDA_SCHEDULE", f"half{threads}")
    box = (3, py // 2 - short[0], pz // 2 - short[1])
    w = W.Workload("half", "RCTGLPRSM", box, 1.5 + 0.05j, 3.0, "GKDLDR", W.uniform_orientations(1, py + pz),
                   pad=(16, py, pz))
    ctx = D.Context(0)
    D.setup_workload(ctx, w)
    prob = odda.build_problem(w.shape, w.shpar, w.m, w.x, w.prescription, w.orientations, e01_lf=w.e01,
                              iorth=w.iorth, pad=w.pad)
    rng = np.random.default_rng(py * pz)
    p = rng.standard_normal((2, 3, ctx.n)) + 1j * rng.standard_normal((2, 3, ctx.n))
    pd = torch.from_numpy(p.astype(np.complex64)).cuda()
    ap = torch.empty_like(pd)
    ctx.dda_matvec(pd, ap)
    assert D.dda_schedule_info(ctx, D.DDA_C64)[:3] == (3, 1, threads)
    rows = np.concatenate([[0, ctx.n - 1], np.sort(rng.choice(ctx.n, 30, replace=False))])
    for b in range(2):
        ref = oint.matvec_direct(prob.target.r, prob.kd, prob.rhs[b].inv_alpha, pd[b].cpu().numpy().astype(complex),
                                 rows=rows)
        got = ap[b].cpu().numpy().astype(complex)[:, rows]
        # complex64 transforms: ~1e-7 relative; the bar of every complex64 product is 1e-5
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
