"""The second set of compile-time FFT lengths (grids the library pads by itself for boxes of no
convenient size) against the oracle's direct sum, on each axis, in both precisions, with boxes that fill
the pruned half and boxes one short of it; a folded BiCGstab solve on such a grid; and the product with
the fixed scratch where the compile-time schedule's longer rows do not fit it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import dda as odda  # noqa: E402
from paper_1002_1505_gb300 import workloads as W  # noqa: E402

LENGTHS = [18, 20, 30, 36, 50, 54, 60, 72, 90, 100, 108, 120, 144, 150, 162, 180, 200, 216, 240, 288]


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda
    return dda


def _problem(D, box, pad, seed):
    w = W.Workload("len", "RCTGLPRSM", box, 1.5 + 0.05j, 2.0, "GKDLDR", W.uniform_orientations(1, seed), pad=pad)
    ctx = D.Context(0)
    D.setup_workload(ctx, w)
    return ctx, odda.build_problem(w.shape, w.shpar, w.m, w.x, w.prescription, w.orientations, e01_lf=w.e01,
                                   iorth=w.iorth, pad=w.pad)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("length", LENGTHS)
def test_products_match_direct_sum(D, length, axis):
    for short in (0, 1):
        box, pad = [3, 4, 3], [16, 18, 24]
        box[axis], pad[axis] = length // 2 - short, length
        ctx, prob = _problem(D, tuple(box), tuple(pad), length)
        assert D.dda_schedule_info(ctx, D.DDA_C64)[:2] == (5, 1)
        rng = np.random.default_rng(length)
        p = rng.standard_normal((2, 3, ctx.n)) + 1j * rng.standard_normal((2, 3, ctx.n))
        for dt, tol in ((torch.complex64, 1e-5), (torch.complex128, 1e-12)):  # the bars of every product
            pd = torch.from_numpy(p).to(dt).cuda()
            ap = torch.empty_like(pd)
            ctx.dda_matvec(pd, ap)
            for b in range(2):
                ref = odda.apply_a(prob, b, pd[b].cpu().numpy().astype(complex), "direct")
                got = ap[b].cpu().numpy().astype(complex)
                assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= tol, (short, dt, b)


def test_folded_solve_matches_lu(D):
    ctx, prob = _problem(D, (9, 10, 5), (18, 20, 18), 5)
    p = torch.zeros((ctx.nrhs, 3, ctx.n), dtype=torch.complex128, device="cuda")
    reps, _ = ctx.dda_solve(p, precision="MIXED", tol=1e-8)
    ps, _ = odda.solve(prob, "lu")
    for b in range(ctx.nrhs):
        # residual 1e-8 times the condition of this matrix (below 100)
        assert reps[b]["converged"] == 1
        assert np.linalg.norm(p[b].cpu().numpy() - ps[b]) / np.linalg.norm(ps[b]) <= 1e-6


def test_fixed_scratch_falls_back_to_short_rows(D):
    """200 x 72 x 108, complex128: 37 MB of workspace with rows of Py, 19 MB with rows of Ny (the general
    engine's plane takes 210 KB of shared memory)."""
    ctx, _ = _problem(D, (100, 36, 54), None, 9)
    p = torch.randn((1, 3, ctx.n), dtype=torch.complex128, device="cuda")
    a, b = torch.empty_like(p), torch.empty_like(p)
    ctx.dda_matvec(p, a, nrhs=1)
    ctx.dda_matvec_noalloc(p, b, nrhs=1)
    assert float((a - b).norm() / a.norm()) <= 1e-13  # two FP64 engines
