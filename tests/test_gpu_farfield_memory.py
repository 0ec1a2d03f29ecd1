"""Far-field buffers with many right-hand sides and directions: what a call leaves in the context is
bounded (64 MiB and the allocator's granularity), directions that take several passes give what they give
alone, and an x row long enough that the averages stage one row at a time matches the oracle."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import observables as oobs  # noqa: E402
from oracle import orientation as oori  # noqa: E402

KEPT = (64 + 4) << 20


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda
    return dda


def _context(D, box, norient, seed, only=None):
    z, y, x = np.meshgrid(*(np.arange(b) for b in box[::-1]), indexing="ij")
    ijk = np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.int32)
    rng = np.random.default_rng(seed)
    ori = [tuple(v) for v in rng.uniform((0, 0, 0), (2 * math.pi, math.pi, 2 * math.pi), (norient, 3))]
    if only is not None:
        ori = ori[only:only + 1]
    ctx = D.Context(0)
    ctx.dda_setup_target(ijk, origin=(0.25, -1.5, 3.0))
    ctx.dda_set_incident(0.2, ori, iorth=2)
    ctx.dda_build_green_fft()
    ctx.dda_set_polarizability("GKDLDR", 1.5 + 0.1j)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    p = torch.randn((ctx.nrhs, 3, len(ijk)), dtype=torch.complex128, device="cuda", generator=gen)
    return ctx, ijk, ori, p


def _left_behind(call):
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    out = call()
    torch.cuda.synchronize()
    return out, free - torch.cuda.mem_get_info()[0]


def test_many_directions(D):
    ctx, _, _, p = _context(D, (32, 48, 48), 16, 1)
    rng = np.random.default_rng(2)
    dirs = np.stack([rng.uniform(0, math.pi, 3001), rng.uniform(0, 2 * math.pi, 3001)], 1)
    alone = [ctx.dda_cross_sections(p, dirs[a:b])[1] for a, b in ((0, 7), (1100, 1181), (2996, 3001))]
    (_, mue), kept = _left_behind(lambda: ctx.dda_cross_sections(p, dirs))
    assert kept <= KEPT
    for (a, b), ref in zip(((0, 7), (1100, 1181), (2996, 3001)), alone):
        np.testing.assert_array_equal(np.asarray(mue)[:, a:b], np.asarray(ref))


def test_averages_in_several_passes(D):
    ctx, _, _, p = _context(D, (32, 48, 48), 16, 3)
    _, nd = ctx.dda_angular_averages(p, 1.0)
    eta = math.sqrt(nd / 26000.0)  # the number of directions goes with 1 / eta^2
    (fine, ndf), kept = _left_behind(lambda: ctx.dda_angular_averages(p, eta))
    assert ndf > 20000  # 112 phases a direction: more than 256 MiB for 16 orientations
    assert kept <= KEPT
    for o in (0, 9, 15):
        one, _, _, _ = _context(D, (32, 48, 48), 16, 3, only=o)
        ref, ndr = one.dda_angular_averages(p[2 * o:2 * o + 2].contiguous(), eta)
        assert ndr == ndf
        # the same row sums, added in other groups: 2304 rows with 48 bits each, 1e-11
        np.testing.assert_allclose(fine[2 * o:2 * o + 2], ref, rtol=1e-9, atol=1e-9)


@pytest.mark.parametrize("box", [(301, 7, 9), (300, 16, 3)])
def test_one_long_row_at_a_time(D, box):
    ctx, ijk, ori, p = _context(D, box, 1, 5)
    kd = 0.2
    out, nd = ctx.dda_angular_averages(p, 2.0)
    r = ijk + np.array([0.25, -1.5, 3.0])
    aeff = (3 * len(ijk) / (4 * math.pi)) ** (1 / 3)
    for b in range(ctx.nrhs):
        axes = oori.lab_axes_in_tf(*ori[0], (1, 0, 0), (0, 1, 0))
        c, g1, g2, gv, ndir = oobs.angular_averages(kd, r, p[b].cpu().numpy(), axes, kd * aeff, 2.0)
        assert nd == ndir
        # FP32 phases and products, rounding 6e-8 a term, averaged over the sum: far below 1e-5
        assert out[b, 0] == pytest.approx(c / (math.pi * aeff ** 2), rel=1e-5)
        np.testing.assert_allclose(out[b, 1:], [g1, g2, *gv], atol=1e-5)
