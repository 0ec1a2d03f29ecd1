"""Far-field sums organised by box rows (filled boxes) and by sites (sparse boxes) against the oracle.

The row kernels pair sites about the centre of each x row, so the sizes here put the pairing at its
edges: rows of one and two sites, odd and even rows, rows with holes whose partner is missing, empty
rows, more rows than a CTA has threads, one polarization and two, more than one tile of directions.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import observables as oobs  # noqa: E402
from oracle import orientation as oori  # noqa: E402


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_1505_gb300 import dda
    return dda


def _sites(box, keep, seed):
    z, y, x = np.meshgrid(*(np.arange(b) for b in box[::-1]), indexing="ij")
    mask = np.random.default_rng(seed).random(x.shape) < keep
    mask.flat[0] = mask.flat[-1] = True  # the box is the target's extent
    return np.stack([x[mask], y[mask], z[mask]], 1).astype(np.int32)


# (box, share of the box filled, iorth); the last two are sparse: at most a quarter filled, site kernels
CASES = [((1, 7, 5), 1.0, 2), ((2, 3, 4), 0.9, 2), ((5, 4, 3), 0.6, 2), ((8, 5, 33), 0.5, 1), ((33, 9, 20), 0.8, 2),
         ((6, 40, 30), 0.1, 2), ((9, 30, 20), 0.05, 1)]


@pytest.mark.parametrize("box,keep,iorth", CASES)
def test_far_field_sums(D, box, keep, iorth):
    ijk = _sites(box, keep, 3 * box[0] + box[1])
    n, kd = len(ijk), 0.35
    ori = [(0.3, 1.1, 2.0), (2.0, 0.4, 5.0)]
    ctx = D.Context(0)
    ctx.dda_setup_target(ijk, origin=(0.25, -1.5, 3.0))
    ctx.dda_set_incident(kd, ori, iorth=iorth)
    ctx.dda_build_green_fft()
    ctx.dda_set_polarizability("GKDLDR", 1.5 + 0.1j)
    rng = np.random.default_rng(n)
    p = rng.standard_normal((ctx.nrhs, 3, n)) + 1j * rng.standard_normal((ctx.nrhs, 3, n))
    pd = torch.from_numpy(p).cuda()
    r = ijk + np.array([0.25, -1.5, 3.0])
    aeff = (3 * n / (4 * math.pi)) ** (1 / 3)
    out, nd = ctx.dda_angular_averages(pd, 0.7)
    for b in range(ctx.nrhs):
        axes = oori.lab_axes_in_tf(*ori[b // iorth], (1, 0, 0), (0, 1, 0))
        c, g1, g2, gv, ndir = oobs.angular_averages(kd, r, p[b], axes, kd * aeff, 0.7)
        assert nd == ndir
        # FP32 phases and products, rounding 6e-8 a term, averaged over the sum: far below 1e-5
        assert out[b, 0] == pytest.approx(c / (math.pi * aeff ** 2), rel=1e-5)
        np.testing.assert_allclose(out[b, 1:], [g1, g2, *gv], atol=1e-5)
    if iorth == 2:
        dirs = [(0.0, 0.0), (0.7, 0.2), (1.9, 3.0), (2.5, 5.5), (math.pi, 0.0)]
        _, mue = ctx.dda_cross_sections(pd, dirs)
        e01, e02 = oori.polarizations_lf([0, 1, 0])
        for o, a in enumerate(ori):
            axes = oori.lab_axes_in_tf(*a, (1, 0, 0), (0, 1, 0))
            for d, (th, ph) in enumerate(dirs):
                f = oobs.far_field_amplitudes(kd, r, [p[2 * o], p[2 * o + 1]], th, ph, axes)
                ref = oobs.mueller(*oobs.amplitude_matrix(f, e01, e02, ph))
                # FP64 sums of n terms of size one: rounding n 1e-16 of their root sum of squares at most
                np.testing.assert_allclose(mue[o, d], ref, atol=1e-11 * n * kd ** 6)
