"""Predictions of fewer points than leaves run a CTA a point instead of a CTA a leaf:
the same bits as in a call with more points than leaves, at the edges of the choice
and of the tiles (one point, one less and one more than the leaves, points crowded
into one leaf across several tiles), and the oracle's values."""
import numpy as np
import pytest

from oracle import mra_oracle as O
from paper_1507_04789_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,r", [("fp64", 16), ("fp64", 30), ("fp64", 49), ("mixed", 32)])
def test_few_points(precision, r):
    from paper_1507_04789_gb300 import mra
    M, leaves = 4, 256
    locs = synth.uniform_locations(5000, 91)
    y = synth.noisy_observations(synth.rff_field(locs, 1.5, 0.1, 1.0, 92), 0.05, 93)
    theta = (1.0, 0.1, 0.05)
    rng = np.random.default_rng(94)
    pts = rng.random((600, 2))
    pts[:140] = 0.51 + 0.05 * pts[:140]                  # one leaf: nine tiles of 16, three of 64
    order = rng.permutation(600)
    pts = pts[order]
    crowd = np.flatnonzero(order < 140)
    with mra.Handle(locs, y, M=M, r=r, family="matern15", precision=precision) as h:
        mean, var = h.predict(theta, pts)
        sets = [np.arange(k) for k in (1, 2, leaves - 1, leaves, leaves + 1)]
        sets += [crowd, crowd[:16], crowd[:17], crowd[:65], np.append(crowd[:33], np.arange(3))]
        for s in sets:
            m, v = h.predict(theta, pts[s])
            np.testing.assert_array_equal(m, mean[s])
            np.testing.assert_array_equal(v, var[s])
    if precision == "fp64":
        mo, vo = O.predict(O.Problem(locs, y, M=M, r=r, family="matern15"), theta, pts[:40])
        assert np.abs(mean[:40] - mo).max() <= 1e-9 * np.abs(mo).max()
        assert np.abs(var[:40] - vo).max() <= 1e-9 * np.abs(vo).max()


def test_few_points_streamed():
    """A chunk's grid of points keeps to the chunk's leaves."""
    from paper_1507_04789_gb300 import mra
    locs = synth.uniform_locations(5000, 95)
    y = synth.noisy_observations(synth.rff_field(locs, 1.5, 0.1, 1.0, 96), 0.05, 97)
    theta = (1.0, 0.1, 0.05)
    pts = np.random.default_rng(98).random((300, 2))
    pts[:40] = 0.51 + 0.05 * pts[:40]
    with mra.Handle(locs, y, M=4, r=24, family="exp", stream_level=-1) as h:
        mean, var = h.predict(theta, pts)
    for s in (1, 3):
        with mra.Handle(locs, y, M=4, r=24, family="exp", stream_level=s) as h:
            for k in (1, 3, 4, 63, 64, 65, 300):     # chunks of 64 and of 4 leaves
                m, v = h.predict(theta, pts[:k])
                np.testing.assert_allclose(m, mean[:k], rtol=1e-12, atol=1e-13)
                np.testing.assert_allclose(v, var[:k], rtol=1e-12, atol=1e-13)
