"""Which kernel predicts on an emulated handle: points, blocks and trees that the
emulation engine takes longer for than the FP64 kernel stay on the FP64 kernel.

The FP64 kernel gives a point the same bits whatever else is in the call and the
engine rounds differently, so a call that equals its own few-point subset bit for
bit ran on the FP64 kernel.
"""
import numpy as np
import pytest

from paper_1507_04789_gb300 import synth

pytestmark = pytest.mark.gpu

LEVEL_J2 = (4, 4, 4, 4, 2)


@pytest.mark.parametrize("M,J,n,r,np_,layout", [
    (5, None, 10000, 33, 1024, "uniform"),      # FP64 / engine 1.09, over a sixteenth of the domain 0.80
    (5, None, 40000, 17, 16384, "uniform"),     # 0.98
    (2, None, 1000, 32, 4096, "uniform"),       # 0.52
    (1, None, 250, 17, 4096, "uniform"),        # 0.44
    (1, None, 24, 48, 4096, "uniform"),         # 0.73
    (4, None, 1500, 20, 25000, "uniform"),      # sparse leaves, r = 17: 0.81
    (5, LEVEL_J2, 30000, 17, 8192, "uniform"),  # 0.85
    (6, None, 100000, 32, 100000, "spot"),      # all in one leaf: 0.8
])
def test_calls_the_engine_would_slow_down(M, J, n, r, np_, layout):
    from paper_1507_04789_gb300 import mra
    locs = synth.uniform_locations(n, 81)
    y = synth.noisy_observations(synth.rff_field(locs, 1.5, 0.1, 1.0, 82), 0.05, 83)
    theta = (1.0, 0.1, 0.05)
    pts = np.random.default_rng(9).random((np_, 2))
    if layout == "spot":
        pts = 0.3 + 1e-4 * pts
    few = np.arange(0, np_, np_ // 16)
    with mra.Handle(locs, y, M=M, r=r, family="matern15", precision="emu", **({} if J is None else {"J": J})) as h:
        many = h.predict(theta, pts)
        alone = h.predict(theta, pts[few])
    for a, b in zip(many, alone):
        np.testing.assert_array_equal(a[few], b)
