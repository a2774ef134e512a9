"""Emulated gradient at the edges of its tiles: leaves on both sides of 64
observations (a second column tile of a few columns), knot grids that are no
multiple of 16, the stationary and the nonstationary variance of the two
closed-form families, against the FP64 form."""
import numpy as np
import pytest

from paper_1507_04789_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M,r,family,nonstat", [
    (256, 1, 64, "matern15", False),   # about 64 a leaf
    (400, 1, 36, "exp", True),         # about 100 a leaf
    (1100, 2, 49, "exp", False),       # about 69 a leaf
    (1500, 2, 25, "matern15", True),   # about 94 a leaf
    (900, 3, 18, "exp", True),         # about 14 a leaf
])
def test_emulated_gradient_equals_fp64(n, M, r, family, nonstat):
    from paper_1507_04789_gb300 import mra
    locs = synth.uniform_locations(n, 41)
    y = synth.noisy_observations(synth.rff_field(locs, 1.5, 0.2, 1.0, 42), 0.05, 43)
    theta = (1.1, 0.25, 0.05)
    out = {}
    for precision in ("fp64", "emu"):
        with mra.Handle(locs, y, M=M, r=r, family=family, nonstat=nonstat, precision=precision) as h:
            out[precision] = h.loglik_grad(theta)
    (l0, g0), (l1, g1) = out["fp64"], out["emu"]
    # an engine product is within 1e-14 of sum |ab|; the chains cancel by up to 1e5
    assert l1 == pytest.approx(l0, rel=1e-10)
    assert np.abs(np.asarray(g1) - np.asarray(g0)).max() <= 1e-9 * np.abs(g0).max()
