"""Emulated aggregation of a parent with sixteen children of 64 knots: 1024 stacked
rows, eight 128-row scale groups."""
import pytest

from oracle import mra_oracle as O
from paper_1507_04789_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,rtol", [("emu", 1e-10), ("mixed", None)])
def test_sixteen_children_of_64_knots(precision, rtol):
    from paper_1507_04789_gb300 import mra
    J, n = (16, 4), 2500
    locs = synth.uniform_locations(n, 31)
    y = synth.noisy_observations(synth.rff_field(locs, 1.5, 0.2, 1.0, 32), 0.05, 33)
    theta = (1.0, 0.2, 0.05)
    ll_o = O.loglik(O.Problem(locs, y, M=2, r=64, family="matern15", J=J), theta)
    with mra.Handle(locs, y, M=2, r=64, family="matern15", precision=precision, J=J) as h:
        ll = h.loglik(theta)
    # (3xTF32: 2e-6 per observation, the bound its other level-varying trees are held to)
    assert abs(ll - ll_o) <= (rtol * abs(ll_o) if rtol else 2e-6 * n)
