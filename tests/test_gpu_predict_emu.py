"""Marginal predictions of emulated handles: the emulation-engine kernel, which
takes many points, and the FP64 kernel, which takes few.

The FP64 form (tested against the oracle on its own) is the reference; two cases
also meet the oracle.  An engine product is within 1e-14 of sum |a b| and the
chains cancel by up to 1e5: 1e-9 of the largest mean and variance, the bar of the
other predictions of emulated handles.  The FP64 kernel gives a point the same bits
whatever else is in the call, so a handle's own few-point prediction tells the
kernels apart.
"""
import numpy as np
import pytest

from oracle import mra_oracle as O
from paper_1507_04789_gb300 import synth

pytestmark = pytest.mark.gpu

RTOL = 1e-9
LEVEL_J2 = (4, 4, 4, 4, 2)


@pytest.fixture(scope="module")
def mra():
    from paper_1507_04789_gb300 import mra as m
    m.load_library()
    return m


def close(a, b):
    for x, y in zip(a, b):
        assert np.abs(x - y).max() <= RTOL * np.abs(y).max()


def data(n, seed, kappa=0.1, clustered=False):
    locs = synth.uniform_locations(n, seed)
    if clustered:   # three patches and a thin strip, most of the domain empty
        k = n // 4
        locs[:k] = 0.2 * locs[:k]
        locs[k:2 * k] = [0.6, 0.05] + 0.15 * locs[k:2 * k]
        locs[2 * k:3 * k] = [0.3, 0.7] + 0.25 * locs[2 * k:3 * k]
        locs[3 * k:] = [0.0, 0.5] + [1.0, 0.02] * locs[3 * k:]
    return locs, synth.noisy_observations(synth.rff_field(locs, 1.5, kappa, 1.0, seed + 1), 0.02, seed + 2)


def near(locs, count, level, seed):
    """Points beside observations, in level-`level` quadtree cells that hold some."""
    rng = np.random.default_rng(seed)
    side = 2 ** level
    cell = lambda x: np.minimum((x * side).astype(int), side - 1) @ [1, side]
    full = np.zeros(side * side, dtype=bool)
    full[cell(locs)] = True
    pts = np.clip(locs[rng.integers(len(locs), size=8 * count)] + 0.02 * rng.standard_normal((8 * count, 2)), 0.0, 1.0)
    pts = pts[full[cell(pts)]]
    assert len(pts) >= count
    return pts[:count]


CASES = {
    # leaves on both sides of 64 observations, about 160 points a region (and still enough with half of them)
    "leaves of 68": dict(n=70000, M=5, r=64, np=40000, family="matern15", half=True),
    # Uhat rows of odd length, nonstationary variance
    "r = 25": dict(n=26000, M=5, r=25, np=26000, family="exp", nonstat=True),
    # a pruned tree, empty leaves under regions with data, nonstationary variance
    "pruned": dict(n=9000, M=5, r=49, np=5000, family="exp", nonstat=True, prune=True, clustered=True),
    # Bessel-function covariance
    "matern": dict(n=4000, M=5, r=36, np=4200, family="matern"),
    # two leaves a region
    "J_M = 2": dict(n=30000, M=5, r=33, np=17000, family="matern15", J=LEVEL_J2),
    # one region, 150 tiles of it, leaves of about 100
    "M = 1": dict(n=400, M=1, r=64, np=19000, family="exp"),
    # leaves of about 95, about 260 points a region
    "leaves of 95": dict(n=6080, M=3, r=48, np=4200, family="matern15", oracle=True),
    # empty leaves of a complete tree (one observation a leaf on average)
    "empty leaves": dict(n=1000, M=5, r=34, np=4200, family="exp", oracle=True),
}


@pytest.mark.parametrize("name", CASES)
def test_many_points(mra, name):
    c = CASES[name]
    locs, y = data(c["n"], 61, clustered=c.get("clustered", False))
    theta = (1.1, 0.12, 0.03) + ((0.8,) if c["family"] == "matern" else ())
    kw = dict(M=c["M"], r=c["r"], family=c["family"], nonstat=c.get("nonstat", False), prune=c.get("prune", False))
    if "J" in c:
        kw["J"] = c["J"]
    pts = near(locs, c["np"], c["M"] - 1, 5) if c.get("prune") else np.random.default_rng(5).random((c["np"], 2))
    few = np.arange(0, c["np"], c["np"] // 24)
    with mra.Handle(locs, y, precision="emu", **kw) as h:
        many = h.predict(theta, pts)
        again = h.predict(theta, pts)
        alone = h.predict(theta, pts[few])
        if c.get("half"):   # the engine's results do not depend on the other points either
            for a, b in zip(h.predict(theta, pts[::2]), many):
                np.testing.assert_array_equal(a, b[::2])
    with mra.Handle(locs, y, **kw) as h:
        ref = h.predict(theta, pts)
    close(many, ref)
    for a, b in zip(many, again):
        np.testing.assert_array_equal(a, b)
    # the same points on the FP64 kernel: other last digits, the same values to the bar
    assert not np.array_equal(many[1][few], alone[1])
    close([m[few] for m in many], alone)
    if c.get("oracle"):
        close([m[few] for m in many], O.predict(O.Problem(locs, y, M=c["M"], r=c["r"], family=c["family"]), theta, pts[few]))


@pytest.mark.parametrize("prune", [False, True])
def test_streamed(mra, prune):
    """Chunks take the whole tree's kernel, on factors formed again."""
    locs, y = data(9000 if prune else 12000, 71, clustered=prune)
    theta = (1.0, 0.1, 0.02)
    pts = near(locs, 5000, 4, 7) if prune else np.random.default_rng(7).random((5000, 2))
    few = np.arange(0, 5000, 200)
    kw = dict(M=5, r=36, family="matern15", precision="emu", prune=prune)
    with mra.Handle(locs, y, stream_level=-1, **kw) as h:
        ref = h.predict(theta, pts)
        assert not np.array_equal(ref[1][few], h.predict(theta, pts[few])[1])
    for s in (1, 2, 4):
        with mra.Handle(locs, y, stream_level=s, **kw) as h:
            got = h.predict(theta, pts)
        for a, b in zip(got, ref):
            np.testing.assert_allclose(a, b, rtol=1e-12, atol=1e-13)
