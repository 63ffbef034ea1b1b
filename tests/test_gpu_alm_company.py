"""A primary's a_lm rows do not depend on the primaries they are asked for with:
bit for bit the same alone, among primaries of its own kind, and in a mixture
of sparse and crowded ones, whose lists a warp accumulates four, two or one at
a time."""
import numpy as np
import pytest

from paper_2604_08855_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctbmod():
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    return ctb


def check(est, counts, nbins):
    """counts: neighbours of each point.  Picks 12 primaries below a mean of 160
    a list, 12 up to 800 and 12 above, and compares their rows in different calls."""
    mean = counts / nbins
    kinds = [np.flatnonzero((mean >= lo) & (mean < hi))[::7][:12].astype(np.int64)
             for lo, hi in ((1, 160), (160, 800), (800, np.inf))]
    assert all(k.size == 12 for k in kinds)
    every = np.concatenate(kinds)[np.random.default_rng(3).permutation(36)]
    rows = dict(zip(every.tolist(), est.get_alm(every)))
    for kind in kinds:
        for got, p in zip(est.get_alm(kind), kind):
            assert np.array_equal(got, rows[int(p)])
        for p in kind[:3]:
            assert np.array_equal(est.get_alm(np.array([p]))[0], rows[int(p)])


@pytest.mark.parametrize("nbins,lmax", [(5, 3), (5, 10), (3, 12), (6, 20)])
def test_rows_in_any_company(ctbmod, nbins, lmax):
    rng = np.random.default_rng(12)
    box, rmax = 400.0, 20.0
    # points thin out from a centre: 40 to some 10^4 neighbours within r_max
    xyz = np.concatenate([rng.normal(200.0, s, (n, 3)) for s, n in ((4.0, 8000), (12.0, 8000), (40.0, 30000))])
    xyz = synth.snap_periodic(xyz, box)
    est = ctbmod.CTB(box, 0.0, rmax, nbins, lmax)
    est.set_points(xyz, rng.uniform(0.5, 1.5, xyz.shape[0]))
    sample = rng.choice(xyz.shape[0], 3000, replace=False)
    counts = np.zeros(xyz.shape[0])
    for p in sample:
        d = xyz - xyz[p]
        counts[p] = np.count_nonzero((d * d).sum(1) < rmax * rmax) - 1
    check(est, counts, nbins)


def test_rows_in_any_company_on_the_sphere(ctbmod):
    rng = np.random.default_rng(13)
    nbins, theta = 4, 0.05
    v = np.concatenate([rng.normal([0.0, 0.0, 1.0], s, (n, 3)) for s, n in ((0.02, 6000), (0.08, 8000), (0.6, 60000))])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    est = ctbmod.CTB.sphere(0.0, theta, nbins, 8)
    est.set_points(v, rng.normal(size=v.shape[0]))
    sample = rng.choice(v.shape[0], 4000, replace=False)
    counts = np.zeros(v.shape[0])
    chord2 = (2 * np.sin(theta / 2)) ** 2
    for p in sample:
        d = v - v[p]
        counts[p] = np.count_nonzero((d * d).sum(1) < chord2) - 1
    check(est, counts, nbins)
