"""Pairs at and beside the first and the last bin edge, where the float
pre-filter, the float bin and the exact integer test hand over: separations
r_edge (1 + d) for d from 1e-8 to 1e-4 on both sides, with bins from a few to
far more than the float coordinate resolves, on short and on long cell rows.

The counts equal those of Python integers exactly: the box is 2^32 units wide
and a bin starts at the smallest squared separation whose root reaches its
edge."""
from fractions import Fraction
from math import ceil

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cpr", [1, 8])                   # rows of hundreds of points, and of a few
@pytest.mark.parametrize("rmin,rmax,nbins", [(0.0, 40.0, 10), (5.0, 40.0, 35), (30.0, 40.0, 20), (39.0, 40.0, 64)])
def test_pairs_beside_the_outer_edges(cpr, rmin, rmax, nbins):
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    rng = np.random.default_rng(23)
    d = np.concatenate([s * np.logspace(-8, -4, 400) for s in (-1.0, 1.0)] + [np.zeros(20)])
    r = np.concatenate([e * (1.0 + d) for e in (rmin, rmax) if e > 0])
    u = rng.normal(size=(r.size, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    shell = 64.0 + r[:, None] * u
    xyz = np.concatenate([[[64.0, 64.0, 64.0]], shell, [[64.0 + e, 64.0, 64.0] for e in (rmin, rmax) if e > 0],
                          rng.uniform(0.0, 128.0, (30000, 3))])
    w = np.ones(len(xyz))
    kw = dict(box=128.0, rmin=rmin, rmax=rmax, nbins=nbins, lmax=0)
    est = ctb.CTB(**kw)
    est.set_option(ctb.OPT_CELLS_PER_RMAX, cpr)
    est.set_points(xyz, w)
    prim = np.arange(3)
    a = est.get_alm(prim)
    q = np.floor(xyz * 2.0 ** 25).astype(np.int64)  # the ingest truncates to units
    dr = (rmax - rmin) / nbins
    edges = [rmin] + [rmin + b * dr for b in range(1, nbins)] + [rmax]
    thr = np.array([ceil(Fraction(e) ** 2 * 2 ** 50) for e in edges], dtype=np.uint64)
    for p in prim:
        d = ((q - q[p] + 2 ** 31) % 2 ** 32 - 2 ** 31).astype(np.uint64)  # squares modulo 2^64 are exact below it
        t = (d * d).sum(axis=1, dtype=np.uint64)
        b = np.searchsorted(thr, t, side="right") - 1
        ref = np.bincount(b[(t > 0) & (b >= 0) & (b < nbins)], minlength=nbins)
        assert np.array_equal(np.rint(a[p, :, 0] * np.sqrt(4 * np.pi)), ref)
