"""Neighbour enumeration where its walk changes: rows of hundreds of points
(four steps of a row at a time), rows of a few (many rows in one step), rows
that wrap around the box, and a full window of rows (r_max = box / 2).

Pair counts equal the oracle's exactly (bins are decided exactly); zeta holds
to 1e-5 of the Gram scale, the FP32 bound of the other parity tests."""
import numpy as np
import pytest

import oracle
from paper_2604_08855_gb300 import synth
from tests.parity import zeta_err

pytestmark = pytest.mark.gpu

TOL_FP32 = 1e-5


@pytest.fixture(scope="module")
def ctbmod():
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    return ctb


@pytest.mark.parametrize("box", [128.0, 0.0])
@pytest.mark.parametrize("n,rmax,cpr", [(2000, 64.0, 1), (2000, 6.0, 12), (15000, 30.0, 2), (15000, 30.0, 16),
                                        (50000, 40.0, 1), (50000, 64.0, 3)])
def test_rows_short_and_long(ctbmod, box, n, rmax, cpr):
    xyz, w = synth.thomas(n, 128.0, max(1, n // 100), 5.0, seed=71, weights="u0.5-1.5")
    if box == 0.0:
        xyz = synth.snap_dyadic(xyz)
    kw = dict(box=box, rmin=1.0, rmax=rmax, nbins=9, lmax=2)
    est = ctbmod.CTB(**kw)
    est.set_option(ctbmod.OPT_CELLS_PER_RMAX, cpr)
    est.set_points(xyz, w)
    prim = synth.sample_primaries(n, 40, seed=6)
    z = est.compute_subset(prim)
    ref = oracle.zeta(xyz, w, prim=prim, **kw)
    assert est.pair_count() == ref["npairs"]
    assert zeta_err(z, ref) < TOL_FP32
