"""a_lm against the FP64 oracle where the accumulation's path changes: lists
of a few neighbours (four bins side by side in a warp), of a few hundred
(two), and long ones (one), with bin counts that do not divide by four or
two, empty bins inside a group and groups that are empty.

Tolerance: 1e-5 of the |w| sum's scale (tests/parity.alm_err), the FP32
bound that the a_lm export is held to everywhere."""
import numpy as np
import pytest

import oracle
from paper_2604_08855_gb300 import synth
from tests.parity import alm_err

pytestmark = pytest.mark.gpu

TOL_FP32 = 1e-5


@pytest.fixture(scope="module")
def ctbmod():
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    return ctb


# points, r_max: mean neighbours a bin from below 1 to above 800
@pytest.mark.parametrize("n,rmax,nbins", [(300, 40.0, 7), (3000, 60.0, 1), (6000, 70.0, 6), (20000, 80.0, 13),
                                          (40000, 95.0, 5), (60000, 100.0, 33)])
@pytest.mark.parametrize("lmax", [0, 4, 10, 13])
def test_alm_at_every_list_length(ctbmod, n, rmax, nbins, lmax):
    xyz, w = synth.thomas(n, 300.0, max(1, n // 100), 5.0, seed=61, weights="u0.5-1.5")
    kw = dict(box=300.0, rmin=0.0, rmax=rmax, nbins=nbins, lmax=lmax)
    est = ctbmod.CTB(**kw)
    est.set_points(xyz, w)
    prim = synth.sample_primaries(n, 24, seed=5)
    a = est.get_alm(prim)
    ref = oracle.alm(xyz, w, prim=prim, **kw)
    w1 = oracle.alm(xyz, np.abs(w), prim=prim, **{**kw, "lmax": 0})[:, :, 0] * np.sqrt(4 * np.pi)
    assert alm_err(a, ref, w1, lmax) < TOL_FP32


@pytest.mark.parametrize("nbins,rmin", [(3, 0.0), (10, 0.3)])
def test_alm_of_isolated_points_and_empty_groups(ctbmod, nbins, rmin):
    """Two close pairs far apart: most bins and whole groups of bins are empty."""
    xyz = np.array([[10.0, 10, 10], [11.0, 10, 10], [90.0, 90, 90], [90.0, 92.5, 90], [50.0, 50, 50]])
    w = np.array([1.0, 2.0, -1.5, 0.5, 3.0])
    kw = dict(box=200.0, rmin=rmin, rmax=3.0, nbins=nbins, lmax=6)
    est = ctbmod.CTB(**kw)
    est.set_points(xyz, w)
    prim = np.arange(5)
    a = est.get_alm(prim)
    ref = oracle.alm(xyz, w, prim=prim, **kw)
    assert np.max(np.abs(a - ref)) < TOL_FP32 * 3.0
