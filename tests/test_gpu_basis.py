"""a_lm against the FP64 oracle for l_max on both sides of every pass split:
each pass has its own scaled Chebyshev basis and its own flush table.

Tolerance, in the |w| sum's scale (tests/parity.alm_err): FP32 directions are
rounded to 6e-8 in each coordinate, and a unit-normalised harmonic of degree
l has an rms gradient below l + 1, so they give at most 2 (l + 1) 6e-8; the
flush's map amplifies the moments' rounding at most 11 times (rms), with 4
roundings in a moment's chain counted at 6e-8.  (2 x 21 + 4 x 11) x 6e-8 =
5.2e-6 at l_max 20, taken for every l_max."""
import numpy as np
import pytest

import oracle
from paper_2604_08855_gb300 import synth
from tests.parity import alm_err

pytestmark = pytest.mark.gpu

TOL = (2 * 21 + 4 * 11) * 6e-8


@pytest.mark.parametrize("lmax", [1, 2, 3, 6, 9, 10, 11, 12, 14, 16, 17, 18, 19, 20])
@pytest.mark.parametrize("n", [4000, 12000])  # two lists a warp, one list a warp
def test_alm_at_every_pass_split(n, lmax):
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    xyz, w = synth.thomas(n, 100.0, n // 40, 4.0, seed=17, weights="u0.5-1.5")
    kw = dict(box=100.0, rmin=10.0, rmax=30.0, nbins=1 if n > 8000 else 2, lmax=lmax)
    est = ctb.CTB(**kw)
    est.set_points(xyz, w)
    prim = synth.sample_primaries(n, 16, seed=3)
    a = est.get_alm(prim)
    ref = oracle.alm(xyz, w, prim=prim, **kw)
    w1 = oracle.alm(xyz, np.abs(w), prim=prim, **{**kw, "lmax": 0})[:, :, 0] * np.sqrt(4 * np.pi)
    assert alm_err(a, ref, w1, lmax) < TOL
