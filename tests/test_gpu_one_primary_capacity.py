"""A list capacity that holds one primary's pairs, with nearly four candidates a
pair: the primary is taken alone, its candidates' codes fill the code buffer
(four bytes an entry of the capacity), and none of that goes to unused room."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cells,rmin", [(60_000, 4, 43.0), (260_000, 8, 44.0), (520_000, 12, 44.0)])
def test_one_primary_fills_the_capacity(n, cells, rmin):
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    xyz = np.random.default_rng(14).uniform(0.0, 120.0, (n, 3))

    def alm(cap):
        est = ctb.CTB(120.0, rmin, 50.0, 4, 2)
        est.set_option(ctb.OPT_CELLS_PER_RMAX, cells)
        est.set_option(ctb.OPT_LIST_CAPACITY, cap)
        est.set_points(xyz)
        return est.get_alm(np.array([7]))

    want = alm(0)
    pairs = int(np.rint(want[:, :, 0].sum() * np.sqrt(4 * np.pi)))
    assert np.array_equal(alm(pairs + 50), want)
