"""The cell table where a tile of it holds far more points than cells: coarse
grids (few cells in all) and points on one line of a fine grid, around the
number of points at which a tile's entries are searched for instead of counted
(16 points a cell: 8192 in a tile of 512 cells, 131,072 in one of 8192).

Points lie on a line along x at whole multiples of the lattice step, so the
pairs of the estimator are counted exactly in integers; a table entry that is
off by one loses or doubles pairs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctbmod():
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    return ctb


def line(n, box, seed):
    """n whole positions in [0, 2^20) on the x axis of a box of 2^20 steps."""
    rng = np.random.default_rng(seed)
    k = np.sort(rng.integers(0, 1 << 20, n))
    xyz = np.full((n, 3), 0.5 * box)
    xyz[:, 0] = k * (box / (1 << 20))
    return rng.permutation(n), k, xyz


def pairs_on_a_circle(k, lo, hi):
    """Ordered pairs with lo <= distance < hi (steps) on a circle of 2^20 steps."""
    ext = np.concatenate([k, k + (1 << 20)])
    right = np.searchsorted(ext, k + hi) - np.searchsorted(ext, k + lo)
    return 2 * int(right.sum())


@pytest.mark.parametrize("n", [8000, 8192, 8193, 20001])
@pytest.mark.parametrize("rmax,cells", [(256.0, 1), (128.0, 2), (64.0, 4)])
def test_coarse_grid(ctbmod, n, rmax, cells):
    box = 1024.0
    perm, k, xyz = line(n, box, 5)
    est = ctbmod.CTB(box, 1.0, rmax, 3, 1)
    est.set_option(ctbmod.OPT_CELLS_PER_RMAX, cells)
    est.set_points(xyz[perm])
    est.compute()
    assert est.pair_count() == pairs_on_a_circle(k, 1 << 10, int(rmax) << 10)


@pytest.mark.parametrize("n", [131_071, 131_073, 150_001])
def test_full_tile_of_a_fine_grid(ctbmod, n):
    """128 cells across, 1024 along x: the line's row lies in one tile of 8192 of the table's 16.8M entries."""
    box = 1024.0
    perm, k, xyz = line(n, box, 6)
    est = ctbmod.CTB(box, 1.0, 8.0, 3, 1)
    est.set_option(ctbmod.OPT_CELLS_PER_RMAX, 1)
    est.set_points(xyz[perm])
    assert est.grid()[1] == 128
    est.compute()
    assert est.pair_count() == pairs_on_a_circle(k, 1 << 10, 8 << 10)
