"""The contraction of given a_lm rows at the edges of its tiles: bins below,
at and past the tile sides (6, 8, 10), tiles moved back to end at the last
bin, rows of one and of several slot chunks, primary counts around the copy
stages and the primary groups, weights of both signs.

Held to the oracle's FP64 contraction of the same rows, 1e-5 of its |w| Gram
scale (the FP32 bound of the other contraction tests)."""
import numpy as np
import pytest

import oracle
from tests.parity import zeta_err

pytestmark = pytest.mark.gpu

TOL_FP32 = 1e-5


@pytest.mark.parametrize("nbins,lmax,m", [(1, 10, 5), (2, 20, 40), (5, 0, 1), (6, 3, 4), (7, 10, 9), (9, 10, 33),
                                          (10, 10, 3), (11, 5, 64), (12, 2, 4097), (13, 12, 17), (16, 7, 5),
                                          (20, 10, 611), (27, 20, 7), (36, 10, 6), (64, 3, 30)])
def test_contract_tile_edges(nbins, lmax, m):
    torch = pytest.importorskip("torch")
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    rng = np.random.default_rng(81)
    a = rng.normal(size=(m, nbins, (lmax + 1) ** 2)).astype(np.float32)
    w = rng.normal(size=m).astype(np.float32)
    out = torch.empty((lmax + 1, nbins, nbins), dtype=torch.float64, device="cuda")
    ctb.contract_noalloc(torch.from_numpy(a).cuda(), torch.from_numpy(w).cuda(), nbins, lmax, out)
    a64, w64 = a.astype(np.float64), w.astype(np.float64)
    ref = {"zeta": oracle.contract(a64, w64, lmax), "gram": oracle.contract(a64, np.abs(w64), lmax)}
    assert zeta_err(out.cpu().numpy(), ref) < TOL_FP32
