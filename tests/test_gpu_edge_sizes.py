"""Edge correction at the ends of its sizes (one multipole, all 21, one bin, 64
bins, pair counts that do not fill a block of warps), in place, and with host
and device arrays mixed.

The oracle solves the same systems in FP64.  Tolerance: the systems' condition
numbers stay below 1e4 (their off-diagonal weights are bounded by 0.9), so two
FP64 eliminations agree to 1e4 * 21 * 2^-53 = 2e-11 of the solution's norm."""
import numpy as np
import pytest

from oracle import edge as oedge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbins,lmax", [(1, 0), (3, 0), (1, 20), (5, 20), (7, 1), (36, 10), (64, 3), (33, 13)])
@pytest.mark.parametrize("mode", ["host", "device", "in_place", "mixed"])
def test_edge_correct_sizes(nbins, lmax, mode):
    torch = pytest.importorskip("torch")
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    rng = np.random.default_rng(17)
    shape = (lmax + 1, nbins, nbins)
    ell = np.arange(lmax + 1)[:, None, None]
    zr = 1e6 * np.where(ell == 0, 1.0, 0.3 * rng.uniform(-1, 1, size=shape) / (1.0 + ell) ** 1.5)
    zn = 1e4 * rng.normal(size=shape)
    ref = oedge.edge_correct(zn, zr)
    est = ctb.CTB(0.0, 1.0, 10.0, nbins, lmax)
    dev = lambda a: torch.from_numpy(a.copy()).cuda()
    if mode == "host":
        got = est.edge_correct(zn, zr)
    elif mode == "device":
        got = est.edge_correct(dev(zn), dev(zr), out=torch.empty(shape, dtype=torch.float64, device="cuda")).cpu().numpy()
    elif mode == "in_place":
        d = dev(zr)
        got = est.edge_correct(dev(zn), d, out=d).cpu().numpy()
    else:
        got = est.edge_correct(zn, dev(zr))
    assert np.max(np.abs(got - ref)) < 2e-11 * np.max(np.abs(ref))
