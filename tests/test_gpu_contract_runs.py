"""The contraction's FP32 runs: how far its float64 output is from 64 bits at
l = 0, and row counts that take the copy ring round many times and flush the
accumulators in the middle of a slice.

An l = 0 entry is one slot's sum: runs of n FP32 additions, whose ends are
added in FP64.  Error bound: rounding n partial sums of equal positive terms,
each by at most u = 2^-24 of itself and independently (rms u / sqrt 3), moves
a run by u / sqrt 3 * sqrt(n / 3 + 1) of its sum at most; the two roundings of
each product (w a, then a's sum) add 2 / n under the root.  A mean over R runs
divides by sqrt R.  A block owns one partial row, one row per SM as far as the
fixed array of 2^20 doubles holds them, and takes its slice in two runs where
every SM has a block, in one otherwise."""
import math

import pytest

pytestmark = pytest.mark.gpu

TOL_FP32 = 1e-5


def _lib():
    torch = pytest.importorskip("torch")
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    return torch, ctb


def _contract64(torch, a, w, lmax):
    """The contraction in 64 bits, its l = 0..lmax planes and the |w| Gram's diagonal."""
    nb = a.shape[1]
    z = torch.zeros((lmax + 1, nb, nb), device=a.device, dtype=torch.float64)
    g = torch.zeros((lmax + 1, nb), device=a.device, dtype=torch.float64)
    for p in range(0, a.shape[0], 50_000):
        b, v = a[p:p + 50_000].double(), w[p:p + 50_000].double()
        for l in range(lmax + 1):
            c = b[:, :, l * l:(l + 1) ** 2].permute(1, 0, 2)
            f = 4 * math.pi / (2 * l + 1)
            z[l] += f * ((c * v[None, :, None]).reshape(nb, -1) @ c.reshape(nb, -1).T)
            g[l] += f * (c.square().sum(2) * v.abs()).sum(1)
    return z, g


@pytest.mark.parametrize("nbins,lmax,m", [(20, 10, 2000), (20, 10, 20000), (16, 10, 20000), (10, 10, 20000),
                                          (36, 10, 20000), (32, 15, 4000), (20, 4, 20000), (6, 3, 50000)])
def test_l0_error_of_the_float64_output(nbins, lmax, m):
    torch, ctb = _lib()
    g = torch.Generator(device="cuda").manual_seed(17)
    a = 0.5 + torch.rand((m, nbins, (lmax + 1) ** 2), generator=g, device="cuda")
    w = 0.5 + torch.rand(m, generator=g, device="cuda")
    out = torch.empty((lmax + 1, nbins, nbins), dtype=torch.float64, device="cuda")
    ctb.contract_noalloc(a, w, nbins, lmax, out)
    ref, _ = _contract64(torch, a[:, :, :1].contiguous(), w, 0)
    rms = ((out[0] - ref[0]) / ref[0]).square().mean().sqrt().item()
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    rows = min(nsm, 2 ** 20 // ((lmax + 1) * nbins ** 2))
    runs = 2 if rows == nsm else 1
    n = math.ceil(m / rows / runs)
    assert rms < 2.0 ** -24 / math.sqrt(3) * math.sqrt((n / 3 + 1 + 2 / n) / (runs * rows))


# many stages a run with every remainder of a stage (20 bins: four primaries a
# stage, about 66 a slice); several flushes of 1024 primaries a group within a
# slice, one group (36 bins) and eight (3 bins); odd counts
@pytest.mark.parametrize("nbins,lmax,m", [(20, 10, 9999), (20, 10, 10100), (20, 10, 10241), (12, 4, 40003),
                                          (36, 3, 320_003), (3, 2, 1_300_001)])
def test_ring_and_flush_restart(nbins, lmax, m):
    torch, ctb = _lib()
    g = torch.Generator(device="cuda").manual_seed(18)
    a = torch.randn((m, nbins, (lmax + 1) ** 2), generator=g, device="cuda")
    w = torch.randn(m, generator=g, device="cuda")
    out = torch.empty((lmax + 1, nbins, nbins), dtype=torch.float64, device="cuda")
    ctb.contract_noalloc(a, w, nbins, lmax, out)
    ref, gram = _contract64(torch, a, w, lmax)
    d = gram.sqrt()
    assert ((out - ref).abs() / (d[:, :, None] * d[:, None, :])).max().item() < TOL_FP32
