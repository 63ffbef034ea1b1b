"""Performance cases: what programs built on this library have it do.

The estimator's cases are whole steps (catalogue in, zeta out) and the a_lm of
chosen primaries, on the catalogue families of synth.py: uniform and Thomas
points in a periodic cube, a cut-sky sector of data and randoms, a field on
the unit sphere.  The rest are the library's other entry points: the batch of
mock catalogues, shared neighbour lists, the contraction of a caller's own
a_lm rows, and the edge correction.

Coordinates lie on the device's fixed-point grid (box / 2^32, or 2^-20 in open
space), as the synthetic catalogues of this repository do, so a bin decision
is the same in any exact arithmetic.  zeta is returned as float32: its pair
sums are FP32 sums (or BF16 / TF32 products of them) whatever the container,
and a program that stacks many of them keeps them so.  The edge correction is
FP64 throughout and stays float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_08855_gb300 import ctb

PRECISIONS = {"fp32": ctb.PREC_FP32, "bf16x3": ctb.PREC_BF16X3, "tf32": ctb.PREC_TF32}
DEV = "cuda"


# ---------------------------------------------------------------------------
# cases

def listed():
    return [
        # the smallest whole call: a quick look at 20k points held on the
        # host, numpy in and numpy out; launches and synchronisations count
        dict(name="uniform_20k_host", do="compute", points="uniform", n=20_000, box=1000.0, rmin=10.0, rmax=100.0,
             nbins=10, lmax=10, prec="fp32", cells=0, host=True),
        # the ordinary survey step: 10^6 clustered points, l_max 10, FP32
        dict(name="thomas_1m_l10", do="compute", points="thomas", n=1_000_000, box=1000.0, rmin=5.0, rmax=200.0,
             nbins=20, lmax=10, prec="fp32", cells=6, host=False),
        # high resolution in angle and radius, the tensor-core contraction:
        # one rank's shard (1/16 of the primaries) of the 4M-point catalogue
        dict(name="thomas_4m_l20_shard", do="subset", points="thomas", n=4_000_000, box=2000.0, rmin=10.0, rmax=200.0,
             nbins=32, lmax=20, prec="bf16x3", cells=4, m=250_000),
        # the parity-size catalogue at l_max 20 in plain FP32: sparse lists
        dict(name="thomas_200k_l20", do="compute", points="thomas", n=200_000, box=2000.0, rmin=10.0, rmax=200.0,
             nbins=32, lmax=20, prec="fp32", cells=4, host=False),
        # a cut sky with an open boundary: data minus randoms, both signs
        dict(name="sector_800k", do="compute", points="sector", n=800_000, box=0.0, rmin=20.0, rmax=200.0,
             nbins=36, lmax=10, prec="fp32", cells=8, host=False),
        # a convergence map on the sphere, 12 * 512^2 pixels, theta < 200'
        dict(name="sphere_nside512", do="sphere", points="sphere", n=3_145_728, tmin=0.0, tmax=200.0, nbins=20,
             lmax=8, cells=0),
        # a covariance run: many small mock catalogues in one call
        dict(name="mock_batch_24", do="batch", points="thomas", k=24, nlo=20_000, nhi=200_000, box=1000.0, rmin=10.0,
             rmax=150.0, nbins=20, lmax=10, prec="fp32", cells=0),
        # the approximate mode: close pivots share one neighbour list
        dict(name="shared_1m", do="shared", points="thomas", n=1_000_000, box=1000.0, rmin=5.0, rmax=200.0,
             nbins=20, lmax=10, prec="fp32", cells=6, h=10.0),
        # multipole coefficients of chosen primaries, as maps for a further
        # analysis: l_max 10, and l_max 20 with more bins than points need
        dict(name="alm_8k_l10", do="alm", points="thomas", n=1_000_000, box=1000.0, rmin=5.0, rmax=200.0, nbins=20,
             lmax=10, cells=6, m=8192),
        dict(name="alm_3k_l20", do="alm", points="thomas", n=4_000_000, box=2000.0, rmin=10.0, rmax=200.0, nbins=32,
             lmax=20, cells=4, m=3001),
        # a caller's own rows, without device allocation (a service loop)
        dict(name="contract_20k_l10", do="contract", m=20_000, nbins=20, lmax=10),
        # the last step of a survey analysis: sums to edge-corrected zeta
        dict(name="edge_36_l10", do="edge", nbins=36, lmax=10),
    ]


# the listed cases' largest estimated cost (see _cost), in pair-multipole
# updates plus a flat cost per pair
_MOST = 1.05e13


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    while True:
        do = rng.choice(["compute", "compute", "subset", "sphere", "batch", "shared", "alm", "alm", "contract", "edge"])
        lmax = rng.choice([rng.randint(2, 10), 10, rng.randint(11, 20), 20])
        c = dict(do=do, nbins=rng.choice([rng.randint(5, 40), 10, 20, 32]), lmax=lmax)
        if do == "edge":
            return c
        if do == "contract":
            c["nbins"] = min(c["nbins"], int(math.sqrt(16384 / (lmax + 1))))
            c["m"] = min(logint(500, 200_000), int(3e8 / (c["nbins"] * (lmax + 1) ** 2)))
            return c
        if do == "sphere":
            c.update(points="sphere", n=logint(50_000, 3_000_000), tmin=rng.choice([0.0, 10.0]),
                     tmax=rng.uniform(100.0, 300.0), lmax=rng.randint(2, 16), cells=0)
        elif do == "batch":
            k = rng.randint(3, 40)
            c.update(points="thomas", k=k, nlo=10_000, nhi=logint(20_000, 300_000), box=1000.0,
                     rmin=rng.choice([0.0, 10.0]), rmax=rng.uniform(80.0, 160.0), lmax=min(lmax, 10), prec="fp32",
                     cells=rng.choice([0, 6]))
        else:
            points = rng.choice(["uniform", "thomas", "thomas", "sector"])
            box = 0.0 if points == "sector" else rng.choice([1000.0, 2000.0])
            n = logint(10_000, 4_000_000)
            c.update(points=points, n=n, box=box, rmin=rng.choice([1.0, 5.0, 20.0]), rmax=rng.uniform(60.0, 200.0),
                     cells=rng.choice([0, 4, 6]))
            if do in ("compute", "subset"):
                c["prec"] = rng.choice(["fp32", "fp32", "bf16x3", "tf32"])
            if do == "compute":
                c["host"] = rng.random() < 0.25
            if do == "subset":
                c["m"] = min(n, logint(1000, 500_000))
            if do == "alm":
                c["m"] = min(n, logint(100, 20_000), int(3e8 / (c["nbins"] * (lmax + 1) ** 2)))
            if do == "shared":
                c.update(h=rng.choice([0.0, rng.uniform(5.0, 30.0)]), prec="fp32")
        if _cost(c) <= _MOST:
            return c


# ---------------------------------------------------------------------------
# inputs

def _sizes(c):
    """Catalogue sizes of a batch: log-spaced from nlo to nhi, in a fixed mixed order."""
    k = c["k"]
    s = [int(round(c["nlo"] * (c["nhi"] / c["nlo"]) ** (i / max(k - 1, 1)))) for i in range(k)]
    return [s[(7 * i + 3) % k] for i in range(k)] if k % 7 else s


def _snap(xyz, box):
    if box > 0:
        u = torch.clamp(torch.floor(torch.remainder(xyz, box) / box * 4294967296.0), 0.0, 4294967295.0)
        return (u * (box / 4294967296.0)).contiguous()
    return (torch.round(xyz * 2.0 ** 20) / 2.0 ** 20).contiguous()


def _sector_dirs(g, n):
    """n points uniform in the sector: RA in [0, 60) deg, |Dec| < 30 deg, 500 < r < 1500."""
    u = torch.rand((n, 3), generator=g, device=DEV, dtype=torch.float64)
    ra, sd = u[:, 0] * (math.pi / 3), u[:, 1] - 0.5
    r = (500.0 ** 3 + u[:, 2] * (1500.0 ** 3 - 500.0 ** 3)) ** (1.0 / 3.0)
    cd = torch.sqrt(1 - sd * sd)
    return torch.stack([r * cd * torch.cos(ra), r * cd * torch.sin(ra), r * sd], 1)


def _clustered(g, parents, n):
    own = torch.randint(0, parents.shape[0], (n,), generator=g, device=DEV)
    return parents[own] + 5.0 * torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64)


def _catalogue(c, n, g):
    """(xyz, w) of one catalogue on the GPU: float64, on the fixed-point grid."""
    f64 = dict(generator=g, device=DEV, dtype=torch.float64)
    kind, box = c["points"], c.get("box", 0.0)
    if kind == "uniform":
        return _snap(torch.rand((n, 3), **f64) * box, box), torch.ones(n, device=DEV, dtype=torch.float64)
    if kind == "thomas":  # about 100 points a cluster, width 5; weights U[0.5, 1.5]
        xyz = _clustered(g, torch.rand((max(1, n // 100), 3), **f64) * box, n)
        return _snap(xyz, box), 0.5 + torch.rand(n, **f64)
    if kind == "sector":  # a quarter clustered data, the rest uniform randoms of the same total weight
        nd = n // 4
        data = _clustered(g, _sector_dirs(g, max(1, nd // 100)), nd)
        xyz = torch.cat([data, _sector_dirs(g, n - nd)])
        w = torch.ones(n, device=DEV, dtype=torch.float64)
        w[nd:] = -nd / (n - nd)
        return _snap(xyz, 0.0), w
    # sphere: golden-angle spiral, a smooth random field plus noise as pixel values
    k = torch.arange(n, device=DEV, dtype=torch.float64) + 0.5
    z, ph = 1 - 2 * k / n, k * (math.pi * (3 - math.sqrt(5.0)))
    r = torch.sqrt(torch.clamp(1 - z * z, min=0))
    xyz = _snap(torch.stack([r * torch.cos(ph), r * torch.sin(ph), z], 1), 0.0)
    cen = torch.randn((64, 3), **f64)
    cen /= cen.norm(dim=1, keepdim=True)
    amp = torch.randn(64, **f64)
    f = torch.cat([torch.exp(400.0 * (x @ cen.T - 1)) @ amp for x in xyz.split(1 << 20)])
    return xyz, f + 0.1 * torch.randn(n, **f64)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _primaries(c, g):
    """m distinct catalogue indices, sorted."""
    return torch.randperm(c["n"], generator=g, device=DEV)[: c["m"]].sort().values.contiguous()


def _inputs(c, seed):
    g = _gen(seed)
    if c["do"] == "contract":  # rows of a clustered catalogue fall with l and vary by primary
        nc = (c["lmax"] + 1) ** 2
        ell = torch.sqrt(torch.arange(nc, device=DEV, dtype=torch.float32)).floor()
        scale = 50.0 * torch.rand((c["m"], c["nbins"], 1), generator=g, device=DEV) + 1.0
        alm = torch.randn((c["m"], c["nbins"], nc), generator=g, device=DEV) * scale / (1.0 + ell)
        alm[:, :, 0] = 8.0 * scale[:, :, 0]
        return alm.contiguous(), 0.5 + torch.rand(c["m"], generator=g, device=DEV)
    if c["do"] == "edge":  # randoms: positive, falling with l; data minus randoms: small, both signs
        f64 = dict(generator=g, device=DEV, dtype=torch.float64)
        shape = (c["lmax"] + 1, c["nbins"], c["nbins"])
        ell = torch.arange(shape[0], device=DEV, dtype=torch.float64)[:, None, None]
        rrr = 1e9 * (0.8 + 0.4 * torch.rand(shape, **f64)) * torch.where(ell == 0, 1.0, 0.05 / (1 + ell))
        return 1e6 * torch.randn(shape, **f64) / (1 + ell), rrr
    if c["do"] == "batch":
        return [_catalogue(c, n, g) for n in _sizes(c)]
    return _catalogue(c, c["n"], g), _primaries(c, g) if "m" in c else None


def _estimator(c):
    if c["do"] == "sphere":
        est = ctb.CTB.sphere(math.radians(c["tmin"] / 60), math.radians(c["tmax"] / 60), c["nbins"], c["lmax"])
    else:
        est = ctb.CTB(c.get("box", 1000.0), c.get("rmin", 1.0), c.get("rmax", 100.0), c["nbins"], c["lmax"])
    if c.get("cells"):
        est.set_option(ctb.OPT_CELLS_PER_RMAX, c["cells"])
    if c.get("prec", "fp32") != "fp32":
        est.set_option(ctb.OPT_PRECISION, PRECISIONS[c["prec"]])
    return est


def prepare(case, seed):
    c, do = case, case["do"]
    if do == "contract":
        alm, w = _inputs(c, seed)
        out = torch.empty((c["lmax"] + 1, c["nbins"], c["nbins"]), device=DEV, dtype=torch.float64)
        return dict(c=c, alm=alm, w=w, out=out)
    s = dict(c=c, est=_estimator(c))
    if do == "edge":
        s["nnn"], s["rrr"] = _inputs(c, seed)
        s["out"] = torch.empty_like(s["nnn"])
        return s
    if do == "batch":
        s["cats"] = _inputs(c, seed)
        s["out"] = torch.empty((c["k"],) + s["est"].zeta_shape, device=DEV, dtype=torch.float64)
        return s
    (s["xyz"], s["w"]), s["idx"] = _inputs(c, seed)
    if do == "alm":  # the catalogue stays loaded while chosen primaries are looked at
        s["est"].set_points(s["xyz"], s["w"])
        s["out"] = torch.empty((c["m"], c["nbins"], s["est"].ncoef), device=DEV, dtype=torch.float32)
    elif c.get("host"):
        s["xyz"], s["w"] = s["xyz"].cpu().numpy(), s["w"].cpu().numpy()
    else:
        s["out"] = torch.empty(s["est"].zeta_shape, device=DEV, dtype=torch.float64)
    return s


def run(state):
    c, do = state["c"], state["c"]["do"]
    if do == "contract":
        ctb.contract_noalloc(state["alm"], state["w"], c["nbins"], c["lmax"], state["out"])
        return {"zeta": state["out"].float()}
    est = state["est"]
    if do == "edge":
        return {"zeta": est.edge_correct(state["nnn"], state["rrr"], out=state["out"])}
    if do == "batch":
        return {"zeta": est.compute_batch(state["cats"], out=state["out"]).float()}
    if do == "alm":
        return {"alm": est.get_alm(state["idx"], out=state["out"])}
    est.set_points(state["xyz"], state["w"])
    if c.get("host"):
        return {"zeta": est.compute().astype(np.float32), "pairs": est.pair_count()}
    if do == "subset":
        z = est.compute_subset(state["idx"], out=state["out"])
    elif do == "shared":
        z = est.compute_shared(c["h"], out=state["out"])
    else:
        z = est.compute(out=state["out"])
    return {"zeta": z.float(), "pairs": est.pair_count()}


# ---------------------------------------------------------------------------
# work

def _volume(c):
    return c["box"] ** 3 if c["box"] > 0 else math.pi / 3 * (1500.0 ** 3 - 500.0 ** 3) / 3


def _pairs(c):
    """Expected pairs at the mean density (a shared list counts once for its pivot cell)."""
    if c["do"] == "sphere":
        return c["n"] ** 2 * 0.5 * (math.cos(math.radians(c["tmin"] / 60)) - math.cos(math.radians(c["tmax"] / 60)))
    share = 4 / 3 * math.pi * (c["rmax"] ** 3 - c["rmin"] ** 3) / _volume(c)
    if c["do"] == "batch":
        return sum(n * n for n in _sizes(c)) * share
    np_ = c.get("m", c["n"])
    if c["do"] == "shared":
        h = c["h"] or (_volume(c) / c["n"]) ** (1 / 3)
        cells = _volume(c) / h ** 3
        np_ = cells * -math.expm1(-c["n"] / cells)  # occupied pivot cells of uniform points
        if c["points"] == "thomas":  # and of clusters of 100 points, width 5
            np_ = min(np_, c["n"] / 100 / (1 / 100 + 1 / (1 + 3 * (18 / h) ** 3)))
    return np_ * c["n"] * share


def _coefs(c):
    return 2 * c["lmax"] + 1 if c["do"] == "sphere" else (c["lmax"] + 1) ** 2


def _cost(c):
    return _pairs(c) * (_coefs(c) + 160.0)


def work(case):
    """One pass: one FMA per pair and coefficient, and per primary, coefficient
    and bin pair b1 <= b2 where a zeta is formed; inputs read and outputs
    written once."""
    c, do = case, case["do"]
    nb, L = c["nbins"], c["lmax"]
    zeta = (L + 1) * nb * nb
    per = _coefs(c) * nb * (nb + 1)  # 2 flops, half the bin pairs
    if do == "contract":
        return {"bytes": c["m"] * (nb * _coefs(c) + 1) * 4 + zeta * 8, "flops": c["m"] * per}
    if do == "edge":
        return {"bytes": 3 * zeta * 8, "flops": nb * nb * (2 * (L + 1) ** 3 + 2 / 3 * (L + 1) ** 3)}
    n = sum(_sizes(c)) if do == "batch" else c["n"]
    np_ = c.get("m", n)
    flops = 2.0 * _pairs(c) * _coefs(c)
    if do == "alm":
        return {"bytes": n * 16 + np_ * nb * _coefs(c) * 4, "flops": flops}
    return {"bytes": n * 32 + zeta * 8 * c.get("k", 1), "flops": flops + np_ * per}


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain torch

def _y_columns(d, r, L):
    """Real orthonormal Y_lm (Condon-Shortley phase) of the separations d,
    one column per l*l + l + m: the normalised associated-Legendre recurrence
    in z, times powers of x + iy."""
    x, y, z = (d / r[:, None]).unbind(1)
    out = torch.empty((d.shape[0], (L + 1) ** 2), device=d.device, dtype=torch.float64)
    re, im = torch.ones_like(x), torch.zeros_like(x)
    cmm = 1.0 / math.sqrt(4 * math.pi)
    for m in range(L + 1):
        if m:
            re, im = re * x - im * y, re * y + im * x
            cmm *= -math.sqrt((2 * m + 1) / (2 * m))
        p2, p1 = None, torch.full_like(z, cmm * (math.sqrt(2.0) if m else 1.0))
        for l in range(m, L + 1):
            if l > m:
                a = math.sqrt((4 * l * l - 1) / (l * l - m * m))
                p = z * p1
                if l > m + 1:
                    p = p - math.sqrt(((l - 1) ** 2 - m * m) / (4 * (l - 1) ** 2 - 1)) * p2
                p2, p1 = p1, a * p
            out[:, l * l + l + m] = p1 * re
            if m:
                out[:, l * l + l - m] = p1 * im
    return out


def _phase_columns(d, r, p, K):
    """cos and sin of m phi of the separations' projections on the tangent
    plane at p (east, north); columns 1, cos phi, sin phi, ..."""
    n = p / p.norm(dim=1, keepdim=True)
    rho = torch.sqrt(n[:, 0] ** 2 + n[:, 1] ** 2)
    ex, ey = -n[:, 1] / rho, n[:, 0] / rho
    u = ex * d[:, 0] + ey * d[:, 1]
    v = (-n[:, 2] * ey) * d[:, 0] + (n[:, 2] * ex) * d[:, 1] + rho * d[:, 2]
    ph = torch.atan2(u, v)
    cols = [torch.ones_like(ph)]
    for m in range(1, K + 1):
        cols += [torch.cos(m * ph), torch.sin(m * ph)]
    return torch.stack(cols, 1)


def _exact_alm(c, xyz, w, prim):
    """a_lm rows (or a_m on the sphere) of the primaries, a block at a time: (first, block)."""
    nb, L, box = c["nbins"], c["lmax"], c.get("box", 0.0)
    nc, sphere = _coefs(c), c["do"] == "sphere"
    if sphere:
        t0, t1 = math.radians(c["tmin"] / 60), math.radians(c["tmax"] / 60)
        edges = torch.tensor([2 * math.sin(0.5 * (t0 + b * (t1 - t0) / nb)) for b in range(nb + 1)], device=DEV,
                             dtype=torch.float64)
    else:
        dr = (c["rmax"] - c["rmin"]) / nb
        edges = torch.tensor([c["rmin"] + b * dr for b in range(nb)] + [c["rmax"]], device=DEV, dtype=torch.float64)
    e2 = edges * edges
    step = max(1, min(int(2e8 // xyz.shape[0]), 4096))
    cut = max(1, int(4e8 // nc))
    for p0 in range(0, prim.shape[0], step):
        pr = prim[p0: p0 + step]
        r2 = torch.zeros((pr.shape[0], xyz.shape[0]), device=DEV, dtype=torch.float64)
        for k in range(3):
            d = xyz[None, :, k] - xyz[pr, k][:, None]
            if box > 0:
                d -= box * torch.round(d / box)
            r2 += d * d
        pi, j = torch.nonzero((r2 >= e2[0]) & (r2 < e2[-1]) & (r2 > 0), as_tuple=True)
        rr = r2[pi, j]
        del r2, d
        seg = pi * nb + (torch.searchsorted(e2, rr, right=True) - 1)
        order = torch.argsort(seg, stable=True)
        pi, j, rr, seg = pi[order], j[order], rr[order], seg[order]
        a = torch.zeros((pr.shape[0] * nb, nc), device=DEV, dtype=torch.float64)
        for q0 in range(0, seg.shape[0], cut):
            q = slice(q0, min(q0 + cut, seg.shape[0]))
            d = xyz[j[q]] - xyz[pr[pi[q]]]
            if box > 0:
                d -= box * torch.round(d / box)
            y = (_phase_columns(d, rr[q], xyz[pr[pi[q]]], L) if sphere
                 else _y_columns(d, torch.sqrt(rr[q]), L)) * w[j[q]][:, None]
            ids, cnt = torch.unique_consecutive(seg[q], return_counts=True)
            a[ids] += torch.segment_reduce(y, "sum", lengths=cnt)
        yield p0, a.view(pr.shape[0], nb, nc)


def _exact_zeta(c, xyz, w, prim):
    nb, L = c["nbins"], c["lmax"]
    z = torch.zeros((L + 1, nb, nb), device=DEV, dtype=torch.float64)
    for p0, a in _exact_alm(c, xyz, w, prim):
        wa = a * w[prim[p0: p0 + a.shape[0]]][:, None, None]
        _add_zeta(z, a, wa, c["do"] == "sphere")
    return z


def _add_zeta(z, a, wa, sphere=False):
    for l in range(z.shape[0]):
        lo, hi = (max(0, 2 * l - 1), 2 * l + 1) if sphere else (l * l, (l + 1) ** 2)
        f = 1.0 if sphere else 4 * math.pi / (2 * l + 1)
        x, y = (t[:, :, lo:hi].permute(1, 0, 2).reshape(z.shape[1], -1) for t in (wa, a))
        z[l] += f * (x @ y.T)


def _exact_edge(c, nnn, rrr):
    """n_l / r_0 = sum_l' M_ll' zeta_l', M_ll' = (2l+1) sum_l'' (l l' l''; 000)^2 f_l'',
    the squared 3j symbols as half the integral of three Legendre polynomials."""
    n = c["lmax"] + 1
    mu, wt = np.polynomial.legendre.leggauss(2 * n)
    P = np.stack([np.polynomial.legendre.Legendre.basis(l)(mu) for l in range(n)])
    tj = np.einsum("aq,bq,cq,q->abc", P, P, P, 0.5 * wt)
    norm = (0.5 * (2 * np.arange(n) + 1))[:, None, None]
    nn, rr = norm * nnn.cpu().numpy(), norm * rrr.cpu().numpy()
    M = np.einsum("abc,cxy->xyab", tj, rr / rr[0]) * (2 * np.arange(n) + 1)[:, None]
    return np.linalg.solve(M, (nn / rr[0]).transpose(1, 2, 0)[..., None])[..., 0].transpose(2, 0, 1).copy()


def exact(case, seed):
    c, do = case, case["do"]
    if do == "shared":  # an approximation by its own definition of groups: no independent value
        return None
    if do == "edge":
        return {"zeta": _exact_edge(c, *_inputs(c, seed))}
    if do == "contract":
        alm, w = _inputs(c, seed)
        z = torch.zeros((c["lmax"] + 1, c["nbins"], c["nbins"]), device=DEV, dtype=torch.float64)
        for a, v in zip(alm.split(4096), w.split(4096)):
            _add_zeta(z, a.double(), a.double() * v.double()[:, None, None])
        return {"zeta": z}
    # brute force: too long for the largest
    far = sum(n * n for n in _sizes(c)) if do == "batch" else c["n"] * c.get("m", c["n"])
    if far > 6e10 or _pairs(c) * _coefs(c) > 1.2e11:
        return None
    if do == "batch":
        return {"zeta": torch.stack([_exact_zeta(c, x, w.float().double(), torch.arange(x.shape[0], device=DEV))
                                     for x, w in _inputs(c, seed)])}
    (xyz, w), idx = _inputs(c, seed)
    w = w.float().double()  # the library stores weights in float32
    if do == "alm":
        out = torch.empty((c["m"], c["nbins"], _coefs(c)), device=DEV, dtype=torch.float64)
        for p0, a in _exact_alm(c, xyz, w, idx):
            out[p0: p0 + a.shape[0]] = a
        return {"alm": out}
    prim = idx if do == "subset" else torch.arange(c["n"], device=DEV)
    return {"zeta": _exact_zeta(c, xyz, w, prim), "pairs": None}
