"""Measured cases of the Lyman-alpha pixel-pair library.

Every case is one call sequence that a program using this library makes
through ``paper_2507_00129_gb300.api``, on catalogues of the repository's own
workloads (``synth.spec_for``): the SDSS-DR16-like log10 grid (natural forest
lengths, about 190 pixels) and the DESI-like linear grid (100-600 pixels), at
their sky densities of 24 to 60 forests per square degree.

The pixel deltas are what the estimators are run on in earnest: a large-scale
field that is correlated in three dimensions (a sum of plane waves with
wavelengths of 50 to 300 Mpc/h, the same for all forests), plus white pixel
noise.  Weights are inverse pixel variances with the log-normal scatter of the
synthetic workloads.  Everything is drawn on the GPU from the seed alone.

``exact`` restates each estimator in plain torch, in 64 bits, without the
library: brute-force forest pairs, padded pixel blocks and dense sums.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2507_00129_gb300 import api

C_OVER_H0 = 2997.92458      # Mpc/h
OMEGA_M = 0.315
LYA = 1215.67               # Angstrom
RF_MIN, RF_MAX = 1040.0, 1200.0
LAM_MIN = 3600.0
DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a field of 200 forests (the tiny workload) whose geometry is kept, as in a loop
        # over sets of deltas; launches and latency count
        dict(name="xi_field_200", kind="xi_kept", grid="log10", n=200, area=9.0, n_par=25, n_perp=25, r_max=100.0),
        # one measurement of a survey: projection, neighbour list and xi/W of the whole SDSS-like catalogue
        dict(name="xi_survey_sdss_60000", kind="xi_step", grid="log10", n=60000, area=2500.0, n_par=50, n_perp=50,
             r_max=200.0),
        # the same on the DESI-like grid, at the size of one mock catalogue and the DESI-Y5-like sky density
        dict(name="xi_survey_desi_9000", kind="xi_step", grid="linear", n=9000, area=150.0, n_par=50, n_perp=50,
             r_max=200.0),
        # the plain 64-bit path, which checks a measurement on a part of the sky
        dict(name="xi_fp64_sdss_3000", kind="xi_fp64", grid="log10", n=3000, area=125.0, n_par=50, n_perp=50,
             r_max=200.0),
        # distortion matrix on a 5% sub-sample of the forest pairs
        dict(name="dmat_sdss_12000", kind="dmat", grid="log10", n=12000, area=500.0, n_par=50, n_perp=50,
             r_max=200.0, p=0.05),
        # one step of a fit through xi: forward and gradient with respect to deltas and weights, geometry kept
        dict(name="grad_desi_4000", kind="grad", grid="linear", n=4000, area=160.0, n_par=50, n_perp=50,
             r_max=200.0),
        # a batch of mocks in one call: xi/W and distortion matrices
        dict(name="mocks_desi_6x1500", kind="mocks", grid="linear", n=1500, area=60.0, n_par=50, n_perp=50,
             r_max=200.0, m=6, p=0.02),
        # covariance from HEALPix sub-samples
        dict(name="covariance_sdss_15000", kind="cov", grid="log10", n=15000, area=625.0, n_par=50, n_perp=50,
             r_max=200.0, nside=8),
        # per-bin means and counts for the export to a fit
        dict(name="bin_means_sdss_15000", kind="means", grid="log10", n=15000, area=625.0, n_par=50, n_perp=50,
             r_max=200.0),
        # forest x quasar cross-correlation and its distortion matrix, full catalogue
        dict(name="cross_sdss_60000", kind="cross", grid="log10", n=60000, area=2500.0, n_par=100, n_perp=50,
             r_max=200.0, p=0.02),
        # three-point function on the 200,000-bin triangle grid
        dict(name="xi3_sdss_5000", kind="xi3", grid="log10", n=5000, area=208.0, n_r=10, n_theta=10, n_alpha=20,
             r_max=40.0),
        # same-forest correlation of the full catalogue
        dict(name="xi1d_sdss_60000", kind="xi1d", grid="log10", n=60000, area=2500.0, n_bins=50, r_max=200.0),
    ]


#: kind -> (smallest and largest number of forests) of the drawn cases
RANGES = {"xi_kept": (150, 3000), "xi_step": (1000, 50000), "xi_fp64": (400, 3000), "dmat": (3000, 12000),
          "grad": (600, 4000), "mocks": (400, 1500), "cov": (2000, 15000), "means": (2000, 15000),
          "cross": (3000, 60000), "xi3": (800, 5000), "xi1d": (2000, 60000)}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(sorted(RANGES))
    n = _log(rng, *RANGES[kind])
    grid = "linear" if kind in ("grad", "mocks") else "log10"
    density = rng.uniform(20.0, 30.0)
    if kind in ("xi_kept", "xi_step", "xi_fp64") and rng.random() < 0.5:
        grid, n = "linear", max(RANGES[kind][0], n // 5)
        density = rng.uniform(20.0, 60.0)
    case = dict(kind=kind, grid=grid, n=n, area=round(n / density, 3))
    if kind == "xi1d":
        return dict(case, n_bins=rng.randint(20, 200), r_max=rng.choice([80.0, 150.0, 200.0]))
    if kind == "xi3":
        return dict(case, n_r=rng.randint(5, 10), n_theta=rng.randint(4, 10), n_alpha=rng.randint(8, 20),
                    r_max=rng.choice([24.0, 32.0, 40.0]))
    r_max = rng.choice([100.0, 150.0, 200.0]) if kind in ("xi_kept", "xi_fp64", "grad") else 200.0
    case.update(n_par=rng.randint(25, 50), n_perp=rng.randint(25, 50), r_max=r_max)
    if kind == "dmat":
        case["p"] = round(rng.uniform(0.03, 0.05), 4)
    elif kind == "mocks":
        case.update(m=rng.randint(2, 6), p=round(rng.uniform(0.01, 0.02), 4))
    elif kind == "cov":
        case["nside"] = rng.choice([4, 8])
    elif kind == "cross":
        case.update(n_par=2 * case["n_par"], p=round(rng.uniform(0.01, 0.02), 4))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_GRID = {}


def _wavelengths(grid):
    """Observed wavelengths of the pixel grid and their comoving distances (flat LCDM), on the GPU."""
    if grid not in _GRID:
        lam_max = RF_MAX * 4.5
        if grid == "log10":
            k = torch.arange(1, int((math.log10(lam_max) - math.log10(LAM_MIN)) / 3e-4) + 2, dtype=torch.float64)
            lam = 10.0 ** (math.log10(LAM_MIN) + 3e-4 * k)
        else:
            lam = LAM_MIN + 0.8 * torch.arange(1, int((lam_max - LAM_MIN) / 0.8) + 2, dtype=torch.float64)
        z = torch.linspace(0.0, lam_max / LYA, 40001, dtype=torch.float64)   # Simpson on a fine grid, then cubic
        inv_e = lambda t: 1.0 / torch.sqrt(OMEGA_M * (1.0 + t) ** 3 + (1.0 - OMEGA_M))   # noqa: E731
        h = z[1] - z[0]
        step = h / 6.0 * (inv_e(z[:-1]) + 4.0 * inv_e(z[:-1] + 0.5 * h) + inv_e(z[1:]))
        chi = torch.cat([torch.zeros(1, dtype=torch.float64), torch.cumsum(step, 0)])
        zl = lam / LYA - 1.0
        i = (zl / h).long().clamp(0, z.numel() - 2)
        t = zl - z[i]
        d = chi[i] + t / 6.0 * (inv_e(z[i]) + 4.0 * inv_e(z[i] + 0.5 * t) + inv_e(zl))
        _GRID[grid] = (lam.to(DEV), (d * C_OVER_H0).to(DEV))
    return _GRID[grid]


def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _field(g, ra, dec, dist, n_pix_forest):
    """Large-scale field at every pixel: 32 plane waves, amplitude 0.1 rms."""
    kk = 2.0 * math.pi / _uniform(g, 32, 50.0, 300.0)
    ck = _uniform(g, 32, -1.0, 1.0)
    ph = _uniform(g, 32, 0.0, 2.0 * math.pi)
    az = _uniform(g, 32, 0.0, 2.0 * math.pi)
    sk = torch.sqrt(1.0 - ck * ck)
    cd = torch.cos(dec)
    out = torch.zeros_like(dist)
    for m in range(32):
        proj = kk[m] * (cd * torch.cos(ra) * sk[m] * torch.cos(az[m]) + cd * torch.sin(ra) * sk[m] * torch.sin(az[m])
                        + torch.sin(dec) * ck[m])
        out += torch.cos((dist * torch.repeat_interleave(proj, n_pix_forest) + ph[m]).float()).double()
    return out * (0.1 * math.sqrt(2.0 / 32))


def _catalog(case, seed):
    """Tensors of a catalogue: a spherical cap of the case's area, quasar redshifts 2.1-3.5, the forest window
    1040-1200 A of the rest frame; on the linear grid a window of 100-600 pixels and a continuum tilt."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["n"]
    lam, chi = _wavelengths(case["grid"])
    cos_t = 1.0 - case["area"] * (math.pi / 180.0) ** 2 / (2.0 * math.pi)
    # the survey's redshifts and forest windows are the case's own (so that every seed has as many pixels), dealt
    # to the sky positions in the seed's order
    own = torch.Generator(device=DEV).manual_seed(20250700129)
    zq = _uniform(own, n, 2.1, 3.5)
    lo = torch.searchsorted(lam, RF_MIN * (1.0 + zq))
    length = torch.searchsorted(lam, RF_MAX * (1.0 + zq), right=True) - lo
    if case["grid"] == "linear":
        keep = torch.minimum(torch.randint(100, 601, (n,), generator=own, device=DEV), length)
        lo = lo + (torch.rand(n, generator=own, device=DEV, dtype=torch.float64) * (length - keep + 1)).long()
        length = keep
    deal = torch.randperm(n, generator=g, device=DEV)
    zq, lo, length = zq[deal], lo[deal], length[deal]
    ra = _uniform(g, n, 0.0, 2.0 * math.pi)
    dec = torch.asin(_uniform(g, n, cos_t, 1.0))
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(length, 0, out=offsets[1:])
    n_pix = int(offsets[-1])
    f = torch.repeat_interleave(torch.arange(n, device=DEV), length)
    k = lo[f] + (torch.arange(n_pix, device=DEV) - offsets[f])
    dist, loglam = chi[k], torch.log(lam[k])
    sigma = torch.exp(math.log(0.15) + 0.3 * torch.randn(n_pix, generator=g, device=DEV, dtype=torch.float64))
    weight = (1.0 / sigma ** 2).float()
    delta = 0.2 * torch.randn(n_pix, generator=g, device=DEV, dtype=torch.float64)
    delta += _field(g, ra, dec, dist, length)
    if case["grid"] == "linear":
        a = 0.1 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
        b = torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
        delta += a[f] + b[f] * (loglam - torch.log(0.5 * (RF_MIN + RF_MAX) * (1.0 + zq))[f])
    return SimpleNamespace(n=n, offsets=offsets, ra=ra, dec=dec, dist=dist, loglam=loglam, delta=delta.float(),
                           weight=weight, zq=zq, gen=g)


def _device(c):
    return api.DeviceCatalog(c.offsets, c.ra, c.dec, c.dist, c.loglam, c.delta, c.weight)


def _bins(case):
    return SimpleNamespace(n_par=case["n_par"], n_perp=case["n_perp"], r_par_max=case["r_max"],
                           r_perp_max=case["r_max"])


def _quasars(case, c):
    """Each forest's own quasar and half as many more, z 1.8-3.5, weights ((1 + z) / 3.25)^0.44."""
    n, extra = case["n"], case["n"] // 2
    cos_t = 1.0 - case["area"] * (math.pi / 180.0) ** 2 / (2.0 * math.pi)
    ra = torch.cat([c.ra, _uniform(c.gen, extra, 0.0, 2.0 * math.pi)])
    dec = torch.cat([c.dec, torch.asin(_uniform(c.gen, extra, cos_t, 1.0))])
    z = torch.cat([c.zq, _uniform(c.gen, extra, 1.8, 3.5)])
    grid = torch.linspace(1.7, 3.6, 20001, dtype=torch.float64, device=DEV)
    inv_e = 1.0 / torch.sqrt(OMEGA_M * (1.0 + grid) ** 3 + (1.0 - OMEGA_M))
    h = float(grid[1] - grid[0])
    zz = torch.linspace(0.0, 1.7, 20001, dtype=torch.float64, device=DEV)
    base = torch.trapezoid(1.0 / torch.sqrt(OMEGA_M * (1.0 + zz) ** 3 + (1.0 - OMEGA_M)), zz)
    chi = base + torch.cat([torch.zeros(1, device=DEV, dtype=torch.float64),
                            torch.cumsum(0.5 * h * (inv_e[1:] + inv_e[:-1]), 0)])
    i = ((z - 1.7) / h).long().clamp(0, 19999)
    d = (chi[i] + (z - grid[i]) / h * (chi[i + 1] - chi[i])) * C_OVER_H0
    w = (((1.0 + z) / 3.25) ** 0.44).float()
    return SimpleNamespace(ra=ra, dec=dec, dist=d, weight=w, own=torch.arange(n, dtype=torch.int64, device=DEV))


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case, kind=kind, handle=api.Handle())
    if kind == "mocks":
        s.mocks = [_device(_catalog(case, seed * 1000 + k)) for k in range(case["m"])]
        s.bins = _bins(case)
        return s
    c = _catalog(case, seed)
    s.cat = _device(c)
    if kind == "xi3":
        s.grid = SimpleNamespace(n_r=case["n_r"], n_theta=case["n_theta"], n_alpha=case["n_alpha"],
                                 r_max=case["r_max"])
        return s
    if kind == "xi1d":
        return s
    s.bins = _bins(case)
    if kind == "cross":
        q = _quasars(case, c)
        s.qso, s.own = api.DeviceQuasars(q.ra, q.dec, q.dist, q.weight), q.own
    if kind == "means":
        s.z = torch.exp(c.loglam) / LYA - 1.0
    if kind == "grad":
        s.gx, s.gw = _loss(case, c)
        s.delta = s.cat.delta.clone().requires_grad_()
        s.weight = s.cat.weight.clone().requires_grad_()
    if kind in ("xi_kept", "grad", "dmat", "xi_fp64"):
        api.lya_pairs_build(s.handle, s.cat, s.bins)   # the geometry that such a program keeps
    return s


def _loss(case, c):
    """Gradient of the program's loss with respect to xi and W."""
    nb = case["n_par"] * case["n_perp"]
    g = torch.randn(nb, generator=c.gen, device=DEV, dtype=torch.float64)
    return g, 1e-9 * torch.randn(nb, generator=c.gen, device=DEV, dtype=torch.float64)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    h, kind, case = s.handle, s.kind, s.case
    if kind == "xi_kept":
        d = api.lya_project(h, s.cat)
        num, w, xi = api.lya_xi(h, s.cat.with_(delta=d), s.bins)
        return {"delta": d, "num": num, "w": w, "xi": xi}
    if kind == "xi_step":
        d = api.lya_project(h, s.cat)
        cat = s.cat.with_(delta=d)
        n = api.lya_pairs_build(h, cat, s.bins)
        num, w, xi = api.lya_xi(h, cat, s.bins)
        return {"delta": d, "pairs": n, "num": num, "w": w, "xi": xi}
    if kind == "xi_fp64":
        num, w, xi = api.lya_xi(h, s.cat, s.bins, "fp64")
        return {"num": num, "w": w, "xi": xi}
    if kind == "dmat":
        D, w = api.lya_dmat(h, s.cat, s.bins, case["p"], 1234)
        return {"d": D, "w": w}
    if kind == "grad":
        s.delta.grad = s.weight.grad = None
        xi, w = api.xi(s.cat, s.bins, h, delta=s.delta, weight=s.weight)
        ((xi * s.gx).sum() + (w * s.gw).sum()).backward()
        return {"xi": xi, "w": w, "grad_delta": s.delta.grad, "grad_weight": s.weight.grad}
    if kind == "mocks":
        num, w, xi = api.lya_xi_batched(h, s.mocks, s.bins)
        D, wd = api.lya_dmat_batched(h, s.mocks, s.bins, case["p"], 1234)
        return {"num": num, "w": w, "xi": xi, "d": D, "wd": wd}
    if kind == "cov":
        num, w, xi, sub = api.lya_xi_subsamples(h, s.cat, s.bins, case["nside"])
        cov, full = api.lya_xi_covariance(h, num, w)
        return {"num": num, "w": w, "xi": xi, "sub": sub, "cov": cov, "full": full}
    if kind == "means":
        return api.lya_xi_bin_means(h, s.cat, s.bins, z_pix=s.z)
    if kind == "cross":
        num, w, xi = api.lya_xcf(h, s.cat, s.qso, s.bins, s.own)
        D, wd = api.lya_xdmat(h, s.cat, s.qso, s.bins, case["p"], 1234, s.own)
        return {"num": num, "w": w, "xi": xi, "d": D, "wd": wd}
    if kind == "xi3":
        num, w, xi = api.lya_xi3(h, s.cat, s.grid)
        return {"num": num, "w": w, "xi": xi}
    num, w, xi = api.lya_xi1d(h, s.cat, case["n_bins"], case["r_max"])
    return {"num": num, "w": w, "xi": xi}


# ---------------------------------------------------------------------------
# work of one pass, estimated from the sizes
# ---------------------------------------------------------------------------
def _cap_fraction(case, r):
    """Share of a disc of radius r (Mpc/h, at 4200 Mpc/h) around a forest that lies in the cap, on average."""
    cap = math.sqrt(case["area"] / math.pi) * math.pi / 180.0 * 4200.0
    return 1.0 / (1.0 + 0.85 * r / cap)


def _pixel_pairs(case):
    """In-grid pixel pairs of the auto-correlation, from the sky density (the constants are the counts of the
    60,000-forest SDSS-like and the 15,000-forest DESI-like workloads at 200 Mpc/h)."""
    c = 1.62e5 if case["grid"] == "log10" else 5.2e5
    r = case["r_max"] / 200.0
    return c * case["n"] * case["n"] / case["area"] * r ** 2.8 * _cap_fraction(case, case["r_max"])


def work(case):
    kind = case["kind"]
    pix = case["n"] * (190 if case["grid"] == "log10" else 335)
    catalog = 24.0 * pix + 24.0 * case["n"]
    nb = case.get("n_par", 0) * case.get("n_perp", 0)
    if kind == "xi1d":
        return {"bytes": catalog + 24.0 * case["n_bins"], "flops": 6.0 * pix * 70 * case["r_max"] / 200.0}
    if kind == "xi3":
        bins = case["n_r"] ** 2 * case["n_alpha"] * case["n_theta"] ** 2
        near = 2.0 * _pixel_pairs(dict(case, n_par=1, n_perp=1)) / pix   # neighbours of a pixel within r_max
        return {"bytes": catalog + 24.0 * bins, "flops": 10.0 * pix * near * near / 2.0}
    if kind == "cross":
        pairs = 3.1e7 * (case["n"] / 60000.0) ** 2 * 2500.0 / case["area"]
        return {"bytes": catalog + 48.0 * case["n"] + 24.0 * nb + 8.0 * nb * nb, "flops": 8.0 * 100 * pairs}
    pp = _pixel_pairs(case)
    out = {"xi_kept": 8.0 * pix + 24 * nb, "xi_step": 8.0 * pix + 24 * nb, "xi_fp64": 24.0 * nb,
           "dmat": 8.0 * nb * nb, "grad": 8.0 * pix, "mocks": 8.0 * nb * nb, "means": 48.0 * nb,
           "cov": 24.0 * 12 * case.get("nside", 0) ** 2 * nb + 8.0 * nb * nb}[kind]
    # per pixel pair: two separations, two products, two sums; the distortion matrix adds about 220 operations per
    # pixel pair of its sub-sample (closed form), the gradient visits each pair from both sides
    flops = {"dmat": 220.0 * case.get("p", 0), "grad": 24.0, "mocks": 8.0 + 220.0 * case.get("p", 0), "means": 14.0}
    m = case.get("m", 1)
    return {"bytes": m * (catalog + out), "flops": m * pp * flops.get(kind, 8.0)}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _unit(ra, dec):
    cd = torch.cos(dec)
    return torch.stack([cd * torch.cos(ra), cd * torch.sin(ra), torch.sin(dec)], 1)


def _padded(c, values):
    """[n, L] of a flat pixel array, and the mask of the real pixels."""
    length = c.offsets[1:] - c.offsets[:-1]
    k = torch.arange(int(length.max()), device=DEV)
    mask = k[None, :] < length[:, None]
    idx = (c.offsets[:-1, None] + k[None, :]).clamp(max=values.numel() - 1)
    return values[idx].masked_fill(~mask, 0.0), mask


def _project(c, delta):
    """Equation (2.7) on every forest, 64 bits."""
    w, mask = _padded(c, c.weight.double())
    x, _ = _padded(c, c.loglam)
    d, _ = _padded(c, delta.double())
    sw = w.sum(1, keepdim=True)
    x = (x - (w * x).sum(1, keepdim=True) / sw).masked_fill(~mask, 0.0)
    out = d - (w * d).sum(1, keepdim=True) / sw - x * (w * x * d).sum(1, keepdim=True) / (w * x * x).sum(1, keepdim=True)
    return out[mask]


def _forest_pairs(c, r_perp):
    """(a, b), a < b, with (d_first,a + d_first,b) sin(theta/2) < r_perp, and cos, sin of theta/2."""
    u = _unit(c.ra, c.dec)
    d0 = c.dist[c.offsets[:-1]]
    got = []
    step = max(1, 20_000_000 // c.n)
    for lo in range(0, c.n, step):
        hi = min(c.n, lo + step)
        s = 0.5 * (u[lo:hi, None, :] - u[None, :, :]).norm(dim=2)
        ok = (d0[lo:hi, None] + d0[None, :]) * s < r_perp
        a, b = ok.nonzero(as_tuple=True)
        a = a + lo
        got.append(torch.stack([a[a < b], b[a < b]]))
    a, b = torch.cat(got, 1)
    return a, b, 0.5 * (u[a] + u[b]).norm(dim=1), 0.5 * (u[a] - u[b]).norm(dim=1)


def _blocks(case, c):
    """Blocks of forest pairs: (a, b, c, s, distances of a and b, bin index [P, L, L], nb where off the grid)."""
    dist, mask = _padded(c, c.dist)
    a, b, cc, ss = _forest_pairs(c, case["r_max"])
    n_par, n_perp = case["n_par"], case["n_perp"]
    nb, width = n_par * n_perp, dist.shape[1]
    step = max(1, 12_000_000 // (width * width))
    for lo in range(0, a.numel(), step):
        i, j = a[lo:lo + step], b[lo:lo + step]
        da, db = dist[i][:, :, None], dist[j][:, None, :]
        x = (da - db).abs() * cc[lo:lo + step, None, None] * (n_par / case["r_max"])
        y = (da + db) * ss[lo:lo + step, None, None] * (n_perp / case["r_max"])
        ok = (x < n_par) & (y < n_perp) & mask[i][:, :, None] & mask[j][:, None, :]
        yield i, j, x, y, da, db, torch.where(ok, x.long() * n_perp + y.long(), nb)


def _ratio(n, w):
    return torch.where(w != 0, n / torch.where(w != 0, w, torch.ones_like(w)), torch.zeros_like(n))


def _sums(case, c, wd, rows=None, n_rows=1):
    """Sums of Eq. (2.4); with `rows` one set per row of the pair's first forest."""
    nb = case["n_par"] * case["n_perp"]
    w, _ = _padded(c, c.weight.double())
    v, _ = _padded(c, wd)
    num = torch.zeros(n_rows * (nb + 1), dtype=torch.float64, device=DEV)
    den = torch.zeros_like(num)
    for i, j, _x, _y, _da, _db, k in _blocks(case, c):
        if rows is not None:
            k = k + rows[i][:, None, None] * (nb + 1)
        num += torch.bincount(k.reshape(-1), (v[i][:, :, None] * v[j][:, None, :]).reshape(-1), num.numel())
        den += torch.bincount(k.reshape(-1), (w[i][:, :, None] * w[j][:, None, :]).reshape(-1), num.numel())
    num, den = (t.view(n_rows, nb + 1)[:, :nb] for t in (num, den))
    return (num[0], den[0]) if rows is None else (num.contiguous(), den.contiguous())


def _too_many(case):
    """Whether the padded pixel pairs take longer than about 15 seconds."""
    width = 330 if case["grid"] == "log10" else 600
    pad = 2.4 if case["grid"] == "log10" else 4.0
    return _pixel_pairs(case) * pad * case.get("m", 1) * (2 if case["kind"] == "grad" else 1) > 2.5e10 or width > 2000


def _exact_grad(case, c):
    nb = case["n_par"] * case["n_perp"]
    gx, gw = _loss(case, c)
    w, mask = _padded(c, c.weight.double())
    d, _ = _padded(c, c.delta.double())
    num, den = _sums(case, c, c.weight.double() * c.delta.double())
    xi = _ratio(num, den)
    zero = torch.zeros(1, dtype=torch.float64, device=DEV)
    gamma = torch.cat([_ratio(gx, den), zero])
    rho = torch.cat([_ratio(gx, den) * xi - gw, zero])
    s1, s2 = torch.zeros_like(w), torch.zeros_like(w)
    for i, j, _x, _y, _da, _db, k in _blocks(case, c):
        for out, tab, v in ((s1, gamma, w * d), (s2, rho, w)):
            t = tab[k]
            out.index_add_(0, i, torch.bmm(t, v[j][:, :, None])[:, :, 0])
            out.index_add_(0, j, torch.bmm(v[i][:, None, :], t)[:, 0, :])
    return {"xi": xi, "w": den, "grad_delta": (w * s1)[mask], "grad_weight": (d * s1 - s2)[mask]}


def _exact_means(case, c):
    nb = case["n_par"] * case["n_perp"]
    w, _ = _padded(c, c.weight.double())
    z, _ = _padded(c, torch.exp(c.loglam) / LYA - 1.0)
    acc = torch.zeros(5, nb + 1, dtype=torch.float64, device=DEV)
    for i, j, x, y, da, db, k in _blocks(case, c):
        ww = w[i][:, :, None] * w[j][:, None, :]
        k = k.reshape(-1)
        for q, v in enumerate((None, x, y, 0.5 * (da + db), 0.5 * (z[i][:, :, None] + z[j][:, None, :]))):
            acc[q] += torch.bincount(k, (ww if v is None else ww * v).reshape(-1), nb + 1)
    acc = acc[:, :nb]
    return {"wsum": acc[0], "rpar_mean": _ratio(acc[1], acc[0]) * (case["r_max"] / case["n_par"]),
            "rperp_mean": _ratio(acc[2], acc[0]) * (case["r_max"] / case["n_perp"]),
            "dist_mean": _ratio(acc[3], acc[0]), "z_mean": _ratio(acc[4], acc[0]), "count": None}


def _exact_cross(case, c):
    q = _quasars(case, c)
    n_par, n_perp, r = case["n_par"], case["n_perp"], case["r_max"]
    nb = n_par * n_perp
    dist, mask = _padded(c, c.dist)
    w, _ = _padded(c, c.weight.double())
    v, _ = _padded(c, c.weight.double() * c.delta.double())
    uf, uq = _unit(c.ra, c.dec), _unit(q.ra, q.dec)
    d0 = c.dist[c.offsets[:-1]]
    num = torch.zeros(nb + 1, dtype=torch.float64, device=DEV)
    den = torch.zeros_like(num)
    step = max(1, 20_000_000 // uq.shape[0])
    for lo in range(0, c.n, step):
        hi = min(c.n, lo + step)
        cut = (2.0 - 2.0 * uf[lo:hi] @ uq.T).clamp_(min=0.0).sqrt_().mul_(0.5) * (d0[lo:hi, None] + q.dist[None, :])
        f, k = (cut < r + 0.1).nonzero(as_tuple=True)
        f = f + lo
        f, k = f[q.own[f] != k], k[q.own[f] != k]
        for p in range(0, f.numel(), 60000):
            a, b = f[p:p + 60000], k[p:p + 60000]
            cc = 0.5 * (uf[a] + uq[b]).norm(dim=1, keepdim=True)
            ss = 0.5 * (uf[a] - uq[b]).norm(dim=1, keepdim=True)
            dq = q.dist[b][:, None]
            x = ((dist[a] - dq) * cc + r) * (n_par / (2.0 * r))
            y = (dist[a] + dq) * ss * (n_perp / r)
            ok = (x >= 0) & (x < n_par) & (y < n_perp) & mask[a]
            idx = torch.where(ok, x.long() * n_perp + y.long(), nb).reshape(-1)
            wq = q.weight[b].double()[:, None]
            num += torch.bincount(idx, (v[a] * wq).reshape(-1), nb + 1)
            den += torch.bincount(idx, (w[a] * wq).reshape(-1), nb + 1)
    num, den = num[:nb], den[:nb]
    return {"num": num, "w": den, "xi": _ratio(num, den), "d": None, "wd": None}


def _exact_1d(case, c):
    n = case["n_bins"]
    dist, mask = _padded(c, c.dist)
    w, _ = _padded(c, c.weight.double())
    v, _ = _padded(c, c.weight.double() * c.delta.double())
    num = torch.zeros(n + 1, dtype=torch.float64, device=DEV)
    den = torch.zeros_like(num)
    for lag in range(1, dist.shape[1]):
        # the pixels `lag` apart in every forest; beyond the range for all once the gap is too wide
        p = ((dist[:, lag:] - dist[:, :-lag]) / (case["r_max"] / n)).floor()
        ok = mask[:, lag:] & (p < n)
        if not bool(ok.any()):
            break
        idx = torch.where(ok, p, float(n)).long().reshape(-1)
        num += torch.bincount(idx, (v[:, lag:] * v[:, :-lag]).reshape(-1), n + 1)
        den += torch.bincount(idx, (w[:, lag:] * w[:, :-lag]).reshape(-1), n + 1)
    return {"num": num[:n], "w": den[:n], "xi": _ratio(num[:n], den[:n])}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dmat", "xi3", "mocks", "cov"):
        return None   # the plain quadruple sum, the sum over triplets and the large pair sums take minutes
    if kind not in ("xi1d", "cross") and _too_many(case):
        return None
    c = _catalog(case, seed)
    if kind == "xi1d":
        return _exact_1d(case, c)
    if kind == "cross":
        return _exact_cross(case, c)
    if kind == "grad":
        return _exact_grad(case, c)
    if kind == "means":
        return _exact_means(case, c)
    delta = c.delta.double() if kind == "xi_fp64" else _project(c, c.delta)
    num, w = _sums(case, c, c.weight.double() * delta)
    out = {"num": num, "w": w, "xi": _ratio(num, w)}
    return out if kind == "xi_fp64" else dict(out, delta=delta, pairs=None)
