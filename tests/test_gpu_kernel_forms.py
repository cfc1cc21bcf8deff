"""The kernels' forms at the sizes where they change: edges of tiles and of
chunks, remainders, and pixel pairs exactly on bin edges, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from conftest import line_catalog  # noqa: E402
from paper_2507_00129_gb300 import synth  # noqa: E402


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_00129_gb300 import api as a, build
    build.build()
    return a


@pytest.fixture()
def handle(api):
    with api.Handle() as h:
        yield h


def _catalog(lengths, step, seed, patch=2e-3):
    """Forests of the given lengths in a patch of `patch` radians: pixels `step` Mpc/h apart with a jitter of
    step / 10 (step a multiple of 1/4 and no jitter where seed < 0), weights in [1, 4)."""
    rng = np.random.default_rng(abs(seed))
    forests = []
    for n in lengths:
        d = 3000.0 + 4.0 * rng.integers(0, 8) + step * np.arange(n)
        if seed >= 0:
            d = d + rng.uniform(0.0, 0.1 * step, n)
        forests.append((rng.uniform(0, patch) if seed >= 0 else 0.01, rng.uniform(0, patch) if seed >= 0 else 0.02,
                        d, np.log(3600.0) + 1e-4 * np.arange(n), rng.normal(0.05, 0.3, n), rng.uniform(1, 4, n)))
    return line_catalog(forests)


@pytest.mark.parametrize("lengths,step,bins,seed", [
    ((1, 2, 7, 8, 9), 1.0, (25, 25, 100.0, 100.0), 1),           # below one block of rows
    ((31, 32, 33, 63, 65), 0.5, (20, 40, 40.0, 20.0), 2),        # edges of a group of diagonals
    ((255, 256, 257, 300), 0.6, (50, 50, 200.0, 200.0), 3),      # edges of a tile
    ((520, 90, 1), 0.25, (256, 4, 128.0, 16.0), 4),              # most r_par bins, three tiles
    ((40, 70, 110), 0.25, (1, 300, 60.0, 30.0), 5),              # one r_par bin, bands of many rows
    ((96, 130, 64), 0.25, (25, 10, 100.0, 50.0), -6),            # one line of sight: every separation on 1/16 bin
    ((64, 64, 64), 4.0, (25, 10, 100.0, 50.0), -7),              # ... and every one exactly on a bin edge
])
def test_fp64_sums_are_those_of_the_definition(api, handle, lengths, step, bins, seed):
    """Bins are the definition's and the sums those of 64 bits.  Tolerance: a run of pixel pairs is rounded at 2^-45
    of the largest product (its integers are scaled to 2^53..2^54), so n pixel pairs are off by at most
    n 2^-45 w_max^2 <= n 2^-41 for weights below 4, and W >= n: 5e-13 of W; the pixels' rounding (2^-54 of the
    largest) and the FP64 sums over tiles add less.  N likewise with (w delta)_max^2 <= (4 delta_max)^2."""
    cat = _catalog(lengths, step, seed)
    b = synth.Bins(*bins)
    ref = oracle.xi.xi_sums(cat, b)
    num, wsum, xi = api.lya_xi(handle, api.DeviceCatalog.from_host(cat), b, "fp64")
    api.lya_sync_status(handle)
    n, w = num.cpu().numpy(), wsum.cpu().numpy()
    assert ref["count"].sum() > 0
    assert np.all((w > 0) == (ref["count"] > 0))
    assert np.all(np.abs(w - ref["wsum"]) <= 1e-12 * ref["wsum"])
    wd = float(np.abs(cat.weight.astype(np.float64) * cat.delta).max())
    assert np.all(np.abs(n - ref["num"]) <= ref["count"] * 2.0 ** -44 * wd * wd + 1e-300)


@pytest.mark.parametrize("lengths,step,bins,seed,kind", [
    ((1, 2, 7, 8, 9), 1.0, (25, 25, 100.0, 100.0), 11, "z"),       # below one block of rows
    ((31, 33, 65, 239, 240, 241), 0.6, (20, 40, 80.0, 60.0), 12, "z"),   # edges of groups and of a tile
    ((500, 90), 0.25, (250, 4, 125.0, 16.0), 13, ""),              # many r_par bins, three tiles
    ((40, 70, 110), 0.25, (1, 300, 60.0, 30.0), 14, "z"),          # one r_par bin, bands of many rows
    ((96, 130, 64), 1.0, (25, 10, 100.0, 50.0), 15, "gap"),        # a gap: diagonals that leave the grid and return
    ((64, 80), 1.0, (25, 10, 100.0, 50.0), 16, "huge"),            # weights whose products exceed the fixed point
    ((64, 80), 1.0, (25, 10, 100.0, 50.0), 17, "nan"),             # a redshift that is not a number
])
def test_bin_means_forms(api, handle, lengths, step, bins, seed, kind):
    """Counts are whole numbers, equal up to the oracle's edge allowance.  The means are FP32 sums of 8 terms and
    integers beyond: 8 x 2^-24 relative to a sum of positive terms is the worst case (5e-7), next to the edge
    allowance of one bin width (one range for the distances and redshifts) times twice the ambiguous weight."""
    cat = _catalog(lengths, step, seed, patch=6e-3)
    if kind == "gap":
        cat.dist[int(cat.offsets[1]) // 2:int(cat.offsets[1])] += 60.0
    if kind == "huge":
        cat.weight *= np.float32(1e16)
    z = np.exp(cat.loglam) / 1215.67 - 1.0
    b = synth.Bins(*bins)
    ref = oracle.xi.bin_means(cat, b, eps_edge=6e-5, z=z)
    dc = api.DeviceCatalog.from_host(cat)
    zt = torch.from_numpy(z).cuda()
    if kind == "nan":
        zt[3] = float("nan")
    got = api.lya_xi_bin_means(handle, dc, b, z_pix=None if kind == "" else zt)
    api.lya_sync_status(handle)
    got = {k: v.cpu().numpy() for k, v in got.items()}
    W = ref["wsum"]
    on = W > 4.0 * ref["edge_w"]
    assert on.sum() > 0
    assert np.all(np.abs(got["count"] - ref["count"]) <= ref["edge_c"])
    assert np.all(np.abs(got["wsum"] - W) <= 1e-6 * W + ref["edge_w"])
    frac = 2.0 * ref["edge_w"][on] / (W[on] - ref["edge_w"][on])
    spread = float(cat.dist.max() - cat.dist.min())
    for key, width in (("rpar_mean", b.r_par_max / b.n_par), ("rperp_mean", b.r_perp_max / b.n_perp),
                       ("dist_mean", spread), ("z_mean", float(z.max() - z.min()))):
        if key not in got:
            continue
        err = np.abs(got[key][on] - ref[key][on])
        if kind == "nan" and key == "z_mean":
            bad = np.isnan(got[key][on])
            assert bad.any()     # ... reaches the bins that hold it
            err = err[~bad]
            assert np.all(err <= 1e-6 * np.abs(ref[key][on][~bad]) + (frac * width)[~bad])
            continue
        assert np.all(err <= 1e-6 * np.abs(ref[key][on]) + frac * width)


def _light_and_heavy(factor, seed=41):
    """Forests of 40 light pixels and 40 of `factor` times their weight: every pixel pair less than 40 Mpc/h apart
    along the line of sight is one of light pixels (of two forests of different kinds)."""
    rng = np.random.default_rng(seed)
    forests = []
    for k in range(2):
        d = np.concatenate([3000.0 + np.arange(40), 3000.0 + (250.0 if k else 100.0) + np.arange(40)])
        forests.append((rng.uniform(0, 2e-3), rng.uniform(0, 2e-3), d + rng.uniform(0.0, 0.2, 80),
                        np.log(3600.0) + 1e-4 * np.arange(80), rng.normal(0.05, 0.3, 80),
                        rng.uniform(1, 4, 80) * np.repeat([1.0, factor], 40)))
    return line_catalog(forests)


@pytest.mark.parametrize("factor", [30.0, 1e4, 1e8, 1e16])
def test_fp64_sums_of_light_pixels(api, handle, factor):
    """Bins that hold light pixels only, beside heavy ones of the same forests.  A run is rounded by at most 2^-36 of
    its smallest product, its products by 2^-38 each and their low halves' sum by 2^-37: W to 2^-35 of the bin's own
    value, N to 2^-35 of its number of pairs times the square of the largest light |w delta|."""
    cat = _light_and_heavy(factor)
    b = synth.Bins(60, 5, 300.0, 25.0)
    ref = oracle.xi.xi_sums(cat, b)
    num, wsum, xi = api.lya_xi(handle, api.DeviceCatalog.from_host(cat), b, "fp64")
    api.lya_sync_status(handle)
    n, w = num.cpu().numpy(), wsum.cpu().numpy()
    light = (ref["count"] > 0) & (np.arange(b.n_par * b.n_perp) // b.n_perp < 8)
    assert light.sum() >= 8 and np.all(ref["wsum"][light] <= 16.0 * ref["count"][light])
    assert np.all((w > 0) == (ref["count"] > 0))
    assert np.all(np.abs(w - ref["wsum"]) <= 2.0 ** -35 * ref["wsum"])
    pix = np.arange(80) < 40
    wd = np.abs(cat.weight.astype(np.float64) * cat.delta).reshape(2, 80)[:, pix].max()
    assert np.all(np.abs(n - ref["num"])[light] <= 2.0 ** -35 * wd * wd * ref["count"][light])


@pytest.mark.parametrize("factor", [30.0, 1e3, 1e5, 1e12])
@pytest.mark.parametrize("with_z", [True, False])
def test_bin_means_of_light_pixels(api, handle, factor, with_z):
    """Bins that hold light pixels only, beside heavy ones of the same forests: W and the means to 1e-6 of the bin's
    own values (FP32 products and sums of 8 terms; the integers round a block by at most 2^-21 of its smallest pair,
    5e-7), next to the edge allowance of test_bin_means_forms."""
    cat = _light_and_heavy(factor)
    z = np.exp(cat.loglam) / 1215.67 - 1.0
    b = synth.Bins(60, 5, 300.0, 25.0)
    ref = oracle.xi.bin_means(cat, b, eps_edge=6e-5, z=z)
    got = api.lya_xi_bin_means(handle, api.DeviceCatalog.from_host(cat), b, z_pix=torch.from_numpy(z).cuda() if with_z else None)
    api.lya_sync_status(handle)
    got = {k: v.cpu().numpy() for k, v in got.items()}
    W = ref["wsum"]
    on = W > 4.0 * ref["edge_w"]
    light = on & (np.arange(b.n_par * b.n_perp) // b.n_perp < 8)
    assert light.sum() >= 8 and np.all(W[light] <= 16.0 * ref["count"][light])
    assert np.all(np.abs(got["count"] - ref["count"]) <= ref["edge_c"])
    assert np.all(np.abs(got["wsum"] - W) <= 1e-6 * W + ref["edge_w"])
    frac = 2.0 * ref["edge_w"][on] / (W[on] - ref["edge_w"][on])
    for key, width in (("rpar_mean", 5.0), ("rperp_mean", 5.0), ("dist_mean", float(cat.dist.max() - cat.dist.min())),
                       ("z_mean", float(z.max() - z.min()))):
        if key in got:
            err = np.abs(got[key][on] - ref[key][on])
            assert np.all(err <= 1e-6 * np.abs(ref[key][on]) + frac * width), key


@pytest.mark.parametrize("factor", [1.0, 30.0, 1e4, 1e8, 1e16])
def test_xi1d_of_light_pixels(api, handle, factor):
    """One pixel of `factor` times the others' weight, 60 Mpc/h beyond them: bins below 50 Mpc/h hold light pixels
    only.  Tolerances as in test_fp64_sums_of_light_pixels."""
    rng = np.random.default_rng(42)
    forests = []
    for k in range(40):
        m = 48 + k % 2
        d = 3000.0 + np.append(np.arange(m - 1), m + 60) + rng.uniform(0.0, 0.2, m)
        w = rng.uniform(1, 4, m)
        w[-1] *= factor if k % 3 else 1.0
        forests.append((0.0, 0.0, d, np.log(3600.0) + 1e-4 * np.arange(m), rng.normal(0.05, 0.3, m), w))
    cat = line_catalog(forests)
    ref = oracle.xi1d.xi1d_sums(cat, 40, 200.0)
    num, wsum, xi = api.lya_xi1d(handle, api.DeviceCatalog.from_host(cat), 40, 200.0)
    api.lya_sync_status(handle)
    n, w = num.cpu().numpy(), wsum.cpu().numpy()
    assert np.all((w > 0) == (ref["wsum"] > 0))
    assert np.all(np.abs(w - ref["wsum"]) <= 2.0 ** -35 * ref["wsum"])
    light = ref["wsum"][:9]     # weights are at least 1: no more pixel pairs than this
    wd = max(np.abs(f[5][:-1] * f[4][:-1]).max() for f in forests)
    assert np.all(np.abs(n - ref["num"])[:9] <= 2.0 ** -35 * wd * wd * light)


@pytest.mark.parametrize("lengths,step,n_bins,r_max,seed", [
    ((1, 2, 8, 9, 33, 34), 1.0, 20, 40.0, 21),           # below and above a block of rows and a group of lags
    ((255, 257, 264, 300), 0.5, 50, 200.0, 22),          # edges of a batch of 256 rows
    ((1200, 5), 0.25, 4096, 300.0, 23),                  # most bins, sums straight to the FP64 outputs
    ((90, 70), 1.0, 513, 60.0, 24),                      # one more than the bins summed per warp
    ((90, 70, 40), 0.5, 1, 30.0, 25),                    # one bin
    ((96, 130, 64), 0.25, 25, 100.0, -26),               # separations on 1/16 bin
    ((64, 64, 200), 4.0, 25, 100.0, -27),                # every separation exactly on a bin edge
])
def test_xi1d_forms(api, handle, lengths, step, n_bins, r_max, seed):
    """Bins are the definition's, sums exact up to the tolerance of test_fp64_sums_are_those_of_the_definition."""
    cat = _catalog(lengths, step, seed)
    ref = oracle.xi1d.xi1d_sums(cat, n_bins, r_max)
    num, wsum, xi = api.lya_xi1d(handle, api.DeviceCatalog.from_host(cat), n_bins, r_max)
    api.lya_sync_status(handle)
    n, w = num.cpu().numpy(), wsum.cpu().numpy()
    assert (ref["wsum"] > 0).any()
    assert np.all((w > 0) == (ref["wsum"] > 0))
    assert np.all(np.abs(w - ref["wsum"]) <= 1e-12 * ref["wsum"])
    wd = float(np.abs(cat.weight.astype(np.float64) * cat.delta).max())
    # pixel pairs of a bin <= W, the weights being at least 1
    assert np.all(np.abs(n - ref["num"]) <= ref["wsum"] * 2.0 ** -44 * wd * wd + 1e-300)


def test_dmat_is_reproducible(api, handle):
    """Every forest pair's contribution is formed in a fixed order and summed in FP64, so two calls differ by the
    order of the FP64 sums only: at most n 2^-53 of the sum of magnitudes, n < 2^16 pairs per entry (1e-11).  (A
    triangle entry left behind where a pair's terms cancel to zero would be added to another pair's entry.)"""
    cat = synth.subset(synth.make(1, n_forests=20000), np.arange(12000))
    dc = api.DeviceCatalog.from_host(cat)
    b = synth.Bins(50, 50, 200.0, 200.0)
    first, w1 = api.lya_dmat(handle, dc, b, 0.05, 7)
    scale = first.abs().amax(dim=1, keepdim=True)
    for _ in range(3):
        again, w2 = api.lya_dmat(handle, dc, b, 0.05, 7)
        assert bool(((again - first).abs() <= 1e-11 * scale).all())
        assert bool(((w2 - w1).abs() <= 1e-11 * w1).all())


def test_dmat_of_a_mock_does_not_depend_on_the_batch(api, handle):
    """D of four catalogues in one call against each one's own call, where the blocks meet the pairs in another
    order: the allowance of test_dmat_is_reproducible."""
    cats = []
    for k in range(4):
        spec = synth.spec_for(4, seed=k, n_forests=3000)
        spec.area_deg2 = 60.0
        cats.append(api.DeviceCatalog.from_host(synth.generate(spec)))
    b = synth.Bins(50, 50, 200.0, 200.0)
    D, w = api.lya_dmat_batched(handle, cats, b, 0.1, 1234)
    for k, c in enumerate(cats):
        own, w1 = api.lya_dmat(handle, c, b, 0.1, 1234)
        assert bool(((w[k] - w1).abs() <= 1e-11 * w1).all())
        assert bool(((D[k] - own).abs() <= 1e-11 * own.abs().amax(dim=1, keepdim=True)).all())


def test_dmat_on_a_grid_of_unequal_sides(api, handle):
    """n_par != n_perp: the accumulators' bin numbering (t n_par + p) against the outputs' (p n_perp + t).  The
    allowance is the one of the square grids (1e-5 of the row maximum and the quotient rule of the edge terms)."""
    cat = synth.subset(synth.make(0), np.arange(60))
    b = synth.Bins(13, 22, 60.0, 90.0)
    pr = oracle.pairs.forest_pairs(cat, b)
    fwd = oracle.xi.xi_sums(cat, b, pr, eps_edge=6e-5)
    ref = oracle.dmat.dmat(cat, b, pr, processes=0, eps_edge=6e-5)
    D, w = api.lya_dmat(handle, api.DeviceCatalog.from_host(cat), b, 1.0, 3)
    api.lya_sync_status(handle)
    W, E, R = fwd["wsum"], fwd["edge_w"], ref["dmat"]
    den = (W - E)[:, None]
    edge = np.divide(ref["edge_d"] + np.abs(R) * E[:, None], den, out=np.zeros_like(R), where=den > 0)
    assert np.all(np.abs(D.cpu().numpy() - R) <= 1e-5 * np.abs(R).max(axis=1)[:, None] + edge + 1e-12)
    assert np.all(np.abs(w.cpu().numpy() - W) <= 1e-6 * W + E + 1e-9)


@pytest.mark.parametrize("lengths,bins,step,patch", [
    # edges of windows and batches
    ((15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65), (13, 22, 60.0, 90.0), (0.3, 3.7), 0.016),
    # far apart pixels: 32 vectors reach more bins than the staging holds, and the batch is halved
    ((40, 36, 44, 38, 33), (20, 40, 100.0, 4.0), (2.0, 20.0), 0.0028),
    # every pixel of a forest in the window
    ((40, 33, 130, 20, 64), (7, 3, 300.0, 6.0), (0.3, 3.7), 0.004),
])
def test_dmat_windows_and_batches(api, handle, lengths, bins, step, patch):
    """Pixels at random spacings, so that neighbouring vectors visit different bins.  Allowance as above."""
    rng = np.random.default_rng(sum(lengths))
    fs = [(*rng.uniform(0, patch, 2), 500.0 + rng.uniform(0, 20) + np.cumsum(rng.uniform(*step, n)),
           8.2 + np.cumsum(rng.uniform(1e-4, 6e-4, n)), rng.standard_normal(n), rng.uniform(0.5, 2.0, n))
          for n in lengths]
    cat = line_catalog(fs)
    b = synth.Bins(*bins)
    pr = oracle.pairs.forest_pairs(cat, b)
    fwd = oracle.xi.xi_sums(cat, b, pr, eps_edge=6e-5)
    ref = oracle.dmat.dmat(cat, b, pr, processes=0, eps_edge=6e-5)
    D, w = api.lya_dmat(handle, api.DeviceCatalog.from_host(cat), b, 1.0, 3)
    api.lya_sync_status(handle)
    W, E, R = fwd["wsum"], fwd["edge_w"], ref["dmat"]
    den = (W - E)[:, None]
    edge = np.divide(ref["edge_d"] + np.abs(R) * E[:, None], den, out=np.zeros_like(R), where=den > 0)
    assert np.all(np.abs(D.cpu().numpy() - R) <= 1e-5 * np.abs(R).max(axis=1)[:, None] + edge + 1e-12)
    assert np.all(np.abs(w.cpu().numpy() - W) <= 1e-6 * W + E + 1e-9)


@pytest.mark.parametrize("lengths,n_qso,bins,seed", [
    ((1, 2, 31, 32, 33), 40, (10, 8, 60.0, 40.0), 31),          # edges of a warp's window step
    ((300, 700, 90), 90, (100, 50, 200.0, 200.0), 32),          # teams of several warps
    ((2600, 1500), 33, (64, 40, 200.0, 200.0), 33),             # one team per block
    ((60, 50), 20, (1, 1, 100.0, 100.0), 34),                   # one bin: the longest runs
])
def test_xcf_forms(api, handle, lengths, n_qso, bins, seed):
    """Pixels are rounded at 2^-44 of the forest's largest value and the sums are double-float, so off the bin edges
    only the FP32 rounding of the packed w delta (2^-24 of each term) remains: 1e-6 of W and of the sum of |terms|,
    next to the oracle's edge allowance."""
    cat = _catalog(lengths, 0.3, seed, patch=8e-3)
    rng = np.random.default_rng(seed)
    q = synth.Quasars(ra=rng.uniform(0, 8e-3, n_qso), dec=rng.uniform(0, 8e-3, n_qso),
                      dist=rng.uniform(2900.0, 3400.0, n_qso), weight=rng.uniform(0.5, 2.0, n_qso).astype(np.float32),
                      z=np.full(n_qso, 2.5))
    b = synth.Bins(*bins)
    own = np.arange(cat.n_forests, dtype=np.int64)
    ref = oracle.xcf.xcf_sums(cat, q, b, forest_qso=own, eps_edge=6e-5)
    num, wsum, _ = api.lya_xcf(handle, api.DeviceCatalog.from_host(cat), api.DeviceQuasars.from_host(q), b, own)
    api.lya_sync_status(handle)
    n, w = num.cpu().numpy(), wsum.cpu().numpy()
    assert ref["wsum"].sum() > 0
    assert np.all(np.abs(w - ref["wsum"]) <= 1e-6 * ref["wsum"] + ref["edge_w"])
    top = float(np.abs(cat.delta).max())
    assert np.all(np.abs(n - ref["num"]) <= 1e-6 * top * ref["wsum"] + ref["edge_n"] + 1e-300)


@pytest.mark.parametrize("factor,forest,quasar", [
    (30.0, 1.0, 1.0), (1e4, 1.0, 1.0), (1e8, 1.0, 1.0),
    (4.0, 1e-12, 1e34), (4.0, 1e-30, 1e3), (4.0, 1e22, 1e-10),   # weights far from 1 whose products are not
])
def test_xcf_of_light_pixels(api, handle, factor, forest, quasar):
    """Bins of light pixels beside heavy ones of the same forests.  The products of the FP32 weights are formed with
    their errors and the sums are double-float: W to 2^-40 of the bin's own value off the bin edges; N is a sum of
    FP32 w delta (2^-24 of each term)."""
    cat = _light_and_heavy(factor)
    rng = np.random.default_rng(7)
    cat.weight *= np.float32(forest)
    nq = 40
    q = synth.Quasars(ra=rng.uniform(0, 2e-3, nq), dec=rng.uniform(0, 2e-3, nq), dist=rng.uniform(3000.0, 3040.0, nq),
                      weight=(rng.uniform(0.5, 2.0, nq) * quasar).astype(np.float32), z=np.full(nq, 2.5))
    b = synth.Bins(100, 5, 300.0, 25.0)
    ref = oracle.xcf.xcf_sums(cat, q, b, eps_edge=6e-5)
    num, wsum, _ = api.lya_xcf(handle, api.DeviceCatalog.from_host(cat), api.DeviceQuasars.from_host(q), b)
    api.lya_sync_status(handle)
    n, w = num.cpu().numpy(), wsum.cpu().numpy()
    sure = (ref["count"] > 0) & (ref["edge_w"] == 0)
    assert sure.sum() > 30
    assert np.all(np.abs(w - ref["wsum"])[sure] <= 2.0 ** -40 * ref["wsum"][sure])
    assert np.all(np.abs(n - ref["num"])[sure] <= 1e-6 * float(np.abs(cat.delta).max()) * ref["wsum"][sure])


@pytest.mark.parametrize("lengths,n_qso,step,bins,p,seed", [
    ((1, 2, 31, 32, 33, 64), 12, 0.3, (10, 8, 60.0, 40.0), 1.0, 51),     # two batches of 32 pairs and a remainder
    ((32,), 32, 0.3, (10, 8, 60.0, 40.0), 1.0, 52),                      # exactly one batch
    ((70, 40), 33, 0.3, (1, 1, 100.0, 100.0), 1.0, 53),                  # one bin: runs over more than 32 pixels
    ((90, 200), 60, 0.3, (41, 7, 200.0, 100.0), 0.4, 54),                # batches filled from several draws
    ((1440, 30), 20, 0.3, (64, 40, 200.0, 200.0), 1.0, 55),              # run lists of eight warps fill shared memory
    ((5780,), 3, 0.15, (64, 40, 200.0, 200.0), 1.0, 56),                 # ... of two warps
])
def test_xdmat_forms(api, handle, lengths, n_qso, step, bins, p, seed):
    """Allowance as in test_gpu_xcf: 1e-5 of the row's largest entry and the edge terms' quotient rule."""
    cat = _catalog(lengths, step, seed, patch=8e-3)
    rng = np.random.default_rng(seed)
    q = synth.Quasars(ra=rng.uniform(0, 8e-3, n_qso), dec=rng.uniform(0, 8e-3, n_qso),
                      dist=rng.uniform(2900.0, 3400.0, n_qso), weight=rng.uniform(0.5, 2.0, n_qso).astype(np.float32),
                      z=np.full(n_qso, 2.5))
    b = synth.Bins(*bins)
    D, Wd = api.lya_xdmat(handle, api.DeviceCatalog.from_host(cat), api.DeviceQuasars.from_host(q), b, p, seed)
    api.lya_sync_status(handle)
    pl = oracle.xcf.forest_quasar_pairs(cat, q, b, np.full(cat.n_forests, -1))
    m = oracle.xcf.keep_xpairs(pl[0], pl[1], seed, p)
    ref = oracle.xcf.xdmat(cat, q, b, (pl[0][m], pl[1][m]), eps_edge=6e-5)
    W = ref["wsum"]
    assert np.count_nonzero(W) > 0
    rel = np.divide(ref["edge_w"], W, out=np.zeros_like(W), where=W > 0)
    col = np.divide(ref["edge_d"], W[:, None], out=np.zeros_like(ref["edge_d"]), where=W[:, None] > 0)
    tol = (1e-5 + 3 * rel)[:, None] * np.abs(ref["dmat"]).max(axis=1)[:, None] + col
    assert np.all(np.abs(D.cpu().numpy() - ref["dmat"]) <= tol + 1e-12)
    assert np.all(np.abs(Wd.cpu().numpy() - W) <= 1e-6 * W + ref["edge_w"] + 1e-9)


def test_dmat_rows_are_divided_by_their_weight(api, handle):
    """With eta = I and whole-number weights every sum is exact, in any order, and D~_AA = W_A: the quotient of equal
    numbers is 1 (times a rounded reciprocal it is not, for one W in seven)."""
    rng = np.random.default_rng(61)
    fs = [(*rng.uniform(0, 8e-3, 2), 3000.0 + 3.0 * rng.uniform(0, 1, 1) + 1.5 * np.arange(60), 8.2 + 1e-4 * np.arange(60),
           rng.standard_normal(60), rng.integers(1, 8, 60)) for _ in range(12)]
    cat = line_catalog(fs)
    q = synth.Quasars(ra=rng.uniform(0, 8e-3, 30), dec=rng.uniform(0, 8e-3, 30), dist=rng.uniform(2950.0, 3150.0, 30),
                      weight=rng.integers(1, 8, 30).astype(np.float32), z=np.full(30, 2.5))
    b = synth.Bins(40, 12, 100.0, 60.0)
    dc = api.DeviceCatalog.from_host(cat)
    for D, w in (api.lya_dmat(handle, dc, b, 1.0, 3, eta="identity"),
                 api.lya_xdmat(handle, dc, api.DeviceQuasars.from_host(q), b, 1.0, 3, eta="identity")):
        D, w = D.cpu().numpy(), w.cpu().numpy()
        on = w > 0
        assert on.sum() > 100
        np.testing.assert_array_equal(D[np.ix_(on, on)], np.eye(on.sum()))


@pytest.mark.parametrize("lengths", [(1, 1, 1, 1, 30, 41), (1, 2, 3, 2, 1, 3)])
def test_forests_of_few_pixels(api, handle, lengths):
    """One pixel has no gap to its neighbour to bound a run by: W of xi and of D to 1e-6, D (whose entries are at most
    1) to 1e-5, next to the edge allowances of test_dmat_on_a_grid_of_unequal_sides."""
    cat = _catalog(lengths, 1.0, 71, patch=6e-3)
    b = synth.Bins(13, 10, 65.0, 50.0)
    pr = oracle.pairs.forest_pairs(cat, b)
    fwd = oracle.xi.xi_sums(cat, b, pr, eps_edge=6e-5)
    ref = oracle.dmat.dmat(cat, b, pr, processes=0, eps_edge=6e-5)
    dc = api.DeviceCatalog.from_host(cat)
    num, wsum, _ = api.lya_xi(handle, dc, b, "mixed")
    D, w = api.lya_dmat(handle, dc, b, 1.0, 3)
    api.lya_sync_status(handle)
    W, E, R = fwd["wsum"], fwd["edge_w"], ref["dmat"]
    assert np.count_nonzero(W) > 5
    top = float(np.abs(cat.delta).max())
    assert np.all(np.abs(wsum.cpu().numpy() - W) <= 1e-6 * W + E)
    assert np.all(np.abs(num.cpu().numpy() - fwd["num"]) <= 1e-6 * top * top * W + fwd["edge_n"])
    assert np.all(np.abs(w.cpu().numpy() - W) <= 1e-6 * W + E)
    den = (W - E)[:, None]
    edge = np.divide(ref["edge_d"] + np.abs(R) * E[:, None], den, out=np.zeros_like(R), where=den > 0)
    assert np.all(np.abs(D.cpu().numpy() - R) <= 1e-5 + edge)


@pytest.mark.parametrize("lengths,step,bins,patch,seed", [
    ((255, 256, 257, 258, 33), 0.3, (25, 25, 100.0, 100.0), 4e-3, 81),   # edges of a staged segment, all in the grid
    ((512, 513, 31, 1, 32), 0.3, (40, 30, 60.0, 100.0), 4e-3, 82),       # ranges that end beside a segment's edge
    ((300, 290, 64), 0.5, (30, 10, 45.0, 30.0), 8e-3, 83),               # clamps along both coordinates
    ((96, 130, 257), 0.6, (25, 10, 50.0, 50.0), 0.0, 84),                # one line of sight: r_perp = 0
])
def test_gradient_forms(api, handle, lengths, step, bins, patch, seed):
    """The gradient's staged segments of 256 pixels and their clamp-free ranges; allowance of
    test_gpu_parity.test_backward_matches_oracle."""
    cat = _catalog(lengths, step, seed, patch=patch)
    b = synth.Bins(*bins)
    pr = oracle.pairs.forest_pairs(cat, b)
    c = np.random.default_rng(seed).normal(size=b.nbins)
    fwd = oracle.xi.xi_sums(cat, b, pr)
    gd_ref, gw_ref, info = oracle.adjoint.xi_grad(cat, b, c, pr, absolute=True, eps_edge=6e-5, fwd=fwd)
    gd, gw = api.lya_xi_backward(handle, api.DeviceCatalog.from_host(cat), b, torch.from_numpy(c).cuda(),
                                 torch.from_numpy(fwd["xi"]).cuda(), torch.from_numpy(fwd["wsum"]).cuda())
    api.lya_sync_status(handle)
    assert np.count_nonzero(gd_ref) > cat.n_pix // 2
    assert np.all(np.abs(gd.cpu().numpy() - gd_ref) <= 1e-5 * info["grad_delta_abs"] + info["grad_delta_edge"] + 1e-12)
    assert np.all(np.abs(gw.cpu().numpy() - gw_ref) <= 1e-5 * info["grad_weight_abs"] + info["grad_weight_edge"] + 1e-12)


@pytest.mark.parametrize("lengths,step,bins,seed", [
    ((1, 2, 7, 8, 9, 16, 33), 1.0, (25, 25, 100.0, 100.0), 91),   # below and above a block of rows
    ((255, 256, 257, 300), 0.6, (50, 50, 200.0, 200.0), 92),      # edges of a tile
    ((520, 90, 1), 0.25, (256, 4, 128.0, 16.0), 93),              # three tiles
    ((40, 70, 110), 0.25, (1, 300, 60.0, 30.0), 94),              # bands of many rows
])
def test_weights_of_many_decades(api, handle, lengths, step, bins, seed):
    """Weights over twelve decades within every forest: the sums that leave the integers.  FP64 path and 1D to the
    order of their FP64 sums (n 2^-53 < 1e-12), bin means to their FP32 sums of 8 pairs (5e-7), cross-correlation to
    2^-40 off the bin edges; N against W times the largest |delta|."""
    cat = _catalog(lengths, step, seed)
    rng = np.random.default_rng(seed)
    cat.weight = (10.0 ** rng.uniform(-6.0, 6.0, cat.n_pix)).astype(np.float32)
    top = float(np.abs(cat.delta).max())
    b = synth.Bins(*bins)
    dc = api.DeviceCatalog.from_host(cat)
    cpu = lambda *t: [x.cpu().numpy() for x in t]   # noqa: E731

    ref = oracle.xi.xi_sums(cat, b)
    n, w, _ = cpu(*api.lya_xi(handle, dc, b, "fp64"))
    assert np.all(np.abs(w - ref["wsum"]) <= 1e-12 * ref["wsum"])
    assert np.all(np.abs(n - ref["num"]) <= 1e-12 * top * top * ref["wsum"])

    ref = oracle.xi1d.xi1d_sums(cat, 37, 60.0)
    n, w, _ = cpu(*api.lya_xi1d(handle, dc, 37, 60.0))
    assert np.all(np.abs(w - ref["wsum"]) <= 1e-12 * ref["wsum"])
    assert np.all(np.abs(n - ref["num"]) <= 1e-12 * top * top * ref["wsum"])

    z = np.exp(cat.loglam) / 1215.67 - 1.0
    ref = oracle.xi.bin_means(cat, b, eps_edge=6e-5, z=z)
    got = api.lya_xi_bin_means(handle, dc, b, z_pix=torch.from_numpy(z).cuda())
    W = ref["wsum"]
    on = W > 4.0 * ref["edge_w"]
    assert on.sum() > 0
    assert np.all(np.abs(got["count"].cpu().numpy() - ref["count"]) <= ref["edge_c"])
    assert np.all(np.abs(got["wsum"].cpu().numpy() - W) <= 1e-6 * W + ref["edge_w"])
    frac = 2.0 * ref["edge_w"][on] / (W[on] - ref["edge_w"][on])
    for key, width in (("rpar_mean", b.r_par_max / b.n_par), ("rperp_mean", b.r_perp_max / b.n_perp),
                       ("dist_mean", float(cat.dist.max() - cat.dist.min())), ("z_mean", float(z.max() - z.min()))):
        err = np.abs(got[key].cpu().numpy()[on] - ref[key][on])
        assert np.all(err <= 1e-6 * np.abs(ref[key][on]) + frac * width), key

    q = synth.Quasars(ra=rng.uniform(0, 2e-3, 30), dec=rng.uniform(0, 2e-3, 30), dist=rng.uniform(2950.0, 3200.0, 30),
                      weight=(10.0 ** rng.uniform(-6.0, 6.0, 30)).astype(np.float32), z=np.full(30, 2.5))
    ref = oracle.xcf.xcf_sums(cat, q, b, eps_edge=6e-5)
    n, w, _ = cpu(*api.lya_xcf(handle, dc, api.DeviceQuasars.from_host(q), b))
    sure = (ref["count"] > 0) & (ref["edge_w"] == 0)
    assert sure.sum() > 0
    assert np.all(np.abs(w - ref["wsum"])[sure] <= 2.0 ** -40 * ref["wsum"][sure])
    assert np.all(np.abs(n - ref["num"])[sure] <= 1e-6 * top * ref["wsum"][sure])
    api.lya_sync_status(handle)


@pytest.mark.parametrize("n_sub,nb", [(2, 65), (33, 64), (1100, 130)])
def test_covariance_of_whole_numbers(api, handle, n_sub, nb):
    """Whole-number sums in two sub-samples (the first and the last) with N adding up to 0: every sum is exact, so an
    entry is the correctly rounded quotient 2 n_A n_B / (W_A W_B)."""
    rng = np.random.default_rng(n_sub)
    n = rng.integers(-50, 51, nb).astype(np.float64)
    num, w = np.zeros((n_sub, nb)), np.zeros((n_sub, nb))
    num[0], num[-1] = n, -n
    w[0], w[-1] = rng.integers(1, 60, nb), rng.integers(0, 60, nb)
    cov, xi = api.lya_xi_covariance(handle, torch.from_numpy(num).cuda(), torch.from_numpy(w).cuda())
    W = w.sum(axis=0)
    np.testing.assert_array_equal(xi.cpu().numpy(), 0.0)
    np.testing.assert_array_equal(cov.cpu().numpy(), 2.0 * np.outer(n, n) / np.outer(W, W))


@pytest.mark.parametrize("n_r,n_alpha,n_theta,nf,factor", [
    (4, 5, 3, 14, 1.0),      # classes summed in shared memory
    (16, 1, 1, 14, 1.0),     # the most |r| bins
    (1, 3, 2, 24, 1.0),      # one class, more records than a word holds
    (4, 5, 3, 14, 1e9),      # products beyond the fixed-point scale
    (4, 5, 3, 14, 0.0),      # all weights zero
])
def test_xi3_grouped_vertices(api, handle, n_r, n_alpha, n_theta, nf, factor):
    """Grids with fewer bins than a group of vertices has records.  Tolerances as in test_gpu_xi3."""
    spec = synth.Spec(n_forests=nf, seed=8, region="box", box_deg=0.3, grid="log10", delta_sigma=0.2)
    cat = synth.generate(spec)
    cat.weight[:] *= np.float32(factor)
    g = oracle.xi3.Grid3(n_r=n_r, n_theta=n_theta, n_alpha=n_alpha, r_max=15.0)
    num, wsum, xi = api.lya_xi3(handle, api.DeviceCatalog.from_host(cat), g)
    api.lya_sync_status(handle)
    ref = oracle.xi3.xi3_sums(cat, g, eps_r=1e-9, eps_c=2e-6)
    W, N, unit = wsum.cpu().numpy(), num.cpu().numpy(), max(float(factor), 1.0) ** 3
    assert np.all(np.abs(W - ref["wsum"]) <= 1e-6 * ref["wsum"] + ref["edge_w"] + 1e-9 * unit)
    assert np.all(np.abs(N - ref["num"]) <= 1e-5 * np.sqrt(ref["num_sq"]) + ref["edge_n"] + 1e-12 * unit)
    Wr = W.reshape(n_r, n_r, n_alpha, n_theta, n_theta)
    np.testing.assert_array_equal(Wr, Wr.transpose(1, 0, 2, 4, 3))


def test_xi3_without_room_for_scratch(api):
    """A grid whose interleaved sums do not fit beside the caller's outputs on the device: the same result, summed in
    the outputs.  A record's FP32 product is rounded twice in an order that follows the order in which its two
    neighbours were found, so two calls differ by up to 2^-22 of each record."""
    cat = synth.generate(synth.Spec(n_forests=14, seed=8, region="box", box_deg=0.3, grid="log10", delta_sigma=0.2))
    g = oracle.xi3.Grid3(n_r=16, n_theta=64, n_alpha=64, r_max=15.0)   # 2^26 bins: 1.07 GB of sums, and a quarter
    dc = api.DeviceCatalog.from_host(cat)
    with api.Handle() as h:
        n0, w0, x0 = api.lya_xi3(h, dc, g)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    block = torch.empty(free - 3 * 8 * n0.numel() - (700 << 20), dtype=torch.uint8, device="cuda")
    try:
        with api.Handle() as h:
            out = api.lya_xi3(h, dc, g)
            api.lya_sync_status(h)
    finally:
        del block
        torch.cuda.empty_cache()
    assert float(w0.sum()) > 0
    assert bool(((out[1] - w0).abs() <= 2.0 ** -22 * w0).all())
    top = float(np.abs(cat.delta).max()) ** 3
    assert bool(((out[0] - n0).abs() <= 2.0 ** -22 * top * w0).all())
    assert bool(((out[2] - x0).abs() <= 2.0 ** -21 * top).all())


def test_a_refused_allocation_does_not_reach_the_next_call(api):
    """A call whose scratch does not fit is refused with LYA_ERR_NO_MEMORY (-4), and the next call runs."""
    from paper_2507_00129_gb300._lib import LyaError
    cat = synth.subset(synth.make(0), np.arange(40))
    dc = api.DeviceCatalog.from_host(cat)
    small, large = synth.bins_for(0), synth.Bins(150, 100, 100.0, 100.0)   # 1.8 GB of D, 2.25 GB of scratch
    with api.Handle() as h:
        n0, w0, _ = api.lya_xi(h, dc, small)
        D = torch.empty((15000, 15000), dtype=torch.float64, device="cuda")
        W = torch.empty(15000, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        block = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
        try:
            with pytest.raises(LyaError) as e:
                api.lya_dmat(h, dc, large, 1.0, 3, D=D, W=W)
            assert e.value.code == -4
        finally:
            del block, D, W
            torch.cuda.empty_cache()
        n1, w1, _ = api.lya_xi(h, dc, small)
        api.lya_sync_status(h)
        assert bool(((w1 - w0).abs() <= 1e-11 * w0).all())


@pytest.mark.parametrize("factor", [30.0, 1e3, 1e6])
def test_xi3_light_triplets_beside_a_heavy_forest(api, handle, factor):
    """One forest, 13.2 Mpc/h from the others, weighs `factor` times as much, so that its records fill bins of their
    own (the outermost |r| bin, theta near 90 degrees) and every other bin holds light ones only.  W to 1e-6 of each
    bin's own value (FP32 products, 2^-23, and at most 2^-21 of a record in its rounding), N as in test_gpu_xi3."""
    rng = np.random.default_rng(3)
    forests = []
    for k in range(8):
        ra, dec = (0.0132, 0.0) if k == 0 else (0.0, 4e-4 * k)
        forests.append((ra, dec, 1000.0 + rng.uniform(0, 1) + np.arange(60) * 1.0, 8.2 + 1e-4 * np.arange(60),
                        rng.normal(0.05, 0.3, 60), rng.uniform(1, 4, 60) * (factor if k == 0 else 1.0)))
    cat = line_catalog(forests)
    g = oracle.xi3.Grid3(n_r=4, n_theta=3, n_alpha=5, r_max=15.0)
    num, wsum, xi = api.lya_xi3(handle, api.DeviceCatalog.from_host(cat), g)
    api.lya_sync_status(handle)
    ref = oracle.xi3.xi3_sums(cat, g, eps_r=1e-9, eps_c=2e-6)
    W, N = wsum.cpu().numpy(), num.cpu().numpy()
    assert ref["count"].sum() > 1e5
    assert np.all(W[ref["wsum"] > ref["edge_w"]] > 0)
    assert np.all(np.abs(W - ref["wsum"]) <= 1e-6 * ref["wsum"] + ref["edge_w"])
    assert np.all(np.abs(N - ref["num"]) <= 1e-5 * np.sqrt(ref["num_sq"]) + ref["edge_n"])
