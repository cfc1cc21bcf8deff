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
