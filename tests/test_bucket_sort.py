"""The per-tile sort at the edges of its paths: one tile lists every surfel, so
the bucket has exactly n keys.  Sizes around a CTA's 2,048 keys and a group's
1,024; depths spread evenly, clustered far below a bin of the depth map (the
bitonic and merge paths), or equal (ties by index).  The expected order is
NumPy's of (depth key, item), exact."""
import math

import numpy as np
import pytest

from paper_2607_04127_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build
    build.build()


def _depths(kind, n, rng):
    if kind == "even":
        return rng.uniform(1.0, 90.0, n)
    if kind == "wall":                      # a flat wall at 10 m, 2 cm noise, and a few outliers
        d = 10.0 + 0.02 * rng.normal(size=n)
        d[: max(1, n // 50)] = rng.uniform(1.0, 90.0, max(1, n // 50))
        return d
    if kind == "equal":
        return np.full(n, 7.0)
    if kind == "tight":                     # three quarters within a few ulps
        d = rng.uniform(1.0, 90.0, n)
        d[: 3 * n // 4] = 10.0 + 1e-6 * rng.integers(0, 4, 3 * n // 4)
        return d
    d = rng.uniform(1.0, 2.0, n)            # two clusters, most keys in the far one
    d[n // 10:] = rng.uniform(80.0, 80.5, n - n // 10)
    return d


@pytest.mark.parametrize("kind", ["even", "wall", "equal", "tight", "two"])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 2047, 2048, 2049, 3072, 4097, 9000, 70_001])
def test_single_tile(n, kind):
    from tests._gpu import run
    rng = np.random.default_rng(n)
    d = rng.permutation(_depths(kind, n, rng))
    az = np.full(n, 1.0) if kind == "equal" else rng.uniform(0.3, 2.8, n)   # (inside the left tile)
    el = rng.uniform(-0.5, 0.5, n) * (kind != "equal")
    pts = d[:, None] * np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], 1)
    surf = scenes.Surfels(pts.astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                          np.full((n, 2), math.log(0.002), np.float32), np.zeros(n, np.float32))
    frame = scenes.Frame(8, 64, 8, 32, -1.4, 1.4)
    tp, ip, rg, dk = run([surf], [frame], read_bins=True)["bins"]
    assert rg[0, 0] == 0 and rg[0, 1] == n and np.all(tp == 0)
    assert np.array_equal(ip, np.lexsort((np.arange(n), dk)).astype(ip.dtype))
