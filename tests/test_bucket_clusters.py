"""Buckets whose depths cluster far below a bin of the sort's depth map: groups
of more than 2,048 keys, partitioned a second time (one, several, and of equal
depths), and clusters within clusters, which stay too large (the merge through
global memory); tiles of up to 2,048 keys (the merge in shared memory).  The
order is NumPy's of (depth key, item), exact."""
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
    if kind == "wall":                      # 1 mm of noise, a near and a far outlier
        d = 10.0 + 0.001 * rng.normal(size=n)
    elif kind == "walls":
        d = np.float64([3.0, 10.0, 30.0])[rng.integers(0, 3, n)] * (1.0 + 1e-6 * rng.integers(0, 3, n))
    elif kind == "equal":
        return np.full(n, 7.0)
    else:                                   # half within an ulp, half spread over a bin of 49 octaves and more
        d = 10.0 + 0.1 * rng.uniform(-1.0, 1.0, n)
        d[: n // 2] = 10.0
        d[-2:] = 1e-9, 1e9
        return d
    d[:2] = 0.3, 100.0
    return d


@pytest.mark.parametrize("kind", ["wall", "walls", "equal", "nested"])
@pytest.mark.parametrize("n", [63, 64, 65, 130, 1000, 1025, 2047, 2048, 2049, 5002, 9000, 70_001])
def test_one_tile(n, kind):
    from tests._gpu import run
    rng = np.random.default_rng(n)
    d = rng.permutation(_depths(kind, n, rng))
    az = np.full(n, 1.0) if kind == "equal" else rng.uniform(0.3, 2.8, n)   # (inside the left tile)
    el = rng.uniform(-0.5, 0.5, n) * (kind != "equal")
    pts = d[:, None] * np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], 1)
    surf = scenes.Surfels(pts.astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                          np.full((n, 2), math.log(0.002), np.float32), np.zeros(n, np.float32))
    tp, ip, rg, dk = run([surf], [scenes.Frame(8, 64, 8, 32, -1.4, 1.4)], read_bins=True)["bins"]
    assert rg[0, 0] == 0 and rg[0, 1] == n and np.all(tp[:n] == 0)   # (a surfel at the sensor lies in both tiles)
    assert np.array_equal(ip[:n], np.lexsort((np.arange(n), dk)).astype(ip.dtype))


def test_many_tiles():
    """60 tiles of 5,000 keys, every one with clusters, and short ones between."""
    from tests._gpu import run
    rng = np.random.default_rng(3)
    per, T = np.where(np.arange(120) % 2, 5000, 300), 120
    d = np.concatenate([_depths(("wall", "walls")[t // 2 % 2], per[t], rng) for t in range(T)])
    az = (np.repeat(np.arange(T), per) + 0.5) * 2 * np.pi / T
    pts = d[:, None] * np.stack([np.cos(az), np.sin(az), 0 * az], 1)
    n = len(d)
    surf = scenes.Surfels(pts.astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                          np.full((n, 2), math.log(0.002), np.float32), np.zeros(n, np.float32))
    tp, ip, rg, dk = run([surf], [scenes.Frame(8, 32 * T, 8, 32, -0.1, 0.1)], read_bins=True)["bins"]
    tile = np.repeat(np.arange(T), per)
    assert np.array_equal(rg[:, 1] - rg[:, 0], per)
    assert np.array_equal(ip, np.lexsort((np.arange(n), dk, tile)).astype(ip.dtype))
