"""Tiles of few keys, sorted by a warp (up to 64 keys), beside tiles sorted by a CTA
and long buckets, on the path of small maps and of large ones: NumPy's order of
(tile, depth key, item), exact."""
import math

import numpy as np
import pytest

from paper_2607_04127_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fill", [0, 2500, 40_000])
@pytest.mark.parametrize("first", [0, 31, 33, 60])
def test_tile_by_tile(first, fill):
    """90 tiles of `first`, first + 1, ... surfels (modulo 80), then one of `fill`."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build
    build.build()
    from tests._gpu import run
    rng = np.random.default_rng(first + fill)
    per = np.append((np.arange(90) + first) % 80, fill)
    T, n = len(per), int(per.sum())
    tile = rng.permutation(np.repeat(np.arange(T), per))
    az, d = (tile + 0.5) * 2 * np.pi / T, rng.choice(rng.uniform(2.0, 60.0, 40), n)   # (many equal depths)
    pts = d[:, None] * np.stack([np.cos(az), np.sin(az), 0 * az], 1)
    surf = scenes.Surfels(pts.astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                          np.full((n, 2), math.log(0.002), np.float32), np.zeros(n, np.float32))
    tp, ip, rg, dk = run([surf], [scenes.Frame(4, 16 * T, 4, 16, -0.1, 0.1)], read_bins=True)["bins"]
    assert np.array_equal(rg[:, 1] - rg[:, 0], per)
    assert np.array_equal(ip, np.lexsort((np.arange(n), dk, tile)).astype(ip.dtype))


def test_dense_call():
    """Above 32 surfels a tile every bucket takes a CTA, tiles of 0 to 70 keys among
    them."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build
    build.build()
    from tests._gpu import run
    rng = np.random.default_rng(5)
    per = np.append(np.arange(71), [900, 2048, 2049])
    T, n = len(per), int(per.sum())
    tile = rng.permutation(np.repeat(np.arange(T), per))
    az, d = (tile + 0.5) * 2 * np.pi / T, rng.uniform(2.0, 60.0, n)
    pts = d[:, None] * np.stack([np.cos(az), np.sin(az), 0 * az], 1)
    surf = scenes.Surfels(pts.astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                          np.full((n, 2), math.log(0.002), np.float32), np.zeros(n, np.float32))
    assert n >= 32 * T
    tp, ip, rg, dk = run([surf], [scenes.Frame(4, 16 * T, 4, 16, -0.1, 0.1)], read_bins=True)["bins"]
    assert np.array_equal(rg[:, 1] - rg[:, 0], per)
    assert np.array_equal(ip, np.lexsort((np.arange(n), dk, tile)).astype(ip.dtype))
