"""Counting an item's tiles: a set of up to 32 tiles is walked by the item's
own thread, a larger one by its warp.  Surfels from a fraction of a tile to
around the sensor (every tile), mixed within each warp, across the azimuth
seam; frames with the CTA's shared counters (at most 4,096 tiles) and without;
a warp whose items lie in two frames.  Bins bit for bit against the oracle."""
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


@pytest.fixture(scope="module")
def oracle():
    from oracle import oracle as O
    O.build()
    return O


def mixed(n, seed):
    """Surfels whose cone's half angle runs over (nearly) all sizes."""
    rng = np.random.default_rng(seed)
    az, el = rng.uniform(-np.pi, np.pi, n), rng.uniform(-0.6, 0.6, n)
    az[::5] = np.pi * rng.choice([-1, 1], len(az[::5])) * rng.uniform(0.98, 1.0, len(az[::5]))
    r = rng.uniform(1.0, 20.0, n)
    mean = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1)
    scale = r[:, None] * np.exp(rng.uniform(np.log(0.002), np.log(0.6), (n, 1))) * rng.uniform(0.5, 1.0, (n, 2))
    return scenes.Surfels(mean.astype(np.float32), rng.normal(size=(n, 4)).astype(np.float32),
                          np.log(scale).astype(np.float32), rng.normal(size=n).astype(np.float32))


@pytest.mark.parametrize("n", [1, 37, 256, 777])
@pytest.mark.parametrize("H,W,th,tw,frames", [(64, 512, 8, 8, 1), (128, 2048, 8, 8, 1), (136, 2048, 8, 8, 1),
                                              (37, 100, 8, 8, 2), (64, 512, 16, 16, 3)])
def test_bins(oracle, n, H, W, th, tw, frames):
    from tests import _gpu
    surf = mixed(n, 11 * n + W)
    fr = []
    for f in range(frames):
        pose = np.array([1, 0, 0, 0.7 * f, 0, 1, 0, -0.4 * f, 0, 0, 1, 0.1 * f], np.float32)
        fr.append(scenes.Frame(H, W, th, tw, -0.7, 0.7, pose))
    tp, ip, rg, dk = _gpu.run([surf], fr, read_bins=True)["bins"]
    tiles = -(-H // th) * -(-W // tw)
    first, largest = 0, 0
    for f in range(frames):
        o = oracle.bin_frame(surf, fr[f])
        m = o["n_pairs"]
        t, i = tp[first:first + m].astype(np.int64) - f * tiles, ip[first:first + m].astype(np.int64) - f * n
        d = dk[f * n:(f + 1) * n]
        assert np.array_equal(d, o["depth_bits"])
        assert np.array_equal(i, o["vals"])
        assert np.array_equal((t.astype(np.uint64) << np.uint64(32)) | d[i].astype(np.uint64), o["keys"])
        r = rg[f * tiles:(f + 1) * tiles].astype(np.int64)
        assert np.array_equal(np.where(r[:, :1] < r[:, 1:], r - first, 0), o["ranges"])
        largest = max(largest, np.bincount(o["vals"].astype(np.int64)).max())
        first += m
    assert first == len(tp)
    if n >= 256:
        assert largest > 32      # a set for the whole warp
