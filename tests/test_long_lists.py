"""Lists beyond 4,096 entries: their masks are found segment by segment (512
entries) for 32 pixels at a time, then every pixel is composited on its own.
Sizes around the limit and a segment's, warps of 4 x 8 pixels and of other
shapes, opaque surfels (later segments skipped behind the stop) and faint ones
(the whole list walked), and a second forward of the same binning (bit for
bit); against the oracle with the parity tests' bars."""
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


@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (2, 16)])
@pytest.mark.parametrize("n,logit", [(4097, 0.0), (4608, -3.0), (4609, 2.0), (9000, -4.0), (20_000, 1.0)])
def test_forward_and_gradients(oracle, n, logit, tile):
    from tests import _gpu
    from tests.test_gpu_parity import (assert_forward, assert_grads, compare_forward, compare_grads, gpu_upstream,
                                       oracle_grads)
    rng = np.random.default_rng(n)
    frame = scenes.Frame(16, 512, tile[0], tile[1], -0.13, 0.13)
    # all within a few pixels about the centre of one tile of every shape
    az = (4.0 + rng.uniform(-1.0, 1.0, n)) * 2 * np.pi / 512
    el = 0.13 - (1.0 + rng.uniform(-0.4, 0.4, n)) * 0.26 / 16
    r = rng.uniform(4.0, 40.0, n)
    mean = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1)
    surf = scenes.Surfels(mean.astype(np.float32), rng.normal(size=(n, 4)).astype(np.float32),
                          np.log(r[:, None] * rng.uniform(0.0005, 0.003, (n, 2))).astype(np.float32),
                          (logit + 0.3 * rng.normal(size=n)).astype(np.float32))
    tgt = scenes.targets_for(frame, surf, 7)
    g = _gpu.run([surf], [frame], targets=[tgt])
    again = _gpu.run([surf], [frame], repeat_fwd=2)
    for k, v in g["fwd"][0].items():
        assert np.array_equal(v, again["fwd"][0][k])
    o = oracle.bin_frame(surf, frame)
    assert (o["ranges"][:, 1] - o["ranges"][:, 0]).max() > 4096
    assert_forward(compare_forward(g["fwd"][0], oracle.render_fwd(surf, frame, o["ranges"], o["vals"])))
    assert_grads(compare_grads(g["grads"][0], oracle_grads(oracle, surf, [frame], [gpu_upstream(g, 0)])))
