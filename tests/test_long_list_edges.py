"""Lists beyond 4,096 entries in a tile that reaches past the frame, so that
some of its warps' pixel blocks lie partly or wholly outside: the backward's
queues, built from every block's word, against the oracle with the parity
tests' bars.  The workspace holds old data first: words of 2^20, or what a call
of another map, frame and tile shape left.  A second cluster of surfels lies in
a later tile, whose chunks are queued after the long list's."""
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


def _scene(shape, at, n, logit, seed):
    """n surfels within a pixel or so of at[0], 600 of at[1] (row, column)."""
    H, W, th, tw = shape
    p = 2 * np.pi / W
    frame = scenes.Frame(H, W, th, tw, -0.5 * H * p, 0.5 * H * p)
    rng = np.random.default_rng(seed)
    m = n + 600
    rc = np.repeat(np.float64(at), [n, 600], axis=0)
    az = (rc[:, 1] + 0.5 + rng.uniform(-1.0, 1.0, m)) * p
    el = 0.5 * H * p - (rc[:, 0] + 0.5 + rng.uniform(-0.4, 0.4, m)) * p
    r = rng.uniform(4.0, 40.0, m)
    mean = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1)
    surf = scenes.Surfels(mean.astype(np.float32), rng.normal(size=(m, 4)).astype(np.float32),
                          np.log(r[:, None] * p * rng.uniform(0.04, 0.25, (m, 2))).astype(np.float32),
                          (logit + 0.3 * rng.normal(size=m)).astype(np.float32))
    return surf, frame


SHAPES = [((32, 200, 16, 16), ((4, 196), (20, 100))),    # the last tile column's right blocks are outside
          ((16, 208, 8, 32), ((3, 200), (12, 40))),
          ((12, 64, 8, 8), ((10, 4), (10, 36))),         # the last tile row's lower blocks
          ((16, 100, 8, 8), ((3, 98), (12, 20))),        # half a block
          ((8, 200, 6, 16), ((6, 24), (7, 120)))]        # blocks of two rows of 16


@pytest.mark.parametrize("old", ["words", "call"])
@pytest.mark.parametrize("n,logit", [(4609, 2.0), (9000, -4.0)])
@pytest.mark.parametrize("shape,at", SHAPES, ids=lambda x: "x".join(map(str, x)) if len(x) == 4 else "")
def test_gradients_beside_the_frame(oracle, shape, at, n, logit, old):
    import torch
    from paper_2607_04127_gb300 import lib
    from tests import _gpu
    from tests.test_gpu_parity import (assert_forward, assert_grads, compare_forward, compare_grads, gpu_upstream,
                                       oracle_grads)
    surf, frame = _scene(shape, at, n, logit, n)
    sess = lib.Session()
    if old == "words":
        sess.reserve([surf.n], [lib.frame_struct(frame)], [0], 8 * surf.n)
        sess.ws[:sess.ws.numel() // 4 * 4].view(torch.int32).fill_(1 << 20)
    else:
        s0, f0 = _scene((16, 512, 8, 8), ((4, 100), (12, 300)), 20_000, 0.0, 1)
        _gpu.run([s0], [f0], targets=[scenes.targets_for(f0, s0, 3)], session=sess)
    g = _gpu.run([surf], [frame], targets=[scenes.targets_for(frame, surf, 7)], session=sess)
    sess.close()
    o = oracle.bin_frame(surf, frame)
    assert (o["ranges"][:, 1] - o["ranges"][:, 0]).max() > 4096
    assert_forward(compare_forward(g["fwd"][0], oracle.render_fwd(surf, frame, o["ranges"], o["vals"])))
    assert_grads(compare_grads(g["grads"][0], oracle_grads(oracle, surf, [frame], [gpu_upstream(g, 0)])))
