"""The chunked backward sums the moments of up to 8 hits at a time over their
pixels, from 96 slots per warp, four lanes per hit.  Surfels that cover about
one pixel, a few, most and all of a 4 x 8 block, opaque and faint, in lists
around one and two chunks of 128 entries and of less than 8 hits; every
gradient value against the oracle within the parity tests' bar (not the share
of values within the bar without the cases' own uncertainty: one value of
these few hundred is more than the share those tests allow)."""
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


@pytest.mark.parametrize("spread", [0.1, 0.5, 1.5, 6.0])
@pytest.mark.parametrize("n,logit", [(1, 0.0), (9, -2.0), (33, -3.0), (128, -4.0), (129, -4.5), (300, 0.0)])
def test_gradients(oracle, n, logit, spread):
    from tests import _gpu
    from tests.test_gpu_parity import compare_grads, gpu_upstream, oracle_grads
    rng = np.random.default_rng(n)
    frame = scenes.Frame(16, 512, 8, 8, -0.13, 0.13)
    px = 2 * np.pi / 512
    # centres within one tile; 3 sigma of about `spread` pixels
    az = (4.0 + rng.uniform(-3.0, 3.0, n)) * px
    el = 0.13 - (4.0 + rng.uniform(-3.0, 3.0, n)) * 0.26 / 16
    r = rng.uniform(4.0, 40.0, n)
    mean = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1)
    surf = scenes.Surfels(mean.astype(np.float32), rng.normal(size=(n, 4)).astype(np.float32),
                          np.log(r[:, None] * px * spread / 3 * rng.uniform(0.7, 1.4, (n, 2))).astype(np.float32),
                          (logit + 0.3 * rng.normal(size=n)).astype(np.float32))
    g = _gpu.run([surf], [frame], targets=[scenes.targets_for(frame, surf, 7)])
    r = compare_grads(g["grads"][0], oracle_grads(oracle, surf, [frame], [gpu_upstream(g, 0)]))
    for name in ("mean", "quat", "log_scale", "logit"):
        assert r[name][0] <= 1.0, (name, r)
