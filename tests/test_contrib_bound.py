"""The backward reads n_contrib from the caller's buffers and never walks past a
tile's list: with every pixel's count raised far beyond it (nothing stopped a
pixel, so the entries after its last composited one add nothing) the gradients
are the same, for short lists and long ones (more than 4,096 entries)."""
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


@pytest.mark.parametrize("n", [3000, 5000])
def test_raised_counts(oracle, n):
    import torch
    from paper_2607_04127_gb300 import render
    from tests.test_gpu_parity import assert_grads, compare_grads, oracle_grads
    rng = np.random.default_rng(n)
    frame = scenes.Frame(16, 512, 8, 8, -0.13, 0.13)
    az = (4.0 + rng.uniform(-2.0, 2.0, n)) * 2 * np.pi / 512
    el = 0.13 - (4.0 + rng.uniform(-2.0, 2.0, n)) * 0.26 / 16
    r = rng.uniform(4.0, 40.0, n)
    mean = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1)
    surf = scenes.Surfels(mean.astype(np.float32), rng.normal(size=(n, 4)).astype(np.float32),
                          np.log(r[:, None] * rng.uniform(0.0005, 0.003, (n, 2))).astype(np.float32),
                          (-4.0 + 0.3 * rng.normal(size=n)).astype(np.float32))
    rast = render.Rasterizer([frame])
    params = [render.map_tensors(surf)]
    S = rast.bin_sort(params)
    out = rast.forward(params, S)[0]
    g = torch.Generator(device="cuda").manual_seed(n)
    up = [tuple(torch.randn(*s, 16, 512, generator=g, device="cuda") for s in ((), (), (3,)))]
    assert float(out.T_final.min()) > 2e-4          # no pixel stopped
    out.n_contrib.fill_(1 << 30)
    grads = [[torch.zeros_like(p) for p in params[0]]]
    rast.backward(params, grads, upstream=up, S=S)
    torch.cuda.synchronize()
    rast.close()
    want = oracle_grads(oracle, surf, [frame], [tuple(u.double().cpu().numpy() for u in up[0])], scale_reg=False)
    assert_grads(compare_grads([x.cpu().numpy() for x in grads[0]], want))
