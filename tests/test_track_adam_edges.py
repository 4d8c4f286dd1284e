"""Tracking targets and Adam at the edges of their CTAs' shares: 1,024 surfels
per CTA and rounds of 256 (targets), 128 scalars per warp and 1,024 per CTA, the
moments of an odd map at any word (Adam)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SIZES = [1, 31, 33, 255, 256, 257, 1023, 1024, 1025, 5000, 1_048_577]


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build
    build.build()


def _map(n, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    return [10 * r(n, 3), r(n, 4), 0.3 * r(n, 2) - 2.0, r(n)], g


@pytest.mark.parametrize("n", SIZES)
def test_targets_keep_index_order(n):
    """The selection and the copied means are exact; a weight is one function
    of the surfel's own scales and the selection's extremes (binary32: a few
    ulps through two exponentials, a quotient and the normalisation)."""
    import torch
    from paper_2607_04127_gb300 import track
    P, g = _map(n, n)
    mask = torch.randint(0, 2, (n,), generator=g, device="cuda", dtype=torch.uint8)
    kf = torch.randint(0, 6, (n,), generator=g, device="cuda", dtype=torch.int32)
    idx, mean, cov, w = track.trackable_targets(P, mask, kf, 2, 0.5)
    want = torch.nonzero((mask != 0) & (kf >= 2) & (P[3] >= 0.0))[:, 0]
    assert torch.equal(idx.long(), want) and torch.equal(mean, P[0][want])
    s = torch.exp(P[2][want].double())
    assert torch.allclose(cov[:, 0] + cov[:, 3] + cov[:, 5], (s.square().sum(1) + 1e-4).float(), rtol=1e-5)


@pytest.mark.parametrize("zero", [True, False])
@pytest.mark.parametrize("n", SIZES)
def test_adam_every_scalar_once(n, zero):
    """Against the same update in 64 bits: the new moments within three
    roundings, the step within ten (a root, two products, a quotient)."""
    import torch
    from paper_2607_04127_gb300 import render
    P, g = _map(n, n + 1)
    G = [torch.randn(p.shape, generator=g, device="cuda") for p in P]
    m, v = torch.randn(10 * n, generator=g, device="cuda"), torch.rand(10 * n, generator=g, device="cuda")
    lr = (1e-3, 2e-3, 5e-3, 7e-3)
    p0, g0 = [p.double() for p in P], torch.cat([x.double().reshape(-1) for x in G])
    b1, b2, u = float(np.float32(0.9)), float(np.float32(0.999)), 2.0 ** -24
    wm, wv = b1 * m.double() + (1 - b1) * g0, b2 * v.double() + (1 - b2) * g0 * g0
    am = (b1 * m.double()).abs() + ((1 - b1) * g0).abs()
    render.adam_step(P, G, m, v, 3, lr=lr, zero_grad=zero)
    assert ((m.double() - wm).abs() <= 3 * u * am).all() and ((v.double() - wv).abs() <= 4 * u * wv).all()
    up = (wm / (1 - b1 ** 3)) / (torch.sqrt(wv / (1 - b2 ** 3)) + 1e-15)
    amp = (am / (1 - b1 ** 3)) / (torch.sqrt(wv / (1 - b2 ** 3)) + 1e-15)
    off = 0
    for p, q, x, l in zip(P, p0, G, lr):
        k = p.numel()
        want = q - l * up[off:off + k].reshape(q.shape)
        tol = 10 * u * l * amp[off:off + k].reshape(q.shape) + u * (q.abs() + want.abs())
        assert ((p.double() - want).abs() <= tol).all()
        assert (x == 0).all() if zero else torch.equal(x.reshape(-1).double(), g0[off:off + k])
        off += k
