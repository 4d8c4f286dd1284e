"""Tracking targets' covariances and weights at the edges of the CTAs' shares
(1,024 surfels, rounds of 256), where the minimum and maximum anisotropy of the
selection are reduced: every value against the same formulas in 64 bits.

Bars, u = 2^-24: the quaternion's components after normalising are within 6 u
relative, a rotation's entry then within 28 u, so a covariance entry, sums of two
entries and a squared scale (9 u), within 128 u of the largest squared scale.  A
kappa is within 11 u (two exponentials of 4 u, a sum, a quotient), so kb = (kappa -
min) / (max - min) within 50 u max / (max - min), and the weight min(1 / (kb +
eps), w_max) lies between those of kb plus and minus that, and 4 u.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.mark.parametrize("share", [0.0, 0.02, 0.5, 1.0])
@pytest.mark.parametrize("n", [1, 33, 255, 257, 1023, 1024, 1025, 2049, 70_001])
def test_covariances_and_weights(n, share):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build, track
    build.build()
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    P = [10 * r(n, 3), r(n, 4), 0.3 * r(n, 2) - 2.0, r(n)]
    mask = (torch.rand(n, generator=g, device="cuda") < share).to(torch.uint8)
    kf = torch.full((n,), 5, device="cuda", dtype=torch.int32)
    P[3] = P[3].abs()
    idx, mean, cov, w = track.trackable_targets(P, mask, kf, 2, 0.5)
    i = torch.nonzero(mask)[:, 0]
    assert torch.equal(idx.long(), i) and len(mean) == len(cov) == len(w) == len(i)
    if len(i) == 0:
        return
    q = P[1][i].double()
    a, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - a * z), 2 * (x * z + a * y),
                     2 * (x * y + a * z), 1 - 2 * (x * x + z * z), 2 * (y * z - a * x),
                     2 * (x * z - a * y), 2 * (y * z + a * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    s = torch.exp(P[2][i].double())
    lam = torch.cat([s * s, torch.full_like(s[:, :1], float(np.float32(0.01)) ** 2)], 1)
    C = R @ torch.diag_embed(lam) @ R.transpose(1, 2)
    want = torch.stack([C[:, j, k] for j, k in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))], 1)
    assert ((cov.double() - want).abs() <= 128 * U * lam.amax(1, keepdim=True)).all()
    eps, w_max = float(np.float32(1e-6)), 10.0
    kap = s.amax(1) / (s.amin(1) + eps)
    span = kap.max() - kap.min()
    kb = (kap - kap.min()) / span if float(span) > 0 else torch.zeros_like(kap)
    err = 50 * U * kap.max() / span if float(span) > 0 else torch.zeros_like(span)
    lo, hi = (1 / (kb + err + eps)).clamp(max=w_max), (1 / ((kb - err).clamp(min=0.0) + eps)).clamp(max=w_max)
    assert (w.double() >= lo * (1 - 4 * U)).all() and (w.double() <= hi * (1 + 4 * U)).all()
