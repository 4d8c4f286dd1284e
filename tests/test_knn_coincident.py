"""The k-NN with many coincident points (a sensor's empty returns at the origin
among them): the sets are the lowest indices (exact, against the oracle), and a
query does not visit the leaves of all of them (a query visits a few leaves on
each level: bounded by 1,024 distances on average, where the pairs of
coincident points alone are 5,000 a point)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [3, 20, 32])
@pytest.mark.parametrize("at", [(0.0, 0.0, 0.0), (7.5, -3.25, 1.125)])
def test_half_of_the_points_coincide(at, k):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import init
    from paper_2607_04127_gb300 import build, keyframe
    build.build()
    n = 40_000
    rng = np.random.default_rng(k)
    pts = (rng.normal(size=(n, 3)) * [20.0, 8.0, 2.0]).astype(np.float32)
    dup = rng.random(n) < 0.5
    pts[dup] = at
    pairs = torch.zeros(1, dtype=torch.int64, device="cuda")
    out = keyframe.initialise(torch.from_numpy(pts).cuda(), np.eye(3, 4).ravel(), keyframe.params(k=k), pairs=pairs)
    rows = np.unique(np.concatenate([rng.integers(0, n, 300), np.nonzero(dup)[0][[0, 1, -1]]]))
    assert np.array_equal(out["knn"].cpu().numpy()[rows], init.knn(pts, k, rows=rows)[0])
    assert int(pairs) <= 1024 * n
