"""The k-NN of keyframe initialisation at the edges of its structure: leaves
of 32 points, nodes of 1,024, batches of 32,768, sort CTAs of 2,048 keys (up
to 2^18 points) and 8,192 beyond, and clouds whose extent vanishes on some
axes (fewer bits of the Morton code).  The neighbour sets are specified
binary32 outcomes, so the comparison with the oracle is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build
    build.build()


def _check(pts, k, rows):
    import torch
    from oracle import init
    from paper_2607_04127_gb300 import keyframe
    pts = np.ascontiguousarray(pts, np.float32)
    out = keyframe.initialise(torch.from_numpy(pts).cuda(), np.eye(3, 4).ravel(), keyframe.params(k=k))
    got = out["knn"][:len(pts)].cpu().numpy()[rows]
    assert np.array_equal(got, init.knn(pts, k, rows=rows)[0])


@pytest.mark.parametrize("n,k", [(3, 3), (31, 8), (32, 32), (33, 32), (1023, 20), (1024, 20), (1025, 24), (2048, 20),
                                 (2049, 5), (32767, 20), (32769, 20), (262144, 20), (262145, 20), (400003, 32)])
def test_sizes(n, k):
    """Clusters of very different density (k-th distances from 1 cm to tens
    of metres), so that neighbours lie in other leaves, nodes and batches."""
    rng = np.random.default_rng(n)
    c = rng.uniform(-60, 60, (12, 3))
    s = 10.0 ** rng.uniform(-1.5, 1.2, 12)
    j = rng.integers(0, 12, n)
    rows = np.unique(np.concatenate([rng.integers(0, n, 300), [0, n - 1]]))
    _check(c[j] + s[j, None] * rng.normal(size=(n, 3)), k, rows)


@pytest.mark.parametrize("axes", [(), (0,), (2,), (0, 1), (1, 2)])
def test_flat_extents(axes):
    """Points that differ on the given axes only (all coincident for none),
    on a coarse grid with many exact ties."""
    rng = np.random.default_rng(7)
    pts = np.full((3000, 3), 2.5)
    for a in axes:
        pts[:, a] = rng.integers(0, 200, 3000) * 0.25
    _check(pts, 20, np.arange(0, 3000, 13))
