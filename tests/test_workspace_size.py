"""What a pair costs in the workspace: its key, tile and item (16 bytes), its
share of the chunk checkpoints (24 bytes a pixel and 128 entries), the window
masks (16) and the backward's queue, and at most as much again for the long
lists as a suffix per chunk and pixel (4 bytes)."""
import pytest

from paper_2607_04127_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(4, 8), (8, 8), (8, 16), (16, 16), (8, 32)])
def test_bytes_per_pair(tile):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build, lib
    build.build()
    frame = lib.frame_struct(scenes.Frame(128, 1024, *tile, -0.7, 0.7))
    sess = lib.Session()
    a, b = 1 << 20, 1 << 24
    size = [lib.lgs_batch_workspace_size(sess.handle, [200_000], [frame], [0], p) for p in (a, b)]
    sess.close()
    px = tile[0] * tile[1]
    assert (size[1] - size[0]) / (b - a) <= 16 + (24 + 16 + 4) * px / 128 + 8 * (px / 32) / 128
