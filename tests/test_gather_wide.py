"""Map management's gather at the edges of a CTA's 1,024 loads: rows of one load,
rows that a share divides, rows wider than a share (few of them, as many
CTAs)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,words", [(1, 1), (1023, 1), (1025, 4), (1024, 1023), (7, 1024), (5, 4097), (3, 65_536),
                                        (130, 514)])
def test_rows_against_indexing(rows, words):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_04127_gb300 import build, lib
    build.build()
    rng = np.random.default_rng(rows + words)
    n = rows + 3
    src = torch.from_numpy(rng.integers(0, n, rows).astype(np.int32)).cuda()
    role = torch.from_numpy(rng.integers(0, 3, rows).astype(np.uint8)).cuda()
    counts = torch.tensor([rows - 1 if rows > 1 else 1, 0, 0, 0, 0, 0], dtype=torch.int64, device="cuda")
    a = torch.randint(-2**31, 2**31 - 1, (n, words), dtype=torch.int32, device="cuda")
    for zero in (0, 1):
        out = torch.full((rows, words), 7, dtype=torch.int32, device="cuda")
        lib.lgs_map_gather(src.data_ptr(), role.data_ptr(), counts.data_ptr(), rows, a.data_ptr(), out.data_ptr(), words,
                           zero, torch.cuda.current_stream().cuda_stream)
        want = a[src.long()]
        if zero:
            want = torch.where((role != 0)[:, None], 0, want)
        want[int(counts[0]):] = 7
        assert torch.equal(out, want)
