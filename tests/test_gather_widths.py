"""Map management's gather of per-surfel arrays at every load width."""
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


@pytest.mark.parametrize("words", [1, 2, 3, 4, 10, 12])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_gather_word_widths(words, offset):
    """Rows of every width and alignment (16-, 8- and 4-byte loads), with and
    without zeroed children: the rows of their parents, exactly."""
    import torch
    from paper_2607_04127_gb300 import lib
    n, cap = 1000, 1103
    rng = np.random.default_rng(words)
    src = torch.from_numpy(rng.integers(0, n, cap).astype(np.int32)).cuda()
    role = torch.from_numpy(rng.integers(0, 3, cap).astype(np.uint8)).cuda()
    counts = torch.tensor([cap - 3, 0, 0, 0, 0, 0], dtype=torch.int64, device="cuda")
    a = torch.randint(-2**31, 2**31 - 1, (n * words + offset,), dtype=torch.int32, device="cuda")[offset:]
    for zero in (0, 1):
        out = torch.full((cap * words + offset,), 7, dtype=torch.int32, device="cuda")[offset:]
        lib.lgs_map_gather(src.data_ptr(), role.data_ptr(), counts.data_ptr(), cap, a.data_ptr(), out.data_ptr(), words,
                           zero, torch.cuda.current_stream().cuda_stream)
        want = a.view(n, words)[src.long()]
        if zero:
            want = torch.where((role != 0)[:, None], 0, want)
        want[cap - 3:] = 7
        assert torch.equal(out.view(cap, words), want)
