"""Block means of narrow grids, several rows of means to a block, and of wide filters: the sequential
binary64 sum (row by row from the left, one product), and few idle lanes."""
import numpy as np
import pytest

from captured_launches import launches
from paper_1705_09807_gb300 import lbmhd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("mx,my,r", [(1, 1, 1), (1, 77824, 2), (1, 77825, 3), (3, 26000, 1), (42, 1900, 2), (43, 1300, 3),
                                     (64, 1217, 2), (127, 700, 1), (128, 3, 2), (2, 40000, 4), (1, 1, 31), (2, 3, 32),
                                     (3, 1, 33), (1, 2, 64), (1, 1, 131)])
def test_sequential_sums(mx, my, r):
    import torch
    f = np.random.default_rng(r).normal(size=(my * r, mx * r))
    out = torch.zeros((my, mx), dtype=torch.float64, device="cuda")
    lbmhd.lbmhd_block_mean_device(torch.tensor(f, device="cuda"), r, out)
    want = np.zeros((my, mx))
    for yy in range(r):
        for xx in range(r):
            want += f[yy::r, xx::r]
    np.testing.assert_array_equal(out.cpu().numpy(), want * (1.0 / (float(r) * r)))


@pytest.mark.parametrize("mx", [1, 3, 8, 33, 64])
def test_few_idle_lanes(mx):
    import torch
    f = torch.ones((1 << 17, 2 * mx), dtype=torch.float64, device="cuda")
    out = torch.zeros((1 << 16, mx), dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    (grid, block), = launches(stream, lambda: lbmhd.lbmhd_block_mean_device(f, 2, out, stream=stream.cuda_stream))
    assert np.prod(grid) * (-(-np.prod(block) // 32) * 32) <= 1.5 * mx * (1 << 16)
