"""Diagnostics of moment fields of tiny grids spread their rows over blocks (a tile's rows are a serial
chain) and give the plain sums and differences."""
import numpy as np
import pytest

from captured_launches import launches
from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import smooth_random_fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("nx,ny,tiles", [(3, 3, 1), (4, 4, 1), (8, 8, 1), (8, 17, 2), (33, 35, 12), (64, 31, 16),
                                         (64, 64, 16), (64, 96, 16), (64, 97, 13), (65, 16, 16), (65, 17, 9)])
def test_rows_are_spread_and_the_values_are_the_sums(nx, ny, tiles):
    """Sums in any order: 1e-13 of the terms' scale; maxima of a few roundings of values below 0.2."""
    import torch
    rho, ux, uy, bx, by = f = smooth_random_fields(nx, ny, seed=nx * ny, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
    dev = [torch.tensor(a, device="cuda") for a in f]
    out = torch.empty(lbmhd.LBMHD_NDIAG + 1, dtype=torch.float64, device="cuda")
    lbmhd.lbmhd_diagnostics_fields_noalloc(dev, out)
    got = out.cpu().numpy()
    stream = torch.cuda.Stream()
    kernels = launches(stream, lambda: lbmhd.lbmhd_diagnostics_fields_noalloc(dev, out, stream=stream.cuda_stream))
    assert max(grid[0] for grid, block in kernels if block[0] == 128) == tiles
    want = [rho.sum(), (rho * ux).sum(), (rho * uy).sum(), bx.sum(), by.sum(), 0.5 * (rho * (ux**2 + uy**2)).sum(),
            0.5 * (bx**2 + by**2).sum()]
    scale = np.array([1, 0.2, 0.2, 0.2, 0.2, 0.02, 0.02]) * nx * ny * 1e-13
    assert np.all(np.abs(got[:7] - want) <= scale)
    dx = lambda a: 0.5 * (np.roll(a, -1, 1) - np.roll(a, 1, 1))  # noqa: E731
    dy = lambda a: 0.5 * (np.roll(a, -1, 0) - np.roll(a, 1, 0))  # noqa: E731
    assert abs(got[8] - np.abs(dx(bx) + dy(by)).max()) <= 4e-16
    assert got[-1] == 0.0
