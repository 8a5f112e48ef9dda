"""Binary32 forward pass of many narrow, low or small grids (a thread per cell) against the same cells on
grids that fill the tiles: periodic repetition leaves every cell's neighbours, hence its bits."""
import numpy as np
import pytest

from oracle import closure as oc
from paper_1705_09807_gb300 import lbmhd

pytestmark = pytest.mark.gpu
ONES = (np.ones(12, np.float32), np.ones(4, np.float32))


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("b,h,w", [(1, 5000, 1), (1, 9800, 3), (2, 4900, 10), (1, 1, 9800), (3, 2, 3300), (400, 4, 4),
                                   (310, 5, 31), (305, 1, 1)])
def test_forward_of_narrow_grids(b, h, w):
    import torch
    rng = np.random.default_rng(b + h + w)
    x = rng.normal(size=(b, 12, h, w)).astype(np.float32)
    ry, rx = -(-32 // h), -(-32 // w)  # sides of at least a tile
    wide = torch.tensor(np.tile(x, (1, 1, ry, rx)), device="cuda")
    x = torch.tensor(x, device="cuda")
    got = torch.empty((b, 4, h, w), device="cuda")
    want = torch.empty((b, 4, h * ry, w * rx), device="cuda")
    with lbmhd.Closure(oc.init_params(4), *ONES) as cl:
        cl.forward(x, got, tensor_cores=False)
        cl.forward(wide, want, tensor_cores=False)
    assert torch.equal(got.repeat(1, 1, ry, rx), want)
