"""Read-out of grids at the widths where a block's shape changes: the same fields repeated to a wide
grid read out the same, bit for bit, and a narrow grid's launch has few idle lanes."""
import numpy as np
import pytest

from captured_launches import launches
from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import smooth_random_fields

pytestmark = pytest.mark.gpu
FORMS = [lbmhd.LBMHD_FP64, lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


def _moments(fields, precision):
    ny, nx = fields[0].shape
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 2.0, precision)
    with lbmhd.Lbmhd(p, *fields) as sim:
        sim.step(5)
        return np.stack(sim.moments())


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("nx,ny", [(3, 3), (3, 86), (4, 65), (5, 700), (16, 17), (17, 16), (33, 8), (64, 5), (85, 4),
                                   (86, 3), (127, 3), (128, 3), (129, 4), (160, 3), (257, 3)])
def test_moments_equal_those_of_the_repeated_fields(nx, ny, precision):
    fields = smooth_random_fields(nx, ny, seed=nx, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
    k = 2 if nx > 64 else -(-130 // nx)
    got = _moments(fields, precision)
    want = _moments([np.tile(f, (1, k)) for f in fields], precision)
    assert np.array_equal(np.tile(got, (1, 1, k)), want)


@pytest.mark.parametrize("nx", [3, 5, 16, 33, 65, 100, 129, 160])
def test_few_idle_lanes(nx):
    """At most half as many lanes again as cells, with blocks rounded up to whole warps."""
    import torch
    ny = 1 << 14
    stream = torch.cuda.Stream()
    f = [torch.full((ny, nx), v, dtype=torch.float64, device="cuda") for v in (1.0, 0.0, 0.0, 0.0, 0.0)]
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 0.0, lbmhd.LBMHD_FP32)
    p.cuda_stream = stream.cuda_stream
    torch.cuda.synchronize()
    with lbmhd.Lbmhd(p, *f, device=True) as sim:
        torch.cuda.synchronize()
        (grid, block), = launches(stream, lambda: sim.moments_device(f))
    lanes = np.prod(grid) * (-(-np.prod(block) // 32) * 32)
    assert lanes <= 1.5 * nx * ny
