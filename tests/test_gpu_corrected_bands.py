"""Corrected steps of an unfiltered grid (Delta = 0) launch the blocks that the corrected steps of a
filtered one do -- the same kernel with the same number of blocks per SM -- although the grid's own
steps, in the plain form, take other bands.  The launches are read from a captured graph."""
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


def _grids(sim, stream):
    """Grid dimensions of the kernels that one step of `sim` launches."""
    return sorted(grid for grid, _ in launches(stream, lambda: sim.step(1)))


@pytest.mark.parametrize("precision,n", [(lbmhd.LBMHD_FP64, 130), (lbmhd.LBMHD_FP64, 512), (lbmhd.LBMHD_FP64, 1024),
                                         (lbmhd.LBMHD_FP32, 64), (lbmhd.LBMHD_FP32, 600), (lbmhd.LBMHD_FP32, 850)])
def test_corrected_steps_have_their_own_bands(precision, n):
    import torch
    fields = [torch.full((n, n), v, dtype=torch.float64, device="cuda") for v in (1.0, 0.01, 0.0, 0.02, 0.0)]
    corr = torch.zeros((4, n, n), dtype=torch.float32, device="cuda")
    rng = np.random.default_rng(0)
    net = lbmhd.Closure(rng.uniform(-0.1, 0.1, 13892), np.ones(12), np.ones(4))
    stream = torch.cuda.Stream()
    grids = {}
    for delta in (0.0, 2.0):
        p = lbmhd.lbmhd_params_srt(n, n, 0.02, 0.02, delta, precision)
        p.cuda_stream = stream.cuda_stream
        torch.cuda.synchronize()
        with lbmhd.Lbmhd(p, *fields, device=True) as sim:
            torch.cuda.synchronize()
            own = _grids(sim, stream)
            lbmhd.lbmhd_set_correction_device(sim.h, corr)
            static = _grids(sim, stream)
            lbmhd.lbmhd_set_correction_device(sim.h, None)
            net.attach(sim.h)
            learned = _grids(sim, stream)
            lbmhd.lbmhd_detach_closure(sim.h)
            assert _grids(sim, stream) == own
        grids[delta] = (static, learned)
    assert len(grids[0.0][0]) == 1 and len(grids[0.0][1]) == 2
    assert grids[0.0] == grids[2.0]
    net.free()
