"""Which unfiltered grids (Delta = 0) take the plain step: tall grids of few strips return to the filtered
form's blocks at a smaller size than wide ones.  Read from captured launches; and the two forms agree
on either side of the line."""
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


FP32, FP16, REL = lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL


# (columns, form, MiB of a state copy below and above the line)
@pytest.mark.parametrize("nx,precision,below,above", [
    (32, FP32, 120, 134), (33, FP32, 50, 60), (128, FP32, 50, 60), (129, FP32, 66, 78), (384, FP32, 98, 110),
    (897, FP32, 120, 134), (128, FP16, 50, 60), (256, FP16, 50, 60), (300, FP16, 82, 94), (896, FP16, 98, 110),
    (897, FP16, 120, 134), (64, REL, 120, 134), (65, REL, 50, 60), (204, REL, 120, 134), (205, REL, 66, 78),
    (300, REL, 120, 134), (384, REL, 98, 110)])
def test_plain_form_by_strips_and_size(nx, precision, below, above):
    import torch
    elem, planes = {lbmhd.LBMHD_FP32: (4, 27), lbmhd.LBMHD_FP16: (2, 27), lbmhd.LBMHD_FP16_REL: (2, 29)}[precision]
    row = (nx + 34 + 31) // 32 * 32 * planes * elem
    stream = torch.cuda.Stream()
    for mib, plain in ((below, True), (above, False)):
        ny = (mib << 20) // row
        y, x = torch.arange(ny, device="cuda")[:, None], torch.arange(nx, device="cuda")[None, :]
        wave = (torch.sin(0.1 * x + 0.003 * y) * 0.03).double().expand(ny, nx).contiguous()
        fields = [1 + wave, wave, wave * 0.5, wave * 0.7, -wave]
        torch.cuda.synchronize()
        grids, pops = [], []
        for delta in (0.0, 1e-30):  # 1e-30: the filtered form, with vanishing gradients
            p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, delta, precision)
            p.cuda_stream = stream.cuda_stream
            with lbmhd.Lbmhd(p, *fields, device=True) as sim:
                torch.cuda.synchronize()
                sim.step(2)
                out = torch.empty((5, ny, nx), dtype=torch.float64, device="cuda")
                torch.cuda.synchronize()
                sim.moments_device(list(out))
                torch.cuda.synchronize()
                pops.append(out)
                grids.append([g for g, _ in launches(stream, lambda: sim.step(1))])
        assert (grids[0] != grids[1]) == plain  # more blocks of the plain form fit an SM
        # (binary32 may contract differently: an ulp of the deviations a step, at most doubled by the
        # relaxation, in each of the nine populations of a moment)
        worst = float((pops[0] - pops[1]).abs().max())
        assert worst <= (9 * 2 * 2 * 2.0 ** -26 if precision == lbmhd.LBMHD_FP32 else 0.0)
