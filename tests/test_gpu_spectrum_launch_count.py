"""lbmhd_launch_count counts the kernels of a spectrum for both transforms (mixed radix, Bluestein)."""
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


@pytest.mark.parametrize("n", [36, 37, 2050])
def test_spectrum_launches_are_counted(n):
    import torch
    fields = [torch.zeros((n, n), dtype=torch.float64, device="cuda") for _ in range(4)]
    out = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2)]
    work = torch.zeros(lbmhd.lbmhd_energy_spectrum_work_bytes(n), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        kernels = len(launches(stream, lambda: lbmhd.lbmhd_energy_spectrum_device(
            *fields, n, *out, work, stream=stream.cuda_stream)))
    p = lbmhd.lbmhd_params_srt(n, n, 0.01, 0.01, 0.0, lbmhd.LBMHD_FP32)
    with lbmhd.Lbmhd(p, *smooth_random_fields(n, n, seed=1)) as sim:
        sim.moments()
        before = sim.launches
        e_kin, _ = sim.spectrum(n)
        assert sim.launches == before + 1 + kernels  # the read-out and the transform
        assert np.all(np.isfinite(e_kin))
