"""Diagnostics of a tall narrow grid when the device has no memory for the moment fields: straight from the
populations, with the same values."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("precision", [lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL])
def test_diagnostics_without_memory_for_the_fields(precision):
    import torch
    nx, ny = 64, 1 << 17  # 336 MB of moment fields
    f = smooth_random_fields(nx, ny, seed=1, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.01, 0.01, 0.0, precision)
    lbmhd.lbmhd_release_cached_memory()
    torch.cuda.empty_cache()
    with lbmhd.Lbmhd(p, *f) as sim:
        free, _ = torch.cuda.mem_get_info()
        rest = torch.empty(free - (200 << 20), dtype=torch.uint8, device="cuda")
        try:
            straight = sim.diagnostics()
        finally:
            del rest
            torch.cuda.empty_cache()
        fields = sim.diagnostics()
        sim.step(1)
        sim.diagnostics()
    # sums of 2^23 terms of at most 2 in another order; maxima of the same differences
    assert np.allclose(straight[:7], fields[:7], rtol=1e-13, atol=1e-6)
    assert np.allclose(straight[7:], fields[7:], rtol=1e-12, atol=1e-15)
