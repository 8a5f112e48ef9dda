"""Memory kept from freed handles, returned by a thread that has made no CUDA call before."""
import threading

import pytest

from paper_1705_09807_gb300 import lbmhd

pytestmark = pytest.mark.gpu


def test_release_from_a_new_thread():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()
    one = torch.ones((2048, 2048), dtype=torch.float64, device="cuda")
    zero = torch.zeros_like(one)
    p = lbmhd.lbmhd_params_srt(2048, 2048, 0.02, 0.02, 0.0, lbmhd.LBMHD_FP32)

    def run():
        with lbmhd.Lbmhd(p, one, zero, zero, zero, zero, device=True) as sim:
            sim.step(1)

    run()  # loads the kernels
    lbmhd.lbmhd_release_cached_memory()
    base = torch.cuda.mem_get_info()[0]
    run()
    assert base - torch.cuda.mem_get_info()[0] > 800 << 20  # two copies of 453 MB are kept
    t = threading.Thread(target=lbmhd.lbmhd_release_cached_memory)
    t.start()
    t.join()
    assert base - torch.cuda.mem_get_info()[0] <= 64 << 20
