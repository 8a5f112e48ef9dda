"""Device memory kept from freed handles: runs in reused blocks equal runs in fresh ones (other
fields, other streams, several threads at once), no more than 1 GiB is kept, and it is given back."""
import threading

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


def _job(nx, ny, precision, seed, delta=2.0, stream=None):
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, delta, precision)
    p.cuda_stream = stream
    with lbmhd.Lbmhd(p, *smooth_random_fields(nx, ny, seed=seed, amp_u=0.05)) as sim:
        sim.step(35)
        out = [sim.populations(), sim.get_state(), sim.diagnostics(), np.stack(sim.moments())]
        if nx == ny:
            out += list(sim.spectrum(nx // 2))
    return out


JOBS = [(64, 64, lbmhd.LBMHD_FP64, 1), (130, 70, lbmhd.LBMHD_FP32, 2), (64, 64, lbmhd.LBMHD_FP64, 3),
        (96, 96, lbmhd.LBMHD_FP16, 4), (130, 70, lbmhd.LBMHD_FP32, 5), (64, 64, lbmhd.LBMHD_FP16_REL, 6)]


def _same(a, b):
    return len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))


def test_reused_blocks_streams_and_threads():
    import torch
    ref = []
    for j in JOBS:
        lbmhd.lbmhd_release_cached_memory()
        ref.append(_job(*j))
    for _ in range(2):
        for j, r in zip(JOBS, ref):
            assert _same(_job(*j), r)
    streams = [torch.cuda.Stream() for _ in range(2)]
    for k, (j, r) in enumerate(zip(JOBS, ref)):
        assert _same(_job(*j, stream=streams[k % 2].cuda_stream), r)
    bad = []

    def work(i):
        for j, r in list(zip(JOBS, ref))[i % 3:]:
            if not _same(_job(*j), r):
                bad.append((i, j))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_kept_memory_is_bounded_and_given_back():
    import torch
    lbmhd.lbmhd_release_cached_memory()
    free0 = torch.cuda.mem_get_info()[0]
    one = torch.ones((2048, 2048), dtype=torch.float64, device="cuda")
    zero = torch.zeros_like(one)
    torch.cuda.synchronize()
    base = torch.cuda.mem_get_info()[0]
    for precision in (lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP64, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP32):
        p = lbmhd.lbmhd_params_srt(2048, 2048, 0.02, 0.02, 0.0, precision)
        with lbmhd.Lbmhd(p, one, zero, zero, zero, zero, device=True) as sim:
            sim.step(2)
        assert base - torch.cuda.mem_get_info()[0] <= (1 << 30) + (64 << 20)
    assert base - torch.cuda.mem_get_info()[0] > 800 << 20  # the last run's two copies are kept
    lbmhd.lbmhd_release_cached_memory()
    assert abs(base - torch.cuda.mem_get_info()[0]) <= 64 << 20
    assert free0 >= base
