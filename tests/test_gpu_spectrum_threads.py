"""Energy spectra of different sizes from several host threads at once: each thread's results are the
ones it gets alone.  The sizes need different amounts of shared memory per block (more than the 48 KB
that a kernel may use without asking), so a limit set for one size must not hinder another's launch."""
import threading

import pytest

from paper_1705_09807_gb300 import lbmhd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


# 1025 and 2039: Bluestein over 4096 points (72 and 80 KB per block), 4093: over 8192 points (160 KB);
# 2500: mixed radices (60 KB).  Enough calls to fill the launch queue: a thread then waits for a slot
# between preparing a launch and making it.
@pytest.mark.parametrize("sizes,calls", [((1025, 2500), 600), ((2039, 4093), 40)])
def test_spectra_of_two_sizes_in_two_threads(sizes, calls):
    import torch
    data = []
    for n in sizes:
        gen = torch.Generator(device="cuda").manual_seed(n)
        f = torch.randn((4, n, n), generator=gen, device="cuda", dtype=torch.float64)
        work = torch.empty(lbmhd.lbmhd_energy_spectrum_work_bytes(n), dtype=torch.uint8, device="cuda")
        data.append((f, work, torch.empty((calls + 1, 2, n // 2), dtype=torch.float64, device="cuda")))
        lbmhd.lbmhd_energy_spectrum_device(*f, n // 2, *data[-1][2][calls], work)
    torch.cuda.synchronize()
    start = threading.Barrier(len(sizes))
    failed = []

    def spectra(n, f, work, out):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            for k in range(calls):
                lbmhd.lbmhd_energy_spectrum_device(*f, n // 2, *out[k], work, stream=stream.cuda_stream)
        except lbmhd.LbmhdError as e:
            failed.append((n, str(e)))
        stream.synchronize()

    threads = [threading.Thread(target=spectra, args=(n, *d)) for n, d in zip(sizes, data)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for _, _, out in data:
        assert torch.equal(out[:calls], out[calls:].expand(calls, -1, -1))
