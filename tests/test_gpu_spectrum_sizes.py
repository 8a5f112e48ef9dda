"""Shell spectra at the sizes where the transform changes form: every radix on its own and
mixed, chirp lengths (a prime factor above 13) just below and above a power of two, several lines
per block with a ragged last block, the largest sides, and shell counts from one to n."""
import numpy as np
import pytest

from oracle import spectrum as osp
from paper_1705_09807_gb300 import lbmhd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("n,nbins", [(3, 3), (4, 1), (5, 5), (7, 4), (8, 8), (9, 5), (11, 11), (13, 7), (22, 12),
                                     (26, 26), (30, 16), (32, 32), (33, 17), (34, 34), (64, 9), (97, 97),
                                     (125, 63), (127, 64), (128, 128), (129, 65), (143, 72), (210, 106), (257, 129),
                                     (510, 256), (512, 257), (693, 60), (1021, 511), (1024, 1024), (1025, 3),
                                     (2053, 1027), (4096, 2049)])
def test_spectrum_of_every_transform_form(n, nbins):
    """Noise of unit variance: every shell carries energy, so the binary64 transforms must agree to
    rounding (1e-11 relative: about 1e3 times the rounding of a 4096-point line)."""
    import torch
    rng = np.random.default_rng(n)
    f = [rng.normal(size=(n, n)) for _ in range(4)]
    dev = [torch.tensor(a, device="cuda") for a in f]
    ek = torch.full((nbins,), -1.0, dtype=torch.float64, device="cuda")
    em = torch.full((nbins,), -1.0, dtype=torch.float64, device="cuda")
    size = lbmhd.lbmhd_energy_spectrum_work_bytes(n)
    work = torch.full((size + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    lbmhd.lbmhd_energy_spectrum_device(*dev, nbins, ek, em, work[:size])
    torch.cuda.synchronize()
    assert bool((work[size:] == 0x5A).all())  # nothing written past the caller's buffer
    rk, rm = osp.energy_spectrum(*f, nbins=nbins)
    np.testing.assert_allclose(ek.cpu().numpy(), rk, rtol=1e-11, atol=1e-20)
    np.testing.assert_allclose(em.cpu().numpy(), rm, rtol=1e-11, atol=1e-20)


@pytest.mark.parametrize("nx,ny,r,offset", [(6, 4, 2, 0), (258, 6, 2, 0), (258, 6, 2, 1), (9, 6, 3, 0), (600, 12, 6, 1),
                                            (129, 129, 1, 0), (130, 130, 130, 0), (256, 300, 4, 0)])
def test_block_mean_of_every_width_and_alignment(nx, ny, r, offset):
    """Even and odd widths, fields on 16-byte boundaries and 8 bytes off them; r^2 additions of
    values of order one in binary64."""
    import torch
    a = np.random.default_rng(nx + r).normal(size=(ny, nx))
    buf = torch.empty(nx * ny + offset, dtype=torch.float64, device="cuda")
    t = buf[offset:].view(ny, nx)
    t.copy_(torch.tensor(a))
    out = torch.full((ny // r + 1, nx // r), 9.0, dtype=torch.float64, device="cuda")
    lbmhd.lbmhd_block_mean_device(t, r, out[:ny // r])
    torch.cuda.synchronize()
    np.testing.assert_allclose(out[:-1].cpu().numpy(), a.reshape(ny // r, r, nx // r, r).mean((1, 3)), rtol=0, atol=1e-14)
    assert bool((out[-1] == 9.0).all())
