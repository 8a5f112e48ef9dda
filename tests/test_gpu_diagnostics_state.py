"""Diagnostics formed straight from the populations against the reduction over moment fields, where
the tiling changes: one strip and many, ragged strips, tiles of one row and of several."""
import numpy as np
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


@pytest.mark.parametrize("precision", [lbmhd.LBMHD_FP64, lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL])
@pytest.mark.parametrize("nx,ny", [(3, 3), (127, 5), (128, 608), (129, 609), (300, 257), (1000, 1100)])
def test_state_matches_fields(precision, nx, ny):
    """The same moments enter: maxima (the same operations on them) are equal, sums agree to 1e-14 of
    the sum of magnitudes (two orders of the same terms)."""
    import torch
    rng = np.random.default_rng(nx * 31 + ny)
    f = rng.normal(size=(5, ny, nx)) * np.array([0.01, 0.02, 0.02, 0.03, 0.03])[:, None, None]
    f[1:3] = np.clip(f[1:3], -0.1, 0.1)
    f[0] += 1.0
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 2.0, precision)
    with lbmhd.Lbmhd(p, *f) as sim:
        got, m = sim.diagnostics(), sim.moments()
    dev = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in m]
    out = torch.zeros(lbmhd.LBMHD_NDIAG + 1, dtype=torch.float64, device="cuda")
    lbmhd.lbmhd_diagnostics_fields_noalloc(dev, out)
    want = out.cpu().numpy()
    rho, u, v, b, d = m
    mags = [np.abs(t).sum() for t in (rho, rho * u, rho * v, b, d, 0.5 * rho * (u * u + v * v), 0.5 * (b * b + d * d))]
    assert want[-1] == 0.0
    assert np.all(np.abs(got[:7] - want[:7]) <= 1e-14 * np.array(mags))
    np.testing.assert_array_equal(got[7:], want[7:-1])
