"""The diagnostics reduction where its tiling changes: one strip and many, rows that do not fill
a tile, sides of three cells, more tiles than partial records, non-finite and unstable cells."""
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


def _reference(f):
    rho, u, v, b, d = f
    sh = lambda a, dx, dy: np.roll(a, (-dy, -dx), (0, 1))  # noqa: E731
    dx = lambda a: (sh(a, 1, 0) - sh(a, -1, 0)) / 3 + (sh(a, 1, 1) - sh(a, -1, 1) + sh(a, 1, -1) - sh(a, -1, -1)) / 12  # noqa: E731
    dy = lambda a: (sh(a, 0, 1) - sh(a, 0, -1)) / 3 + (sh(a, 1, 1) - sh(a, 1, -1) + sh(a, -1, 1) - sh(a, -1, -1)) / 12  # noqa: E731
    terms = [rho, rho * u, rho * v, b, d, 0.5 * rho * (u * u + v * v), 0.5 * (b * b + d * d)]
    der = [dx(b), dy(b), dx(d), dy(d)]
    cen = 0.5 * (sh(b, 1, 0) - sh(b, -1, 0) + sh(d, 0, 1) - sh(d, 0, -1))
    peaks = [np.abs(der[0] + der[3]).max(), np.abs(cen).max(), max(np.abs(a).max() for a in der)]
    return [t.sum() for t in terms], [np.abs(t).sum() for t in terms], peaks


def _call(f):
    import torch
    out = torch.full((lbmhd.LBMHD_NDIAG + 1,), -1.0, dtype=torch.float64, device="cuda")
    dev = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in f]
    lbmhd.lbmhd_diagnostics_fields_noalloc(dev, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _fields(nx, ny):
    rng = np.random.default_rng(nx * 31 + ny)
    f = rng.normal(size=(5, ny, nx)) * np.array([0.01, 0.05, 0.05, 0.03, 0.03])[:, None, None]
    f[1:3] = np.clip(f[1:3], -0.25, 0.25)
    f[0] += 1.0
    return f


@pytest.mark.parametrize("nx,ny", [(3, 3), (127, 3), (128, 4), (129, 5), (3, 5000), (300, 257), (256001, 3),
                                   (1000, 1100)])
def test_reduction_of_every_tiling(nx, ny):
    """Sums to 1e-14 of the sum of magnitudes; derivatives of values below 0.2 to 5 roundings."""
    f = _fields(nx, ny)
    got = _call(f)
    sums, mags, peaks = _reference(f)
    assert np.all(np.abs(got[:7] - sums) <= 1e-14 * np.array(mags))
    assert np.all(np.abs(got[7:10] - peaks) <= 5 * 0.2 * 2.0 ** -53)
    assert got[10] == 0.0


@pytest.mark.parametrize("field,value,flag", [(0, 0.0, 1), (0, -1.0, 1), (0, np.nan, 1), (0, np.inf, 1), (1, 0.41, 1),
                                              (2, -0.41, 1), (1, np.nan, 1), (2, np.inf, 1), (3, np.nan, 1),
                                              (4, -np.inf, 1), (1, 1e200, 1), (3, 7.0, 0), (0, 5e-324, 0)])
def test_flag_of_one_cell(field, value, flag):
    f = _fields(200, 70)
    f[:, 69, 199] = (1.0, 0.0, 0.0, 0.0, 0.0)
    f[field, 69, 199] = value
    got = _call(f)
    assert got[10] == flag
    if np.isnan(value):  # maxima over the cells that are numbers, as without it
        assert np.all(np.isfinite(got[7:10]))
