"""Diagnostics of narrow grids, whose tiles hold several pieces one below the other: against sums and
differences of the moment fields in numpy, at the widths and heights where the pieces, their rows or
the way from the state change, and with few idle lanes."""
import numpy as np
import pytest

from captured_launches import launches
from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import smooth_random_fields

pytestmark = pytest.mark.gpu
FORMS = [lbmhd.LBMHD_FP64, lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


def _shift(a, dx, dy):
    return np.roll(a, (-dy, -dx), (0, 1))


def _iso(a, axis):
    """3 w_i c_i a(x + c_i) summed over the eight neighbours."""
    out = np.zeros_like(a)
    for c in ((1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)):
        w = 1 / 3 if 0 in c else 1 / 12
        out += w * c[axis] * _shift(a, *c)
    return out


def _reference(m):
    rho, u, v, b, d = m
    g = [_iso(b, 0), _iso(b, 1), _iso(d, 0), _iso(d, 1)]
    central = 0.5 * (_shift(b, 1, 0) - _shift(b, -1, 0) + _shift(d, 0, 1) - _shift(d, 0, -1))
    return np.array([rho.sum(), (rho * u).sum(), (rho * v).sum(), b.sum(), d.sum(), 0.5 * (rho * (u * u + v * v)).sum(),
                     0.5 * (b * b + d * d).sum(), np.abs(g[0] + g[3]).max(), np.abs(central).max(),
                     max(np.abs(x).max() for x in g)])


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("nx,ny", [(3, 3), (3, 168), (3, 169), (4, 1216), (5, 1217), (42, 13), (43, 9), (63, 1217),
                                   (64, 17), (64, 1216), (64, 1217), (64, 8193), (65, 1217), (3, 172035)])
def test_narrow_grids(nx, ny, precision):
    """Sums: binary64 rounding of at most nx ny additions of terms below their scale, in any order,
    1e-13 of it; differences: a few roundings of values below 0.2."""
    import torch
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 2.0, precision)
    with lbmhd.Lbmhd(p, *smooth_random_fields(nx, ny, seed=ny, amp_u=0.05, amp_b=0.04, amp_rho=0.02)) as sim:
        sim.step(3)
        m = np.stack(sim.moments())
        got = sim.diagnostics()
    want = _reference(m)
    out = torch.empty(lbmhd.LBMHD_NDIAG + 1, dtype=torch.float64, device="cuda")
    lbmhd.lbmhd_diagnostics_fields_noalloc([torch.tensor(a, device="cuda") for a in m], out)
    out = out.cpu().numpy()
    assert out[-1] == 0.0
    scale = np.array([1, 0.2, 0.2, 0.2, 0.2, 0.02, 0.02]) * nx * ny * 1e-13
    for values in (got, out[:-1]):
        assert np.all(np.abs(values[:7] - want[:7]) <= scale)
        assert np.all(np.abs(values[7:] - want[7:]) <= 4e-16)
    assert np.array_equal(got[7:], out[7:-1])


@pytest.mark.parametrize("nx", [3, 5, 16, 33, 64])
def test_few_idle_lanes(nx):
    """At four rows a thread, at most half as many lanes again as that takes."""
    import torch
    ny = 1 << 12
    f = [torch.full((ny, nx), v, dtype=torch.float64, device="cuda") for v in (1.0, 0.0, 0.0, 0.0, 0.0)]
    out = torch.empty(lbmhd.LBMHD_NDIAG + 1, dtype=torch.float64, device="cuda")
    lbmhd.lbmhd_diagnostics_fields_noalloc(f, out)  # the first call looks its scratch up
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    first, last = launches(stream, lambda: lbmhd.lbmhd_diagnostics_fields_noalloc(f, out, stream=stream.cuda_stream))
    grid, block = max((first, last), key=lambda k: k[0][0])
    assert np.prod(grid) * np.prod(block) <= 1.5 * nx * ny / 4
