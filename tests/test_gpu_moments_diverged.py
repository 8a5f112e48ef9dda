"""Read-out of relative binary16 states that have diverged: an infinite population makes rho or B
infinite (not NaN, as sums that subtract infinities would), and the diagnostics see the same fields."""
import numpy as np
import pytest

from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import smooth_random_fields

pytestmark = pytest.mark.gpu
CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
# planes of a row: groups by c_y = 1, 0, -1 of f, g_x, g_y
PLANE = {}
for _k, _group in enumerate(((2, 5, 6), (0, 1, 3), (4, 7, 8))):
    for _c in range(3):
        for _j, _i in enumerate(_group):
            PLANE[9 * _c + _i] = 9 * _k + 3 * _c + _j


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("q,value", [(0, np.inf), (1, -np.inf), (6, np.inf), (9, np.inf), (16, -np.inf), (26, np.inf),
                                     (3, np.nan), (20, np.nan)])
def test_infinite_population(q, value):
    """Population q of the cell that stores it at (x, y) is pulled by the cell at (x + c_x, y + c_y);
    every other cell is untouched."""
    import torch
    nx, ny, x, y = 150, 9, 129, 4
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 2.0, lbmhd.LBMHD_FP16_REL)
    with lbmhd.Lbmhd(p, *smooth_random_fields(nx, ny, seed=2, amp_u=0.05, amp_b=0.04)) as sim:
        sim.step(3)
        before = np.stack(sim.moments())
        state = sim.get_state()
        rows = state.view(np.float16).reshape(ny, 29, -1)
        rows[y, PLANE[q], 32 + x] = value
        sim.set_state(state)
        pops = sim.populations()
        got = np.stack(sim.moments())
        dev = torch.empty((5, ny, nx), dtype=torch.float64, device="cuda")
        sim.moments_device(list(dev))
        with pytest.raises(lbmhd.LbmhdUnstable) as e:
            sim.diagnostics()
        diag = e.value.values
        ref = torch.empty(lbmhd.LBMHD_NDIAG + 1, dtype=torch.float64, device="cuda")
        lbmhd.lbmhd_diagnostics_fields_noalloc(list(dev), ref)
    cx, cy = x + CX[q % 9], y + CY[q % 9]
    assert np.isnan(pops[q, cy, cx]) if np.isnan(value) else pops[q, cy, cx] == value
    want = before.copy()
    if q < 9:
        want[0, cy, cx], want[1:3, cy, cx] = value, np.nan
    else:
        want[3 if q < 18 else 4, cy, cx] = value
    assert np.array_equal(got, want, equal_nan=True)
    assert np.array_equal(dev.cpu().numpy(), want, equal_nan=True)
    # sums and maxima over the same fields (sums that stay finite: another order of binary64 additions)
    ref = ref.cpu().numpy()[:lbmhd.LBMHD_NDIAG]
    assert np.array_equal(diag[7:], ref[7:], equal_nan=True)
    assert np.allclose(diag[:7], ref[:7], rtol=1e-12, atol=1e-12, equal_nan=True)
