"""Binary64 steps of a cell whose density is zero (a state that has diverged): 1/rho is infinite, so what
depends on the electric field becomes infinite with its sign and the rest stays finite, as by a division."""
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


@pytest.mark.parametrize("delta", [0.0, 2.0])
@pytest.mark.parametrize("sign", [-1.0, 1.0])
def test_step_of_a_cell_without_density(delta, sign):
    nx, ny, x, y = 150, 9, 60, 4
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, delta, lbmhd.LBMHD_FP64)
    with lbmhd.Lbmhd(p, *smooth_random_fields(nx, ny, seed=2, amp_u=0.02, amp_b=0.02)) as sim:
        state = sim.get_state()
        rows = state.view(np.float64).reshape(ny, 27, -1)
        # what the cell (x, y) pulls: rho - 1 = -1, J = (1, 1/2), B = (0, +-1/2)
        cell = np.zeros(27)
        cell[:5] = -1.0, 0.5, 0.25, -0.5, -0.25
        cell[18] = 0.5 * sign
        for q in range(27):
            rows[y - CY[q % 9], PLANE[q], 32 + x - CX[q % 9]] = cell[q]
        sim.set_state(state)
        sim.step(1)
        pops = sim.populations()
    got = np.array([pops[q, y + CY[q % 9], x + CX[q % 9]] for q in range(27)])
    # E = (J_x B_y - J_y B_x) / rho has the sign of B_y; g_x^eq = w (B_x - 3 c_y E), g_y^eq = w (B_y + 3 c_x E)
    for q, e in [(9 + i, -CY[i]) for i in range(9)] + [(18 + i, CX[i]) for i in range(9)]:
        if e == 0:
            assert np.isfinite(got[q]), (q, got)
        else:
            assert got[q] == e * sign * np.inf, (q, got)
    assert got[0] == -np.inf  # f_0: the trace of J J / rho
