"""The moments read-out of every storage form against binary64 sums of the same stored
populations: ragged and degenerate grids (one warp and four warps per block, ghost columns at both
edges), densities for which the binary16 sums are exact in binary32 and ones for which they are
not, and a state with non-finite cells."""
import numpy as np
import pytest

from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import smooth_random_fields

pytestmark = pytest.mark.gpu
CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1.0])
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1.0])


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("nx,ny", [(3, 3), (33, 5), (64, 64), (129, 7), (300, 257)])
@pytest.mark.parametrize("precision", [lbmhd.LBMHD_FP64, lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL])
@pytest.mark.parametrize("scale", [1.0, 3.0])
def test_moments_equal_the_sums_of_the_populations(nx, ny, precision, scale):
    """rho, B: binary64 sums of 9 values below 2 (and the weights' rounding in the widened
    populations), 2e-15; u of the reduced forms: binary32(J) x binary32(1 / binary32(rho)), where J
    and rho may each have rounded the other way (one ulp, 2^-23, each)."""
    f = list(smooth_random_fields(nx, ny, seed=nx + ny, amp_u=0.05, amp_b=0.3, amp_rho=0.05))
    f[0] = scale * f[0]
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 2.0, precision)
    with lbmhd.Lbmhd(p, *f) as sim:
        sim.step(3)
        pop, m = sim.populations(), sim.moments()
    rho = pop[:9].sum(0)
    u = [np.tensordot(c, pop[:9], 1) / rho for c in (CX, CY)]
    np.testing.assert_allclose(m[0], rho, rtol=0, atol=2e-15 * scale)
    for k in (0, 1):
        np.testing.assert_allclose(m[3 + k], pop[9 + 9 * k:18 + 9 * k].sum(0), rtol=0, atol=2e-15)
        if precision == lbmhd.LBMHD_FP64:
            np.testing.assert_allclose(m[1 + k], u[k], rtol=1e-15, atol=2e-15)
        else:
            want = (u[k] * rho).astype(np.float32) * (np.float32(1) / rho.astype(np.float32))
            np.testing.assert_allclose(m[1 + k], want.astype(np.float64), rtol=2 * 2.0 ** -23, atol=2e-15)


@pytest.mark.parametrize("precision", [lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL])
def test_non_finite_cells_stay_non_finite_and_local(precision):
    nx, ny = 40, 9
    f = [np.array(a) for a in smooth_random_fields(nx, ny, seed=1)]
    f[0][4, 7] = np.nan
    f[3][2, 30] = np.inf
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 2.0, precision)
    with lbmhd.Lbmhd(p, *f) as sim:
        m = sim.moments()
        with pytest.raises(lbmhd.LbmhdUnstable):
            sim.diagnostics()
    assert np.isnan(m[0][4, 7]) and not np.isfinite(m[3][2, 30])
    assert np.all(np.isfinite(m[0][6:])) and np.all(np.isfinite(m[3][5:]))
