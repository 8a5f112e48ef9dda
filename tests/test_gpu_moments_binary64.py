"""Velocity read-out of binary64 states where its quotient changes form: zero momentum, momenta
below and above the range in which the corrected product is used, densities far from one."""
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


@pytest.mark.parametrize("u0", [0.0, 0.05, -0.05, 1e-60, 1e-76, 1e-78, -1e-90, 1e-300])
@pytest.mark.parametrize("rho0", [1.0, 0.7, 3.0])
def test_velocity_of_a_uniform_state(u0, rho0):
    """Six populations of at most w_i rho0 |3 u0 + ...| each with a few roundings: 1e-14 of |u0|, and
    1e-16 of the density part that rho0 != 1 leaves in every population."""
    nx, ny = 40, 5
    one = np.ones((ny, nx))
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.02, 0.02, 2.0, lbmhd.LBMHD_FP64)
    with lbmhd.Lbmhd(p, rho0 * one, u0 * one, 0 * one, 0 * one, 0 * one) as sim:
        m = sim.moments()
    base = 0.0 if rho0 == 1.0 else 4e-16
    np.testing.assert_allclose(m[0], rho0, rtol=1e-15)
    np.testing.assert_allclose(m[1], u0, rtol=1e-14, atol=base)
    np.testing.assert_allclose(m[2], 0.0, atol=base + 1e-15 * abs(u0))


def test_values_that_are_not_numbers_stay_local():
    f = [np.ones((9, 40)), np.full((9, 40), 0.01)] + [np.zeros((9, 40)) for _ in range(3)]
    f[0][4, 7] = np.nan
    f[0][4, 20] = np.inf
    p = lbmhd.lbmhd_params_srt(40, 9, 0.02, 0.02, 2.0, lbmhd.LBMHD_FP64)
    with lbmhd.Lbmhd(p, *f) as sim:
        m = sim.moments()
    for x in (7, 20):
        assert not np.isfinite(m[0][4, x]) and not np.isfinite(m[1][4, x])
    keep = np.ones((9, 40), bool)
    keep[4, [7, 20]] = False
    np.testing.assert_allclose(m[1][keep], 0.01, rtol=1e-14)
