"""Velocities of a coarse state inside and outside the range in which the features take them from a
reciprocal: densities near one and far from it, zero momentum."""
import numpy as np
import pytest

from oracle import closure as oc
from paper_1705_09807_gb300 import lbmhd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("rho", [1.0, 2.0 ** 250, 2.0 ** 300, 2.0 ** -300])
@pytest.mark.parametrize("u", [0.05, 0.0])
def test_velocity_features_of_a_uniform_state(rho, u):
    """u / scale with a rounding each of J, the quotient and the product, then one to binary32."""
    import torch
    n, r, m = 24, 2, 12
    scale = np.full(12, 0.05, np.float32)
    fine = torch.zeros((5, n, n), dtype=torch.float64, device="cuda")
    fine[0], fine[1], fine[2] = rho, u, -u
    x = torch.full((12, m, m), 5.0, dtype=torch.float32, device="cuda")
    t = torch.empty((4, m, m), dtype=torch.float32, device="cuda")
    work = torch.empty((9, m, m), dtype=torch.float64, device="cuda")
    with lbmhd.Closure(np.zeros(oc.num_params(), np.float32), scale, np.ones(4, np.float32)) as cl:
        cl.training_pair(fine, r, 2.0, x, t, work)
    got = x.cpu().numpy()
    want = u / float(scale[0])
    np.testing.assert_allclose(got[0], want, rtol=2.0 ** -23)
    np.testing.assert_allclose(got[1], -want, rtol=2.0 ** -23)
    assert np.all(got[2:] == 0.0)
