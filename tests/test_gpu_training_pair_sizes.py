"""Training pairs and features at the sizes where their kernels change form: filters of one cell,
of widths that do not divide a block, of exactly a block and wider than a block; coarse sides from
three cells, not multiples of the 32 x 4 tiles."""
import numpy as np
import pytest

from oracle import closure as oc
from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import smooth_random_fields

pytestmark = pytest.mark.gpu
IN_SCALE = np.array([0.05, 0.05, 0.03, 0.03] + [0.005] * 8, dtype=np.float32)
OUT_SCALE = np.array([1e-6, 2e-6, 3e-6, 4e-6], dtype=np.float32)


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("m,r", [(3, 1), (5, 3), (33, 2), (70, 7), (9, 64), (37, 20), (3, 128), (4, 130), (131, 1)])
def test_training_pair_and_features(m, r):
    """Features to two binary32 roundings.  Targets are differences of products below 0.02 (about
    50 roundings of 2e-18 each, 1e-16) over out_scale >= 1e-6: 1e-9 absolute, and one binary32
    rounding."""
    import torch
    n, delta = m * r, 2.0
    f = smooth_random_fields(n, n, seed=m + r, amp_u=0.05, amp_b=0.04, amp_rho=0.02, kmax=1)
    fine = torch.tensor(np.stack(f), device="cuda")
    pad = 100
    x = torch.full((12 * m * m + pad,), 5.0, dtype=torch.float32, device="cuda")
    t = torch.full((4 * m * m + pad,), 5.0, dtype=torch.float32, device="cuda")
    an = torch.full((4 * m * m + pad,), 5.0, dtype=torch.float32, device="cuda")
    work = torch.full((9 * m * m + pad,), 5.0, dtype=torch.float64, device="cuda")
    with lbmhd.Closure(np.zeros(oc.num_params(), np.float32), IN_SCALE, OUT_SCALE) as cl:
        cl.training_pair(fine, r, delta, x[:12 * m * m].view(12, m, m), t[:4 * m * m].view(4, m, m), work[:9 * m * m])
        xr, tr = oc.training_pair(*f, r, delta, IN_SCALE, OUT_SCALE)
        got_x, got_t = x[:-pad].cpu().numpy().reshape(12, m, m), t[:-pad].cpu().numpy().reshape(4, m, m)
        np.testing.assert_allclose(got_x, xr, rtol=2.0 ** -22, atol=1e-10)
        np.testing.assert_allclose(got_t, tr, rtol=2.0 ** -22, atol=1e-9)
        # the same coarse state through its velocities, with the analytic closure
        R, jx, jy, bx, by = (oc.box(a, r) for a in (f[0], f[0] * f[1], f[0] * f[2], f[3], f[4]))
        state = torch.tensor(np.stack([R, jx / R, jy / R, bx, by]), device="cuda")
        cl.features(state, delta, x[:12 * m * m].view(12, m, m), an[:4 * m * m].view(4, m, m))
        np.testing.assert_allclose(x[:-pad].cpu().numpy().reshape(12, m, m), xr, rtol=2.0 ** -22, atol=1e-10)
        ar = oc.analytic(R, jx, jy, bx, by, delta)
        np.testing.assert_allclose(an[:-pad].cpu().numpy().reshape(4, m, m), ar, rtol=2.0 ** -22, atol=1e-15)
    for a in (x, t, an, work):
        assert bool((a[-pad:] == 5.0).all())  # nothing written past the planes
