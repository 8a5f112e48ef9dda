"""Box filter where its scaling and its loads change form: powers of two (scaled by the exponent)
and others, odd and even widths, sums that are zero, tiny, huge or not numbers."""
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


@pytest.mark.parametrize("mx,my,r", [(9, 5, 1), (130, 4, 2), (5, 3, 3), (7, 6, 4), (3, 2, 6), (129, 2, 8), (2, 3, 16)])
def test_means_in_order(mx, my, r):
    """Sums row by row from the left and one product, as the sequential binary64 sum gives them: equal."""
    import torch
    rng = np.random.default_rng(r)
    f = rng.normal(size=(my * r, mx * r))
    specials = [0.0, -0.0, 5e-324, 2.0 ** -1022, 1e-310, 1.7e308, np.inf, -np.inf, np.nan, 2.0 ** -1018]
    for k, v in enumerate(specials[:mx * my // 2]):
        j, i = divmod(2 * k, mx)
        f[j * r:(j + 1) * r, i * r:(i + 1) * r] = v
    out = torch.zeros((my, mx), dtype=torch.float64, device="cuda")
    lbmhd.lbmhd_block_mean_device(torch.tensor(f, device="cuda"), r, out)
    want = np.zeros((my, mx))
    with np.errstate(all="ignore"):
        for yy in range(r):
            for xx in range(r):
                want += f[yy::r, xx::r]
        want *= 1.0 / (float(r) * r)
    np.testing.assert_array_equal(out.cpu().numpy(), want)
