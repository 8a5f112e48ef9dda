"""Members of three columns in a binary16 ensemble, beside others: bit for bit the same fields repeated to
six columns, also in device memory that other runs have used before."""
import numpy as np
import pytest

import oracle
from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import smooth_random_fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("persistent", [False, True])
def test_three_columns_in_an_ensemble(stencil, persistent):
    def members(seed):
        f = smooth_random_fields(3, 9, seed=seed, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
        sets = [f, [np.tile(a, (1, 2)) for a in f], smooth_random_fields(140, 9, seed=seed)]
        return [(lbmhd.make_params(s[0].shape[1], 9, oracle.srt_rates(0.02), 1.4, 2.0, lbmhd.LBMHD_FP16, stencil), s)
                for s in sets]

    for seed in (41, 42, 43):  # the last run's result counts; the others leave their values behind
        with lbmhd.Ensemble(members(seed)) as ens:
            ens.set_schedule(4, persistent)
            ens.step(6)
            ens.sync()
            narrow, wide = ens.populations(0), ens.populations(1)
        assert np.array_equal(np.tile(narrow, (1, 1, 2)), wide)
