"""Grids of three columns, whose middle column is a periodic neighbour on both sides, in every storage
form: the same fields repeated to six columns give the same state, bit for bit (every cell's
arithmetic is the same), also in device memory that other runs have used before."""
import numpy as np
import pytest

import oracle
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


def _run(fields, precision, delta, stencil, steps):
    ny, nx = fields[0].shape
    p = lbmhd.make_params(nx, ny, oracle.srt_rates(0.02), 1.4, delta, precision, stencil)
    with lbmhd.Lbmhd(p, *fields) as sim:
        sim.step(steps)
        return sim.populations()


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("ny,delta", [(3, 2.0), (7, 2.0), (40, 2.0), (7, 0.0)])
def test_three_columns_equal_their_repetition(precision, stencil, ny, delta):
    fields = smooth_random_fields(3, ny, seed=5, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
    # other runs leave their values in blocks of the same size
    for seed in (31, 32, 33):
        _run(smooth_random_fields(3, ny, seed=seed, amp_u=0.08, amp_b=0.08), precision, delta, stencil, 4)
    got = _run(fields, precision, delta, stencil, 6)
    want = _run([np.tile(f, (1, 2)) for f in fields], precision, delta, stencil, 6)
    assert np.array_equal(np.tile(got, (1, 1, 2)), want)
