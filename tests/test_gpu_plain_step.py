"""The step of unfiltered grids (Delta = 0), which needs no moments of other cells, against the
filtered form: with Delta = 1e-30 the gradient products vanish in rounding, so both must give the
same state -- on grids of one and several strips, ragged and degenerate, single steps and graphs,
SRT and unequal rates -- and against the oracle."""
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


@pytest.mark.parametrize("nx,ny,steps", [(3, 3, 5), (4, 130, 3), (127, 4, 2), (128, 64, 33), (129, 5, 1), (257, 3, 7),
                                         (300, 701, 6)])
@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("stencil", [0, 1])
def test_plain_step_equals_the_filtered_form(nx, ny, steps, precision, stencil):
    """Bitwise where both forms' gradients are written out as FMAs (binary64, binary16); binary32
    leaves the contractions to the compiler, so with the nine-point stencil each step may round
    differently by an ulp of the deviations (below 0.25: 2^-26), at most doubled by the relaxation."""
    f = smooth_random_fields(nx, ny, seed=7, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
    s = oracle.srt_rates(0.02)
    s[5:9] = 1.5, 1.5, 1.3, 1.4
    sm = oracle.rate_from_diffusivity(0.01)
    pops = []
    for delta in (0.0, 1e-30):
        with lbmhd.Lbmhd(lbmhd.make_params(nx, ny, s, sm, delta, precision, stencil), *f) as sim:
            sim.step(steps)
            pops.append(sim.populations())
    if precision == lbmhd.LBMHD_FP32:
        assert np.max(np.abs(pops[0] - pops[1])) <= 2 * steps * 2.0 ** -26
    else:
        assert np.array_equal(pops[0], pops[1])
    if precision == lbmhd.LBMHD_FP64:
        fo, go = oracle.step(*oracle.init(*f), s, sm, 0.0, steps)
        assert np.max(np.abs(pops[0] - np.concatenate([fo, go.reshape(18, ny, nx)]))) < 1e-13


@pytest.mark.parametrize("precision", FORMS)
def test_correction_planes_need_the_general_form(precision):
    """A handle with Delta = 0 steps with correction planes attached and without them again."""
    import torch
    if precision in (lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL):
        pytest.skip("correction planes need binary64 or binary32 storage")
    nx, ny = 150, 40
    f = smooth_random_fields(nx, ny, seed=3)
    corr = torch.zeros((4, ny, nx), dtype=torch.float32, device="cuda")
    p = lbmhd.lbmhd_params_srt(nx, ny, 0.01, 0.01, 0.0, precision)
    with lbmhd.Lbmhd(p, *f) as a, lbmhd.Lbmhd(p, *f) as b:
        lbmhd.lbmhd_set_correction_device(a.h, corr)
        a.step(3)
        lbmhd.lbmhd_set_correction_device(a.h, None)
        a.step(2)
        b.step(5)
        assert np.max(np.abs(a.populations() - b.populations())) <= (1e-15 if precision == lbmhd.LBMHD_FP64 else 2e-7)
