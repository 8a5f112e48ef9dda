"""Self-checks of the step of unfiltered grids (Delta = 0): its bounded wait, and its index checks in the
bounds-checking build (clean on ragged and degenerate grids; skipped and reported when forced)."""
import os
import subprocess
import sys
import textwrap
import time

import numpy as np
import pytest

from paper_1705_09807_gb300 import lbmhd
from paper_1705_09807_gb300.inputs import kh_jet

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FORMS = [lbmhd.LBMHD_FP64, lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1705_09807_gb300 import build
    build.build()
    lbmhd.load_library()


@pytest.mark.parametrize("precision", FORMS)
def test_missing_row_copy_is_reported_and_the_run_continues(precision):
    """One block leaves out one staged-row copy: its wait runs out, the host gets LBMHD_ERR_TIMEOUT, and a
    restored state continues exactly."""
    p = lbmhd.lbmhd_params_srt(96, 96, 0.01, 0.01, 0.0, precision)
    fields = kh_jet(96, seed=6)
    with lbmhd.Lbmhd(p, *fields) as ref:
        ref.step(5)
        want = ref.populations()
    with lbmhd.Lbmhd(p, *fields) as sim:
        sim.step(4)
        state = sim.get_state()
        lbmhd.lbmhd_test_skip_row_copy(sim.h, True)
        t0 = time.perf_counter()
        sim.step(1)
        with pytest.raises(lbmhd.LbmhdError) as e:
            sim.moments()
        assert e.value.code == lbmhd.LBMHD_ERR_TIMEOUT
        assert time.perf_counter() - t0 > 1.5  # the wait limit, not an early exit
        lbmhd.lbmhd_test_skip_row_copy(sim.h, False)
        sim.set_state(state)
        sim.step(1)
        assert np.array_equal(sim.populations(), want)


def _checked(script, **env):
    from paper_1705_09807_gb300 import build
    code = f"ROOT = {ROOT!r}\nLIB = {build.build_checked()!r}\n" + textwrap.dedent(script)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, **env))
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    return r.stdout.splitlines()


HEAD = '''
    import sys
    import numpy as np
    sys.path.insert(0, ROOT)
    import oracle
    from paper_1705_09807_gb300 import lbmhd
    from paper_1705_09807_gb300.inputs import smooth_random_fields
    lbmhd.load_library(LIB)
    F = (lbmhd.LBMHD_FP64, lbmhd.LBMHD_FP32, lbmhd.LBMHD_FP16, lbmhd.LBMHD_FP16_REL)
'''


def test_bounds_checked_build_runs_clean():
    out = _checked(HEAD + '''
    worst = dict.fromkeys(F, 0.0)
    for nx, ny in [(3, 3), (33, 17), (129, 20), (257, 9), (300, 70), (130, 5), (128, 4), (256, 512)]:
        fields = smooth_random_fields(nx, ny, seed=nx + ny, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
        s, sm = oracle.srt_rates(0.01), oracle.rate_from_diffusivity(0.015)
        fo, go = oracle.step(*oracle.init(*fields), s, sm, 0.0, 34)
        ref = np.concatenate([fo, go.reshape(18, ny, nx)])
        for prec in F:
            with lbmhd.Lbmhd(lbmhd.make_params(nx, ny, s, sm, 0.0, prec, 0), *fields) as sim:
                sim.step(34)            # one captured graph of 32 steps + 2 launches
                sim.moments()           # synchronises: reports a failed check
                worst[prec] = max(worst[prec], float(np.max(np.abs(sim.populations() - ref))))
    print("CLEAN", *(worst[prec] for prec in F))
''')
    e64, e32, e16, e16r = (float(v) for v in [ln for ln in out if ln.startswith("CLEAN")][-1].split()[1:])
    # rounding order (binary64); the stored deviations' rounding at each of 34 steps (the others)
    assert e64 < 1e-13 and e32 < 3e-6 and e16 < 3e-4 and e16r < 3e-4, out


def test_forced_check_failures_are_skipped_and_reported():
    out = _checked(HEAD + '''
    fields = smooth_random_fields(129, 20, seed=9, amp_u=0.05, amp_b=0.04, amp_rho=0.02)
    for prec in F:
        with lbmhd.Lbmhd(lbmhd.make_params(129, 20, oracle.srt_rates(0.01), 1.5, 0.0, prec, 0), *fields) as sim:
            before = sim.populations()
            sim.step(2)                 # even: back on the buffer the state was set in
            code = 0
            try:
                sim.moments()
            except lbmhd.LbmhdError as ex:
                code = ex.code if "flags 0xd" in str(ex) else -1
            print("FORCED", code, bool(np.array_equal(sim.populations(), before)))
''', LBMHD_BOUNDS_FORCE="0xd")  # staged column, global store, copy
    assert [ln for ln in out if ln.startswith("FORCED")] == [f"FORCED {lbmhd.LBMHD_ERR_INVALID} True"] * 4, out
