"""What a handle reports after the autotuner when it keeps the inverse form: the work
of the factorisation is the inverse form's own, as before the autotuner (the block
Cholesky's task lists that it timed do not run and are not counted)."""
from dataclasses import replace

import numpy as np
import pytest

from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("waves", [1, 2])
def test_executed_flops_after_autotune(precision, waves):
    from paper_2211_13893_gb300 import MSGFEM, plan
    cfg = replace(get_config("t3"), NX=25, NY=7, NZ=8, sx=3, sy=2, overlap=2, oversampling=3, n_loc=9)
    wave_mb = 0.0 if waves == 1 else 1.01 * plan(cfg, precision)["pool_mb"] / waves
    m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, precision=precision, wave_mb=wave_mb)
    chol = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, precision=precision, wave_mb=wave_mb, factor_schedule=1)
    m.local_spaces(cfg.n_loc)
    chol.local_spaces(cfg.n_loc)
    before, block = m.profile(), chol.profile()
    assert before["waves"] >= waves and before["factor_flops"] != block["factor_flops"]
    m.autotune(reps=1)
    m.local_spaces(cfg.n_loc)
    after = m.profile()
    kept = after["factor_flops"] == before["factor_flops"]
    want = before["factor_flops_executed"] if kept else block["factor_flops_executed"]
    assert after["factor_flops_executed"] == pytest.approx(want, rel=0.0 if kept else 0.2)
    assert np.isfinite(after["factor_flops_executed"])
    m.close()
    chol.close()


@pytest.mark.parametrize("kw", [dict(), dict(precision=1), dict(solve_kernel=2)])
def test_tuning_names_the_form(kw):
    """msgfem_tuning.inverse_form is the form of the next local stage, with both forms'
    times; a handle set up by a Cholesky kernel measures the block Cholesky only."""
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), NX=25, NY=7, NZ=8, sx=3, sy=2, overlap=2, oversampling=3, n_loc=9)
    m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, **kw)
    m.local_spaces(cfg.n_loc)
    t = m.autotune(reps=1)
    m.local_spaces(cfg.n_loc)
    p = m.profile()
    # (only the inverse form counts no separate inverses of diagonal factors)
    assert t["inverse_form"] == (1 if p["factor_flops_inverse"] == p["factor_flops"] else 0)
    assert all((v > 0.0) == ("solve_kernel" not in kw) for v in t["inverse_ms"])
    if t["inverse_form"]:
        assert t["inverse_ms"][1] > 0.0 and t["inverse_ms"][0] > 0.0
    m.close()
