"""A case of a batch whose state is not finite: the other cases go on bit for bit as beside
a finite one (the sums, the Givens steps and the ends of cycles are each system's
own), and a NaN stops its case with a status (an infinity makes its step 0)."""
import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]
MIXED = dict(precision=1, basis_fp32=1, ilu_fp16=1, warm_extrap=2)


@pytest.mark.parametrize("kw", [{}, dict(limiter=1, limit_char=1), MIXED, dict(MIXED, limiter=1), dict(MIXED, flux_lead=2),
                                dict(precision=1), dict(cls_global=1)])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_the_other_cases_go_on(kw, value):
    from paper_1802_00704_gb300 import build, gks
    build.build()
    cases = [I.advection_case(6, seed=2), I.advection_case(9, seed=3), I.advection_case(20, seed=4)]
    T = [c.w0.shape[1] for c in cases]
    m = gks.GksMesh.batch([c.mesh for c in cases], **kw)
    w0 = np.concatenate([c.w0 for c in cases], axis=1)
    ref = dev(w0)
    assert m.batch_run(ref, max_steps=3)["n_failed"] == 0
    for var in (0, 1, 3):
        bad = w0.copy()
        bad[var, T[0] + 5] = value
        w = dev(bad)
        m.reset_warm_start()
        r = m.batch_run(w, max_steps=3)
        assert r["status"][0] == r["status"][2] == 0
        if np.isnan(value):
            assert r["status"][1] != 0 and r["n_failed"] == 1
        good = np.r_[0:T[0], T[0] + T[1]:sum(T)]
        assert np.array_equal(host(w)[:, good], host(ref)[:, good])
