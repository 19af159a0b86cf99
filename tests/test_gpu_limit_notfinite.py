"""The limiter beside a cell whose state is not finite: the flags are the oracle's (a
neighbour without a pressure leaves the cell its average only), and no coefficient is
touched otherwise."""
import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("charm", [0, 1])
@pytest.mark.parametrize("var", [0, 1, 3])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_flags_and_coefficients_beside_it(value, var, charm):
    from oracle import oracle as O
    from paper_1802_00704_gb300 import build, gks
    O.build()
    build.build()
    c = I.advection_case(12)
    w = c.w0.copy()
    w[var, 37] = value
    coef = 0.02 * np.random.default_rng(5).standard_normal((4, 5, c.w0.shape[1]))
    ref, rflag = O.OracleMesh(c.mesh, limiter=1, limit_char=charm).limit(w, coef)
    out, flags = gks.GksMesh(c.mesh, limiter=1, limit_char=charm).limit(dev(w), dev(coef))
    assert np.array_equal(host(flags), rflag)
    a, b = host(out).reshape(4, 5, -1), np.asarray(ref).reshape(4, 5, -1)
    assert np.all(np.isfinite(a))
    # the bound of the other limiter tests for characteristic variables
    assert np.max(np.abs(a - b)) <= 1.3e-9 * np.max(np.abs(b))
