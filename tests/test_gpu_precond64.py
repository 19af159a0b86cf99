"""One application of the FP64 sweeps against their CPU statement, for 0 to 3 sweeps each
way (every rotation of the row buffers): a cycle of one iteration gives x = a M^-1 b
with a = <b, K M^-1 b> / |K M^-1 b|^2, so a stale or aliased buffer shows directly
instead of costing iterations.

Tolerance: a row is at most 25 + 3 * 10 products per sweep on either side, six sweeps
and the pivot: 400 roundings of terms that the factors amplify by their condition
(below 20 on these cells), 8,000 * 2^-53 = 1e-12."""
import numpy as np
import pytest

from tests.cls_statement import Statement, stretched_case
from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("n,aspect", [(4, 1), (13, 3)])
def test_one_application(n, aspect):
    from paper_1802_00704_gb300 import build, gks
    build.build()
    c = stretched_case(n, aspect)
    s, w = Statement(c), dev(c.w0)
    for fwd in range(4):
        for bwd in range(4):
            m = gks.GksMesh(c.mesh, ilu_sweeps=fwd, ilu_sweeps_bwd=bwd, gmres_m=1, gmres_maxit=1)
            coef, info = m.cls_reconstruct(w, check=False)
            assert info["iters"] == [1] * 4
            got = host(coef)
            for v in range(4):
                z = s.precond(s.b[v], fwd, bwd)
                kz = s.K @ z
                ref = s.coefficients((s.b[v] @ kz) / (kz @ kz) * z)
                assert np.max(np.abs(got[v] - ref)) <= 1e-12 * np.max(np.abs(ref)), (fwd, bwd, v)
