"""The second Gram-Schmidt pass of the FP64 solve, in a block per system (up to 1,000
triangles, one to four cell blocks) and in launches of its own (1, 2, 4 and 8 cells per
thread), on systems whose CPU statement needs it."""
import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.cls_statement import Statement, stretched_case
from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("n,aspect", [(3, 1), (5, 10), (5, 50), (11, 1), (16, 1), (16, 10), (22, 3), (36, 3)])
def test_reconstruction_with_second_passes(n, aspect):
    """Coefficients within 1e-9 of the oracle's (the bound of the other reconstruction
    tests), and the statement's iterations up to one at the stopping test."""
    from oracle import oracle as O
    from paper_1802_00704_gb300 import build, gks
    build.build()
    c = stretched_case(n, aspect)
    want = [Statement(c).gmres(v, 2, 2, 1e-12, 30, 500) for v in range(4)]
    assert all(second > 0 for _, second in want)
    ref, _, _, bad = O.OracleMesh(c.mesh).cls_solve(c.w0)
    assert not bad
    coef, info = gks.GksMesh(c.mesh).cls_reconstruct(dev(c.w0))
    assert max(info["relres"]) <= 1e-12
    assert all(abs(a - b) <= 1 for a, (b, _) in zip(info["iters"], want))
    assert np.max(np.abs(host(coef) - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("big", [142, 202, 284])
def test_launches_with_several_cells_per_thread(big):
    """Small cases that need the pass, beside a mesh that makes the batch's threads take
    2, 4 and 8 cells each: the same step as on their own (1e-13, as the batch tests)."""
    from paper_1802_00704_gb300 import build, gks
    build.build()
    cases = [stretched_case(3, 1), I.advection_case(big), stretched_case(16, 1), stretched_case(11, 1)]
    t_end = np.array([0.01, 1e-4, 0.01, 0.01])
    w = dev(np.concatenate([c.w0 for c in cases], axis=1))
    gks.GksMesh.batch([c.mesh for c in cases]).batch_run(w, t_final=t_end, max_steps=2)
    got, o = host(w), 0
    for q, c in enumerate(cases):
        T = c.w0.shape[1]
        if q != 1:
            ws = dev(c.w0)
            gks.GksMesh(c.mesh).run(ws, t_final=float(t_end[q]), max_steps=2)
            assert np.max(np.abs(got[:, o:o + T] - host(ws))) <= 1e-13 * np.max(np.abs(host(ws)))
        o += T
