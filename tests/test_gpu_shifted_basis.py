"""The FP64 solve's Krylov basis grows by K M^-1 V_j - V_j with one Gram-Schmidt
pass, and a second one where less than half of the norm is orthogonal to the basis.

On the 3 x 3 and 4 x 4 quad meshes with two sweeps each way the orthogonal part
drops below half in the middle of a cycle (0.43 and 0.40 at Arnoldi indices 4 and
3, where eight and nine are run), so both branches run in one cycle; with no sweeps (block
Jacobi) and 30 x 30 quads it stays above.  A restart length of 5 ends cycles at both
kinds of index.  The reconstruction is compared with the oracle's at the bound of
the repository's FP64 reconstruction tests (1e-9), and the reported residuals
with the tolerance of the solve."""
import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("n", [3, 4, 30])
@pytest.mark.parametrize("sweeps", [0, 2])
@pytest.mark.parametrize("gmres_m", [5, 30])
def test_reconstruction_matches_oracle(n, sweeps, gmres_m):
    from oracle import oracle as O
    from paper_1802_00704_gb300 import build, gks
    O.build()
    build.build()
    c = I.advection_case(n)
    ref, _, _, bad = O.OracleMesh(c.mesh).cls_solve(c.w0)
    assert not bad
    gm = gks.GksMesh(c.mesh, ilu_sweeps=sweeps, gmres_m=gmres_m, gmres_maxit=200)
    coef, info = gm.cls_reconstruct(dev(c.w0))
    assert max(info["relres"]) <= 1e-12
    assert np.max(np.abs(host(coef) - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [3, 4, 12])
@pytest.mark.parametrize("inner_rtol,gmres_m", [(1e-3, 8), (1e-7, 8), (1e-7, 3), (1e-7, 30)])
def test_mixed_reconstruction_matches_oracle(n, inner_rtol, gmres_m):
    """The mixed solve ends each Arnoldi index in the update's launch, with the new
    vector's norm from the projections: cycles that end early, at the restart
    length, and beyond the indices that are unrolled (1e-7 takes five or six)."""
    from oracle import oracle as O
    from paper_1802_00704_gb300 import build, gks
    O.build()
    build.build()
    c = I.advection_case(n)
    ref, _, _, bad = O.OracleMesh(c.mesh).cls_solve(c.w0)
    assert not bad
    gm = gks.GksMesh(c.mesh, precision=gks.MIXED, basis_fp32=1, inner_rtol=inner_rtol, gmres_m=gmres_m, gmres_maxit=200)
    coef, info = gm.cls_reconstruct(dev(c.w0))
    assert max(info["relres"]) <= 1e-12
    assert np.max(np.abs(host(coef) - ref)) <= 1e-9 * np.max(np.abs(ref))


def test_second_pass_on_either_side_of_its_size_rule():
    """The 3 x 3 mesh needs the second pass (above); alone it runs inside the last
    kernel of the index, in a batch with 16,200 triangles in launches of its own.
    Both give the same step (1e-13, as the batch tests: sums over other blocks)."""
    from paper_1802_00704_gb300 import build, gks
    build.build()
    cases = [I.advection_case(3), I.advection_case(90), I.advection_case(4)]
    t_end = np.array([0.01, 0.002, 0.01])
    w = dev(np.concatenate([c.w0 for c in cases], axis=1))
    gks.GksMesh.batch([c.mesh for c in cases]).batch_run(w, t_final=t_end, max_steps=2)
    got, o = host(w), 0
    for q, c in enumerate(cases):
        ws = dev(c.w0)
        gks.GksMesh(c.mesh).run(ws, t_final=float(t_end[q]), max_steps=2)
        T = c.w0.shape[1]
        assert np.max(np.abs(got[:, o:o + T] - host(ws))) <= 1e-13 * np.max(np.abs(host(ws)))
        o += T
