"""The FP64 solve with a thread per cell and variable, at the sizes where its
shapes change: meshes that do not fill a warp or a cell block, the cells per
thread (1, 2, 4, 8), the size up to which the block-diagonal pass is folded in,
restart lengths whose sums need more than 48 KiB of shared memory, and cases of
a batch that stop at different times."""
import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.fixture(scope="module")
def G():
    from paper_1802_00704_gb300 import build, gks
    build.build()
    return gks


@pytest.mark.parametrize("n,kw", [
    (3, {}), (4, dict(ilu_sweeps=1)), (5, dict(ilu_sweeps=3, ilu_sweeps_bwd=1)), (17, dict(ilu_sweeps_bwd=0)),
    (17, dict(ilu_sweeps=0)), (17, dict(ilu_sweeps=0, ilu_sweeps_bwd=3)), (23, dict(gmres_m=4)),
    (23, dict(gmres_m=64, ilu_sweeps=0, ilu_sweeps_bwd=0)), (90, {}), (143, {}), (202, {}), (285, {})])
def test_reconstruction_matches_the_oracle(G, n, kw):
    """Coefficients within 1e-9 of the oracle's (the tolerance of the other
    reconstruction tests: residuals of 1e-12 on both sides)."""
    from oracle import oracle
    c = I.advection_case(n, seed=5 + n)
    a, info = G.GksMesh(c.mesh, **kw).cls_reconstruct(dev(c.w0))
    assert max(info["relres"]) <= 1e-12
    b = oracle.OracleMesh(c.mesh).cls_solve(c.w0)[0]
    a, b = host(a), np.asarray(b).reshape(4, 5, -1)
    assert np.max(np.abs(a - b)) <= 1e-9 * np.max(np.abs(b))


@pytest.mark.parametrize("n", [23, 89, 90])
def test_folded_first_pass_is_bit_identical(G, n):
    """ilu_fuse_first on either side of the size where it stops to act."""
    c = I.advection_case(n, seed=3)
    w = dev(c.w0)
    a = host(G.GksMesh(c.mesh, ilu_fuse_first=1).cls_reconstruct(w)[0])
    b = host(G.GksMesh(c.mesh, ilu_fuse_first=0).cls_reconstruct(w)[0])
    assert np.array_equal(a, b)


def test_batch_cases_stop_on_their_own(G):
    """A batch whose cases converge at different iterations and end at different
    times: every case equals its own run (1e-13), also with one-variable systems
    (b = 0) beside full ones."""
    cases = [I.advection_case(6, seed=2), I.acoustic_pulse_case(9, seed=4), I.advection_case(20, k=3, seed=6)]
    t_end = np.array([0.0, 0.004, 0.002])
    b = G.GksMesh.batch([c.mesh for c in cases])
    w = dev(np.concatenate([c.w0 for c in cases], axis=1))
    info = b.batch_run(w, t_final=t_end, max_steps=4)
    got, o = host(w), 0
    for q, c in enumerate(cases):
        ws = dev(c.w0)
        r = G.GksMesh(c.mesh).run(ws, t_final=float(t_end[q]), max_steps=4)
        ref = host(ws)
        assert abs(info["t"][q] - r["t"]) <= 1e-13 * r["t"]
        assert np.max(np.abs(got[:, o:o + c.mesh.n_tri] - ref)) <= 1e-13 * np.max(np.abs(ref))
        o += c.mesh.n_tri
