"""The mixed solve with packed FP32 vectors and factors, at the sizes where its
shapes change: meshes that do not fill a block, more Arnoldi indices than are
unrolled, FP16 and FP32 factors, FP64 and FP32 bases, every combination of
sweeps, and a batch whose cases stop at different iterations."""
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


@pytest.mark.parametrize("n", [3, 8, 23, 91])
@pytest.mark.parametrize("kw", [
    dict(basis_fp32=1), dict(basis_fp32=1, ilu_fp16=1), dict(), dict(ilu_fp16=1),
    dict(basis_fp32=1, ilu_sweeps=0), dict(basis_fp32=1, ilu_sweeps=0, ilu_sweeps_bwd=2),
    dict(basis_fp32=1, ilu_sweeps=1, ilu_sweeps_bwd=0), dict(basis_fp32=1, ilu_sweeps=3, ilu_sweeps_bwd=3),
    dict(ilu_sweeps=3, ilu_sweeps_bwd=4, ilu_fuse_first=0), dict(basis_fp32=1, inner_rtol=1e-7, ilu_sweeps=1),
    dict(basis_fp32=1, inner_rtol=1e-7, spmv_dots=0, ilu_sweeps=1), dict(basis_fp32=1, gmres_m=2)])
def test_reconstruction_matches_the_oracle(G, n, kw):
    """Coefficients within 1e-9 of the oracle's (the tolerance of the other
    reconstruction tests: FP64 residuals of 1e-12 on both sides)."""
    from oracle import oracle
    c = I.advection_case(n, seed=7 + n)
    a, info = G.GksMesh(c.mesh, precision=G.MIXED, **kw).cls_reconstruct(dev(c.w0))
    assert max(info["relres"]) <= 1e-12
    b = oracle.OracleMesh(c.mesh).cls_solve(c.w0)[0]
    assert np.max(np.abs(host(a) - b)) <= 1e-9 * np.max(np.abs(b))


@pytest.mark.parametrize("kw", [dict(basis_fp32=1), dict(basis_fp32=1, ilu_fp16=1, gmres_m=12), dict()])
def test_batch_cases_stop_on_their_own(G, kw):
    """A batch whose cases converge at different iterations and end at different
    times: every case equals its own run (1e-13, bit-equal arithmetic but for the
    blocks its sums are taken over), also with b = 0 systems beside full ones."""
    cases = [I.advection_case(6, seed=2), I.acoustic_pulse_case(9, seed=4), I.advection_case(20, k=3, seed=6)]
    t_end = np.array([0.0, 0.004, 0.002])
    kw = dict(precision=G.MIXED, warm_extrap=2, **kw)
    b = G.GksMesh.batch([c.mesh for c in cases], **kw)
    w = dev(np.concatenate([c.w0 for c in cases], axis=1))
    info = b.batch_run(w, t_final=t_end, max_steps=5)
    got, o = host(w), 0
    for q, c in enumerate(cases):
        ws = dev(c.w0)
        r = G.GksMesh(c.mesh, **kw).run(ws, t_final=float(t_end[q]), max_steps=5)
        ref = host(ws)
        assert abs(info["t"][q] - r["t"]) <= 1e-13 * r["t"]
        assert np.max(np.abs(got[:, o:o + c.mesh.n_tri] - ref)) <= 1e-13 * np.max(np.abs(ref))
        o += c.mesh.n_tri
