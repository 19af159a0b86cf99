"""A handle holds one layout of each array that its solve reads: bytes per cell of the
options that choose between layouts, from the handle's own count (gks_mesh_get_stats).

FP64, per-cell equations: the sweeps read P O (30 doubles), the triangular solves alpha,
dx, dy as uploaded (9) and a flag (4 bytes, the sync-free ones), block Jacobi neither.
Mixed: the operator is six groups of four floats where the products are fused into it,
else 15 + 9 floats; the factors 34 values, packed for the sweeps, as uploaded for the
triangular solves (with 9 floats of off-diagonal blocks that the unfused operator shares),
25 for block Jacobi."""
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]
EXACT, SWEEP, BJACOBI, LEVELS = 0, 1, 2, 3
FUSED = dict(precision=1, basis_fp32=1)


@pytest.mark.parametrize("a,b,per_cell", [
    (dict(precond=SWEEP), dict(precond=BJACOBI), 240), (dict(precond=EXACT), dict(precond=BJACOBI), 72 + 4),
    (dict(precond=LEVELS), dict(precond=BJACOBI), 72),
    (dict(FUSED, spmv_dots=1), dict(FUSED, spmv_dots=0), 0),
    (FUSED, dict(FUSED, ilu_fp16=1), 68), (FUSED, dict(FUSED, precond=LEVELS), 0), (FUSED, dict(FUSED, precond=EXACT), -4),
    (FUSED, dict(FUSED, precond=BJACOBI), 36), (dict(FUSED, ilu_fp16=1), dict(FUSED, ilu_fp16=1, precond=LEVELS), 0),
    (dict(FUSED, ilu_fp16=1), dict(FUSED, ilu_fp16=1, precond=BJACOBI), 18),
    (dict(precision=1, ilu_fp16=1), dict(precision=1, ilu_fp16=1, precond=LEVELS), 0),
    (dict(precision=1), dict(precision=1, precond=LEVELS), 136 - 100)])
def test_bytes_per_cell(a, b, per_cell):
    from paper_1802_00704_gb300 import build, gks
    build.build()
    c = I.advection_case(16)
    size = []
    for kw in (a, b):
        m = gks.GksMesh(c.mesh, **kw)
        coef, info = m.cls_reconstruct(dev(c.w0))
        assert info["converged"] == 1
        size.append(m.stats()["device_bytes"])
    assert size[0] - size[1] == per_cell * c.mesh.n_tri
