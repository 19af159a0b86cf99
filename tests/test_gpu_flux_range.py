"""The FP64 flux of a cell at the end of the number range: an internal energy of which
four times overflows is refused as non-physical, with a zero flux through the cell's
faces, and one just below that is not."""
import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, host, needs_gpu, torch

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("kw", [{}, dict(precision=1, basis_fp32=1, flux_lead=2)])
@pytest.mark.parametrize("energy,refused", [(2.0 ** 1021, False), (2.0 ** 1022, True), (1e308, True), (np.inf, True)])
def test_energy_at_the_end_of_the_range(kw, energy, refused):
    from paper_1802_00704_gb300 import build, gks
    build.build()
    c = I.advection_case(4)
    w0 = np.zeros_like(c.w0)
    w0[0], w0[3] = 1.0, 2.5
    w0[3, 7] = energy
    m = gks.GksMesh(c.mesh, **kw)
    coef = torch.zeros((4, 5, m.T), dtype=torch.float64, device="cuda")
    f, st = m.flux(dev(w0), coef, 1e-4, check=False)
    f = host(f)
    cells = c.mesh.faces[:, 2:4]
    mine = np.any(cells == 7, axis=1)
    assert mine.sum() == 3 and np.all(np.isfinite(f[:, ~mine]))
    assert (st == gks.GKS_ENONPHYS) == refused
    if refused:
        assert np.all(f[:, mine] == 0.0)
