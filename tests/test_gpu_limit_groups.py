"""The limiter's two splits (a warp per flagged cell, or eight cells per warp above
two cells per SM sub-partition) against the oracle, with every cell flagged, so that
the number of cells on the list is the mesh's: at most 32 (one block's worth), the
last size of the first split on 152 SMs (1,216), the first of the second, and a
ragged larger one.

Tolerances.  The exponent S <= 20 of the weights d^-S (|ln d| < 6 here) leaves
20 * 6 * a few roundings in a weight, 600 eps; u_0 tan(a) turns an error e of its
argument into |u_0| (1 + t^2) e, t = tan(a) at most the largest |u_j / u_0|.
The candidates lie within a factor 10 here, so an error is at most 10 * 600 eps
= 1.3e-12 of the largest coefficient; in characteristic variables the own candidate
is a difference, t is taken as 1e4 (80,000 candidates): 1.3e-9.  Flags are equal."""
import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("charm", [0, 1])
@pytest.mark.parametrize("nx,ny", [(3, 3), (76, 8), (87, 7), (89, 23)])
def test_every_cell_flagged_matches_oracle(nx, ny, charm):
    from oracle import oracle as O
    from paper_1802_00704_gb300 import build, gks
    O.build()
    build.build()
    c = I.riemann_strip_case(nx, ny, left=(1.0, 0.3, 0.1, 1.0), right=(0.8, 0.2, 0.0, 0.9), seed=11, name="noise")
    T = c.w0.shape[1]
    assert T == 2 * nx * ny
    rng = np.random.default_rng(nx * 100 + ny)
    w = c.w0 * (1.0 + 0.05 * rng.standard_normal(c.w0.shape))
    size = rng.uniform(0.6, 1.0, (4, 5, T)) * np.array([0.2, 0.2, 0.02, 0.02, 0.02])[None, :, None] * (8.0 if T < 100 else 1.0)
    coef = size * rng.choice([-1.0, 1.0], (4, 5, T)) * np.abs(c.w0[[0, 0, 0, 3]]).max(axis=1)[:, None, None]
    om = O.OracleMesh(c.mesh, limiter=1, limit_char=charm)
    ref, rflag = om.limit(w, coef)
    assert np.all(rflag > 0)
    out, flags = gks.GksMesh(c.mesh, limiter=1, limit_char=charm).limit(dev(w), dev(coef))
    assert np.array_equal(host(flags), rflag)
    a, b = host(out).reshape(4, -1), np.asarray(ref).reshape(4, -1)
    err = np.max(np.abs(a - b), axis=1) / np.max(np.abs(b))
    assert np.all(err <= (1.3e-9 if charm else 1.3e-12)), err
