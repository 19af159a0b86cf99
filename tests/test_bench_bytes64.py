"""The byte model of the FP64 solve of the per-cell equations, per cell and launch: what
its kernels read and write (gks_solve64.cuh), not what the generic ones do."""
import pytest

import bench

PIVOT = 160 + 200 + 160                       # r, P, z
SWEEP = 12 + 64 + 48 + 64 + 64                # indices, base, products of one triangle, in, out (rows 0 and 1)
LAST = 12 + 160 + 240 + 160                   # indices, z, products, x


def _bytes(cls, sweeps=2, bwd=-1, **prof):
    return bench.class_bytes(cls, prof, T=1, F=0, steps=1, sweeps=sweeps, exact=False, mixed=False, basis32=False,
                             sweeps_bwd=bwd, fuse_first=True, pairs=True, fused_dots=False, percell64=True)


@pytest.mark.parametrize("fwd,bwd,per_application", [
    (0, 0, PIVOT), (1, 0, PIVOT + LAST + 64), (0, 1, PIVOT + LAST + 64), (1, 2, PIVOT + 2 * SWEEP + LAST + 128),
    (2, -1, PIVOT + 3 * SWEEP + LAST + 128), (3, 0, PIVOT + 2 * SWEEP + LAST + 64)])
def test_sweeps(fwd, bwd, per_application):
    """The options that the FP64 sweeps ignore (folding, pairs) take no bytes off."""
    assert _bytes("ilu", fwd, bwd, arnoldi=0, arnoldi_jsum=0, precond=3) == 3 * per_application


def test_operator_and_gram_schmidt():
    work = dict(arnoldi=6, arnoldi_jsum=21, precond=6)
    # z, operator, y, and V_0 .. V_j; the update reads them again, w twice
    assert _bytes("spmv", **work) == 6 * (160 + 192 + 12 + 160) + 160 * 21
    assert _bytes("orth", **work) == 160 * (21 + 2 * 6)
