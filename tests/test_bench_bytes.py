"""The byte model of the solves of the per-cell equations, per cell and launch: what their
kernels read and write (gks_solve64.cuh, gks_solve32.cuh), not what the generic ones
do.  The reads are those that ncu counts at 399,424 (FP64) and 1,000,000 triangles
(mixed): pivot 360, last launch 540; first forward sweep 140, second 192, backward
pair 160 bytes per cell."""
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


def _mixed(sweeps=2, bwd=-1, fuse=True, pairs=True, basis32=True, ilu16=True):
    return bench.class_bytes("ilu", dict(arnoldi=0, arnoldi_jsum=0, precond=1), T=1, F=0, steps=1, sweeps=sweeps,
                             exact=False, mixed=True, basis32=basis32, ilu16=ilu16, sweeps_bwd=bwd, fuse_first=fuse,
                             pairs=pairs, packed32=True)


def test_mixed_sweeps():
    """Reads and writes of each launch with FP16 factors: r 80, factors 2 per value, indices
    12, neighbours' rows 32; rows 0 and 1 32, all rows 80."""
    first, second, pair = 80 + 48 + 12 + 32, 80 + 32 + 68 + 12 + 80, 80 + 68 + 12 + 80
    assert _mixed() == first + second + pair
    assert _mixed(pairs=False) == first + second + (32 + 48 + 12 + 32) + (pair + 32)
    assert _mixed(1, 2) == (first + 20 + 48) + pair                 # the first sweep is the last: all rows
    assert _mixed(0, 0) == 80 + 68 + 80                             # z = P r
    assert _mixed(1, 0, fuse=False) == (80 + 32 + 32) + second
    assert _mixed(2, 2, basis32=False) == _mixed() + 80 + 80        # the FP64 source, and its rounded copy
    assert _mixed(ilu16=False) == _mixed() + 2 * (24 + 34 + 34)
