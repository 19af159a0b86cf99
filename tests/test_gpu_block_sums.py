"""The mixed solve's sums over a block's warps are FP64 sums: the block sums compiled on
their own, on values whose sums within a warp are exact, so that each result is a
sum of FP32 numbers in FP64.

Tolerance: eight numbers are seven additions, 256 / 4 = 64 numbers 63, each within
half a unit in the last place of a partial sum, none of which exceeds sum |x|."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

from tests.gpu_util import host, needs_gpu, torch

pytestmark = [pytest.mark.gpu, needs_gpu]

HEAD = """
#include "gks_solve32.cuh"
using namespace gks;
"""
ROWS = HEAD + """
__global__ void kernel(const float *x, double *part)
{
    __shared__ float sh[8][NSUM][4];
    float sv[NSUM][4];
    for (int k = 0; k < NSUM; ++k)
        for (int v = 0; v < 4; ++v) sv[k][v] = x[((blockIdx.x * NSUM + k) * 4 + v) * 256 + threadIdx.x];
    block_rows32<NSUM>(sv, sh, part, 0);
}
"""
QUADS = HEAD + """
__global__ void kernel(const float *x, double *part)
{
    __shared__ double sh[8][4];
    block_quads(double(x[blockIdx.x * 256 + threadIdx.x]), sh, part);
}
"""
TAIL = """
extern "C" __attribute__((visibility("default"))) int run(int blocks, const float *x, double *part)
{
    kernel<<<blocks, 256>>>(x, part);
    return cudaDeviceSynchronize();
}
"""


def _compiled(tmp, source, nsum=1):
    from paper_1802_00704_gb300 import build
    src, so = os.path.join(tmp, "sums.cu"), os.path.join(tmp, "sums.so")
    with open(src, "w") as f:
        f.write(f"#define NSUM {nsum}\n" + source + TAIL)
    subprocess.run([build._nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-I", build.CSRC, "-shared", "-o", so, src],
                   check=True, capture_output=True)
    return C.CDLL(so)


def _run(lib, x, n):
    xd = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
    part = torch.zeros((n, x.shape[0]), dtype=torch.float64, device="cuda")
    assert lib.run(x.shape[0], C.c_void_p(xd.data_ptr()), C.c_void_p(part.data_ptr())) == 0
    return host(part)


def _values(rng, shape):
    return (rng.uniform(0.5, 1.0, shape) * 2.0 ** rng.integers(-28, 1, shape)).astype(np.float32)


@pytest.mark.parametrize("k", [1, 2, 5])
def test_sums_across_warps(tmp_path, k):
    rng = np.random.default_rng(k)
    blocks = 64
    x = np.zeros((blocks, k, 4, 8, 32), dtype=np.float32)
    one = _values(rng, (blocks, k, 4, 8))
    one[0, :, :, :] = 0.0
    one[0, :, :, :3] = [1.0, 2.0 ** -25, 2.0 ** -50]           # exact in FP64
    lane = rng.integers(0, 32, (blocks, k, 4, 8))
    np.put_along_axis(x, lane[..., None], one[..., None], axis=-1)
    got = _run(_compiled(str(tmp_path), ROWS, k), x.reshape(blocks, -1), 4 * k).reshape(k, 4, blocks)
    for b in range(blocks):
        for q in range(k):
            for v in range(4):
                ref = math.fsum(map(float, one[b, q, v]))
                assert abs(got[q, v, b] - ref) <= (7 * 2.0 ** -53 * ref if b else 0.0), (b, q, v)


def test_sums_of_a_residual(tmp_path):
    rng = np.random.default_rng(7)
    x = _values(rng, (64, 256))
    x[0] = 0.0
    x[0, 4 * np.arange(3)] = [1.0, 2.0 ** -25, 2.0 ** -50]     # variable 0, exact in FP64
    got = _run(_compiled(str(tmp_path), QUADS), x, 4)
    for b in range(64):
        for v in range(4):
            ref = math.fsum(map(float, x[b, v::4]))
            assert abs(got[v, b] - ref) <= (63 * 2.0 ** -53 * ref if b else 0.0), (b, v)
