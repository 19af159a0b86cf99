"""Handles used from two threads at once, each on a stream of its own."""
import copy
import threading

import numpy as np
import pytest

from paper_1802_00704_gb300 import inputs as I
from tests.gpu_util import dev, host, needs_gpu, torch

pytestmark = [pytest.mark.gpu, needs_gpu]


def test_restart_lengths_above_45_in_two_threads():
    """FP64 restart lengths of 64 and 46 each need more than 48 KiB of shared memory
    in the kernels that sum over the basis; a solve with the longer one is the same,
    bit for bit, while another thread starts solves with the shorter one.  (Stretched
    cells and block Jacobi: all 128 iterations run, two full restarts.)"""
    from paper_1802_00704_gb300 import build, gks
    build.build()
    c = I.advection_case(20, seed=7)
    mesh = copy.deepcopy(c.mesh)
    mesh.nodes, mesh.face_shift = mesh.nodes * [1.0, 0.02], mesh.face_shift * [1.0, 0.02]
    w = dev(c.w0)
    kw = dict(no_graphs=1, precond=gks.PC_BJACOBI)
    long = gks.GksMesh(mesh, gmres_m=64, gmres_maxit=128, **kw)
    short = gks.GksMesh(mesh, gmres_m=46, gmres_maxit=2, **kw)
    coef, info = long.cls_reconstruct(w, check=False)
    assert info["iters"] == [128] * 4 and info["status"] == gks.GKS_ENOCONV
    ref = host(coef)
    stop = threading.Event()
    other = []

    def solves():
        s = torch.cuda.Stream()
        while not stop.is_set():
            other.append(short.cls_reconstruct(w, stream=s, check=False)[1]["status"])

    t = threading.Thread(target=solves)
    t.start()
    try:
        for _ in range(10):
            long.reset_warm_start()
            coef, info = long.cls_reconstruct(w, check=False)
            assert info["status"] == gks.GKS_ENOCONV, gks.last_error()
            assert np.array_equal(host(coef), ref)
    finally:
        stop.set()
        t.join()
    assert other and set(other) <= {gks.GKS_OK, gks.GKS_ENOCONV}
