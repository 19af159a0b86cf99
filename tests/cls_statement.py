"""A plain CPU statement of the preconditioned CLS system, from the oracle's matrix: the
block ILU(0) factors on the RCM order, their application by sweeps, and the Arnoldi
process of the FP64 solve on it.  Cells are in RCM order (perm: RCM index -> cell)."""
import copy

import numpy as np
import scipy.sparse as sp

from paper_1802_00704_gb300 import inputs as I


def stretched_case(n, aspect, seed=7):
    """The advection case of n x n quads on cells flattened aspect : 1."""
    c = copy.deepcopy(I.advection_case(n, seed=seed))
    s = np.array([1.0, 1.0 / aspect])
    c.mesh.nodes, c.mesh.face_shift = c.mesh.nodes * s, c.mesh.face_shift * s
    return c


class Statement:
    def __init__(self, case):
        from oracle import oracle as O
        O.build()
        om = O.OracleMesh(case.mesh)
        rp, col, val, _ = om.cls_matrix()
        T = self.T = om.T
        assert om.ndof == 5 * T
        self.perm = om.rcm_perm()
        idx = (5 * self.perm[:, None] + np.arange(5)).ravel()
        self.K = sp.csr_matrix((val, col, rp), shape=(5 * T, 5 * T))[idx][:, idx].tocsr()
        self.b = om.cls_rhs(case.w0)[:, idx]
        B = self.K.tobsr((5, 5))
        blk = {(i, int(B.indices[q])): B.data[q] for i in range(T) for q in range(B.indptr[i], B.indptr[i + 1])}
        nb = [[int(j) for j in B.indices[B.indptr[i]:B.indptr[i + 1]]] for i in range(T)]
        self.P = np.zeros((T, 5, 5))
        for i in range(T):
            d = blk[i, i].copy()
            for j in nb[i]:
                if j < i:
                    d -= blk[i, j] @ self.P[j] @ blk[j, i]
            self.P[i] = np.linalg.inv(d)

        def part(keep):
            rows = [[j for j in nb[i] if keep(i, j)] for i in range(T)]
            data = np.array([blk[i, j] for i in range(T) for j in rows[i]]).reshape(-1, 5, 5)
            ptr = np.cumsum([0] + [len(r) for r in rows])
            return sp.bsr_matrix((data, np.array([j for r in rows for j in r], dtype=int), ptr), shape=(5 * T, 5 * T))
        self.L, self.U = part(lambda i, j: j < i), part(lambda i, j: j > i)

    def pivot(self, y):
        return np.einsum("iab,ib->ia", self.P, y.reshape(self.T, 5)).ravel()

    def precond(self, r, fwd, bwd):
        """M^-1 r: z^0 = P r, z = P (r - L z) fwd times, then x = z - P U x bwd times from x = z."""
        z = self.pivot(r)
        for _ in range(fwd):
            z = self.pivot(r - self.L @ z)
        x = z
        for _ in range(bwd):
            x = z - self.pivot(self.U @ x)
        return x

    def coefficients(self, x):
        """x of one variable as [5][cell] in the caller's order."""
        out = np.zeros((5, self.T))
        out[:, self.perm] = x.reshape(self.T, 5).T
        return out

    def gmres(self, v, fwd, bwd, rtol, m, maxit):
        """Iterations of variable v and how many of them need the second Gram-Schmidt pass:
        the basis grows by w = K M^-1 V_j - V_j, a second pass where less than half of |w|
        is orthogonal to it."""
        b = self.b[v]
        x, it, second = np.zeros_like(b), 0, 0
        bn = np.linalg.norm(b)
        while it < maxit:
            r = b - self.K @ x
            beta = np.linalg.norm(r)
            if not beta > rtol * bn:
                break
            V, Z, H = [r / beta], [], np.zeros((m + 1, m))
            for j in range(m):
                Z.append(self.precond(V[j], fwd, bwd))
                w = self.K @ Z[j] - V[j]
                A = np.array(V)
                n0, h = np.linalg.norm(w), A @ w
                w = w - h @ A
                if np.linalg.norm(w) < 0.5 * n0:
                    second += 1
                    h2 = A @ w
                    w, h = w - h2 @ A, h + h2
                H[:j + 1, j], H[j + 1, j] = h, np.linalg.norm(w)
                H[j, j] += 1.0
                it += 1
                e = np.zeros(j + 2)
                e[0] = beta
                y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
                res = np.linalg.norm(H[:j + 2, :j + 1] @ y - e)
                if res <= rtol * bn or it >= maxit or not H[j + 1, j] > 0.0:
                    break
                V.append(w / H[j + 1, j])
            x = x + np.array(Z).T @ y
        return it, second
