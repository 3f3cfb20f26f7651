"""The GMRES kernels step by step: iterates after 1 to 25 iterations, where
the products switch between shares of the rows (up to 16 vectors) and one
warp per four vectors, against GMRES in NumPy on the assembled matrix."""
import numpy as np
import pytest

import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def gmres_iterates(A, b, steps):
    """x after each of the given numbers of steps (Householder QR of the Krylov basis)."""
    n, m = len(b), max(steps)
    V = np.zeros((n, m + 1))
    H = np.zeros((m + 1, m))
    V[:, 0] = b / np.linalg.norm(b)
    for j in range(m):
        w = A @ V[:, j]
        for _ in range(2):
            h = V[:, :j + 1].T @ w
            w = w - V[:, :j + 1] @ h
            H[:j + 1, j] += h
        H[j + 1, j] = np.linalg.norm(w)
        V[:, j + 1] = w / H[j + 1, j]
    out = {}
    for k in steps:
        e = np.zeros(k + 1)
        e[0] = np.linalg.norm(b)
        y, res, *_ = np.linalg.lstsq(H[:k + 1, :k], e, rcond=None)
        out[k] = (V[:, :k] @ y, np.linalg.norm(H[:k + 1, :k] @ y - e) / e[0])
    return out


def test_iterates():
    """FP64 throughout; 640 unknowns in three blocks of 214 rows, the last one
    short.  The two sides share the matrix to 1e-13 and lose at most a few
    digits more while the residual falls: 1e-8 for the iterates, relative."""
    import paper_2103_01048_gb300 as pb
    V, F = synthetic.icosphere(2, 2.0)
    V = V * (1 + 0.3 * np.sin(5 * V[:, :1]) * np.cos(3 * V[:, 1:2]))        # no symmetry, slower convergence
    F = F.astype(np.int32)
    n = 2 * len(F)
    atoms, q = np.array([[0.3, -0.2, 0.5], [-0.6, 0.1, -0.2]]), np.array([0.7, -0.4])
    ctx = pb.pb_create(0, None)
    try:
        mesh = pb.pb_mesh_setup(ctx, V, F, 3, 8, 4096)       # one leaf: direct sums
        A, e, y = np.zeros((n, n)), np.zeros(n), np.zeros(n)
        for k in range(n):
            e[:] = 0.0
            e[k] = 1.0
            pb.pb_mesh_matvec(ctx, mesh, e, y, 4.0, 80.0, 0.125, precision=pb.PB_FP64, precond=True)
            A[:, k] = y

        def solve(tol, steps):
            res, _ = pb.pb_solve(ctx, mesh, atoms, q, 4.0, 80.0, 0.125, tol, steps, precision=pb.PB_FP64)
            it, rr, x = pb.pb_result_get(res, len(F))
            pb.pb_result_destroy(res)
            return it, rr, x

        steps = [1, 2, 3, 4, 5, 7, 8, 9, 12, 13, 16, 17, 20, 25]
        it, _, x = solve(1e-14, 500)
        assert it > steps[-1]
        want = gmres_iterates(A, A @ x, steps)
        for k in steps:
            it, rr, x = solve(0.0, k)
            xr, resid = want[k]
            print(k, np.linalg.norm(x - xr) / np.linalg.norm(xr), rr, resid)
            assert it == k
            assert np.linalg.norm(x - xr) <= 1e-8 * np.linalg.norm(xr)
            assert abs(rr - resid) <= 1e-8
        pb.pb_mesh_destroy(mesh)
    finally:
        pb.pb_destroy(ctx)
