"""The Gram-Schmidt products of GMRES at the edges of their loops: basis sizes
around the eight vectors of a pass, systems of one tile up to more tiles than
one round of the last tile adds, and a second cycle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


def _gmres_residual(A, b, d, steps):
    """||b - A x|| / ||b|| after `steps` iterations of GMRES, right Jacobi preconditioner, in numpy."""
    r, left = b.copy(), steps
    while left:
        m = min(left, 30)
        V, W = [r / np.linalg.norm(r)], []
        for _ in range(m):
            w = A @ (d * V[-1])
            W.append(w)
            for _ in range(2):
                Q = np.array(V)
                w = w - Q.T @ (Q @ w)
            V.append(w / np.linalg.norm(w))
        W = np.array(W).T
        y, *_ = np.linalg.lstsq(W, r, rcond=None)
        r = r - W @ y
        left -= m
    return np.linalg.norm(r) / np.linalg.norm(b)


# rows 256 (1 tile), 2464 (10 tiles, the last ragged), 32768 (128 tiles), 33792 (132 tiles)
@pytest.mark.parametrize("dims", [(5, 7, 7), (9, 13, 21), (33, 31, 31), (34, 31, 31)])
def test_residual_of_a_given_number_of_steps(dims):
    from scipy.sparse import csr_matrix
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, vi.build_problem(dims, [], jitter=0.2, seed=7, lam_m="lognormal", ratio=1e3))
    e = s.export_system()
    A, b = csr_matrix((e["val"], e["col"], e["rowptr"])), e["rhs"]
    for steps in (1, 7, 8, 9, 16, 17, 30, 31):
        # the residual is a minimum: errors of size eps in the basis move it by less than 1e-10 of itself
        # while it is above 1e-5 of b (a wrong product moves it by the order of one step's reduction)
        _, info = s.solve(krylov=vag.VAG_KRYLOV_GMRES, rtol=1e-14, maxit=steps, raise_on_error=False)
        assert info.iterations == steps
        assert abs(info.rel_residual - _gmres_residual(A, b, 1.0 / A.diagonal(), steps)) < 1e-8
    s.close()
    ctx.close()
