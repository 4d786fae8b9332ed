"""The per-system sums of the Krylov kernels at the edges of their ways: one
tile of 256 rows, one group of 32 tiles, the largest system whose sums its last
tile makes alone (1024 tiles), and one tile past each."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


def _jacobi_cg_residual(s, steps):
    """||b - A x|| / ||b|| after `steps` iterations of Jacobi CG, in numpy."""
    from scipy.sparse import csr_matrix
    e = s.export_system()
    A, b = csr_matrix((e["val"], e["col"], e["rowptr"])), e["rhs"]
    d = 1.0 / A.diagonal()
    x, r = np.zeros_like(b), b.copy()
    p = d * r
    rz = r @ p
    for _ in range(steps):
        q = A @ p
        a = rz / (p @ q)
        x += a * p
        r -= a * q
        z = d * r
        rz, old = r @ z, rz
        p = z + rz / old * p
    return np.linalg.norm(b - A @ x) / np.linalg.norm(b)


# rows = (nx - 1)(ny + 1)(nz + 1): both ends in x hold the pressure
@pytest.mark.parametrize("dims,tiles", [((2, 7, 7), 1), ((5, 7, 7), 1), ((3, 15, 15), 2), ((9, 31, 31), 32),
                                        ((34, 15, 15), 33), ((65, 63, 63), 1024), ((42, 79, 79), 1025)])
def test_sums_of_all_tiles(dims, tiles):
    pb = vi.build_problem(dims, [], jitter=0.2, seed=7, lam_m="lognormal", ratio=1e3)
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, pb)
    assert -(-s.info().n_rows // 256) == tiles
    # a product and two updates a step, each with sums: a tile lost or added twice moves the
    # residual by about 1 / tiles; rounding by a few n_rows^(1/2) eps < 1e-12
    _, info = s.solve(rtol=1e-14, maxit=3, raise_on_error=False)
    assert info.iterations == 3
    assert abs(info.rel_residual / _jacobi_cg_residual(s, 3) - 1.0) < 1e-10
    s.close()
    ctx.close()
