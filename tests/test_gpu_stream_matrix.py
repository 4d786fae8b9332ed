"""Matrices too large for the L2 are read as packed streams: the same products
and solutions, bit for bit, as the plain arrays of a context with a budget."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


# below the line; above it with ragged slices and fracture rows in all directions; planes so
# wide that the columns of an interior slice span more than 16 bits
@pytest.mark.parametrize("dims", [(40, 38, 41), (79, 77, 83), (201, 198, 13)])
def test_packed_columns(dims):
    nx, ny, nz = dims
    frac = [(0, nx // 2, 0, ny, 0, nz), (1, ny // 3, 3, nx - 2, 0, nz), (2, nz // 2, 0, nx // 2, 0, ny)]
    pb = vi.build_problem(dims, frac, jitter=0.2, seed=7, lam_m="lognormal", ratio=1e3)
    got = []
    for budget in (0, 100 << 30):
        ctx = vag.Context(0, budget_bytes=budget)
        s = vag.assemble_problem(ctx, pb)
        x = np.random.default_rng(2).normal(size=s.info().n_rows)
        got.append([s.spmv(x)])
        for precision, precond in [(vag.VAG_MIXED, vag.VAG_PC_AMG), (vag.VAG_FP64, vag.VAG_PC_CHEBYSHEV),
                                   (vag.VAG_MIXED, vag.VAG_PC_JACOBI), (vag.VAG_FP64, vag.VAG_PC_AMG)]:
            got[-1].append(s.solve(precision=precision, precond=precond, rtol=1e-10, maxit=12, raise_on_error=False)[0])
        s.close()
        ctx.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
