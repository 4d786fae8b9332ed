"""The device-ended Krylov loops: an iteration cap is met exactly (whatever the
number of iterations in a pass over the loop's body), and a system that needs
no iteration ends the loop in its first pass."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402

SOLVERS = [(vag.VAG_PC_JACOBI, vag.VAG_KRYLOV_CG), (vag.VAG_PC_CHEBYSHEV, vag.VAG_KRYLOV_CG),
           (vag.VAG_PC_AMG, vag.VAG_KRYLOV_CG), (vag.VAG_PC_AMG_RS, vag.VAG_KRYLOV_CG),
           (vag.VAG_PC_JACOBI, vag.VAG_KRYLOV_BICGSTAB), (vag.VAG_PC_AMG, vag.VAG_KRYLOV_BICGSTAB)]


@pytest.fixture(scope="module")
def ctx():
    c = vag.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("maxit", [1, 3, 4, 5])
@pytest.mark.parametrize("precond,krylov", SOLVERS)
def test_iteration_cap_is_exact(ctx, precond, krylov, maxit):
    s = vag.assemble_problem(ctx, vi.random_dfn_problem(9, 3, 1e3, 5))
    _, info = s.solve(precond=precond, krylov=krylov, rtol=1e-12, maxit=maxit, raise_on_error=False)
    assert info.status == vag.VAG_ENOTCONVERGED and info.iterations == maxit
    s.close()


@pytest.mark.parametrize("precision", [vag.VAG_FP64, vag.VAG_MIXED])
@pytest.mark.parametrize("precond,krylov", SOLVERS)
def test_zero_right_hand_side_needs_no_iteration(ctx, precision, precond, krylov):
    if precision == vag.VAG_MIXED and (precond == vag.VAG_PC_CHEBYSHEV or
                                       (precond == vag.VAG_PC_JACOBI and krylov != vag.VAG_KRYLOV_CG)):
        pytest.skip("not a combination the interface accepts")
    pb = vi.random_dfn_problem(6, 2, 1e3, 5)
    pb.dir_values = np.zeros_like(pb.dir_values)
    s = vag.assemble_problem(ctx, pb)
    u, info = s.solve(precision=precision, precond=precond, krylov=krylov, rtol=1e-12)
    assert info.iterations == 0 and not u.any()
    s.close()
