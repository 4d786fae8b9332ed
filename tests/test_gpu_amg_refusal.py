"""A hierarchy with a terminal block that is not positive definite refuses the
solve before anything is written: VAG_EINVAL, no fluxes from it, the fluxes and
the pressures that were there stay, and later solves do not meet its status."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402

SOLVERS = [(vag.VAG_FP64, vag.VAG_PC_AMG, vag.VAG_KRYLOV_CG), (vag.VAG_FP64, vag.VAG_PC_AMG_RS, vag.VAG_KRYLOV_CG),
           (vag.VAG_FP64_PC32, vag.VAG_PC_AMG_RS, vag.VAG_KRYLOV_CG), (vag.VAG_MIXED, vag.VAG_PC_AMG, vag.VAG_KRYLOV_CG),
           (vag.VAG_MIXED_F16, vag.VAG_PC_AMG, vag.VAG_KRYLOV_CG), (vag.VAG_FP64, vag.VAG_PC_AMG, vag.VAG_KRYLOV_BICGSTAB),
           (vag.VAG_FP64, vag.VAG_PC_AMG, vag.VAG_KRYLOV_GMRES), (vag.VAG_MIXED, vag.VAG_PC_AMG_RS, vag.VAG_KRYLOV_GMRES)]


@pytest.fixture(scope="module")
def ctx():
    c = vag.Context(0)
    yield c
    c.close()


def refused(call):
    with pytest.raises(vag.VagError) as e:
        call()
    assert e.value.code == vag.VAG_EINVAL


# 77 unknowns, one dense block: the tensors' xy term is twice their diagonal, so that the matrix has positive
# diagonals and nine negative eigenvalues
@pytest.mark.parametrize("zero_rhs", [False, True])
@pytest.mark.parametrize("precision,precond,krylov", SOLVERS)
def test_indefinite_terminal_block(ctx, precision, precond, krylov, zero_rhs):
    pb = vi.random_dfn_problem(4, 1, 1e2, 5)
    good = np.array(pb.lambda_m)
    bad = np.tile([1.0, 1.0, 1.0, 2.0, 0.0, 0.0], (pb.n_cells, 1))
    if zero_rhs:
        pb.dir_values = np.zeros_like(pb.dir_values)
    pb.lambda_m = bad
    s = vag.assemble_problem(ctx, pb)
    out = np.full(pb.n_nodes + pb.n_ff + pb.n_cells, 7.0)

    def solve():
        s.solve(out=out, precision=precision, precond=precond, krylov=krylov, rtol=1e-12, maxit=50)

    def transport():
        s.transport(pb.c0(), pb.phi_m, pb.phi_f, pb.cbar, n_steps=2, cfl=0.9)

    refused(solve)
    assert (out == 7.0).all()
    refused(transport)
    refused(s.export_fluxes)
    refused(s.solve_infos)
    refused(lambda: s.kernel_time(vag.VAG_KERNEL_SMOOTH, 1))
    # given fluxes survive a refused solve
    s.update_props(good.ravel(), pb.lambda_f, pb.d_f, pb.mu)
    s.solve(rtol=1e-12)
    flux = s.export_fluxes()
    s.update_props(bad.ravel(), pb.lambda_f, pb.d_f, pb.mu)
    s.set_fluxes(*flux)
    refused(solve)
    for a, b in zip(flux, s.export_fluxes()):
        np.testing.assert_array_equal(a, b)
    # and the next solve is judged by its own matrix
    s.update_props(good.ravel(), pb.lambda_f, pb.d_f, pb.mu)
    s.solve(rtol=1e-12)
    solve()
    s.close()


# 251 unknowns, whose coarse operators have non-positive diagonals (FP64 and FP32 hierarchies): the setup ends
# before its levels are complete
@pytest.mark.parametrize("precision", [vag.VAG_FP64, vag.VAG_MIXED])
@pytest.mark.parametrize("precond", [vag.VAG_PC_AMG, vag.VAG_PC_AMG_RS])
def test_a_setup_that_fails_half_way_leaves_no_hierarchy(ctx, precision, precond):
    pb = vi.random_dfn_problem(6, 1, 1e2, 5)
    s = vag.assemble_problem(ctx, pb)
    s.solve(precision=precision, precond=precond, rtol=1e-10)
    assert s.kernel_time(vag.VAG_KERNEL_SMOOTH, 1) > 0.0
    bad = np.tile([1.0, 1.0, 1.0, 2.0, 0.0, 0.0], pb.n_cells)
    s.update_props(bad, pb.lambda_f, pb.d_f, pb.mu)
    refused(lambda: s.solve(precision=precision, precond=precond, rtol=1e-10, maxit=50))
    refused(lambda: s.kernel_time(vag.VAG_KERNEL_SMOOTH, 1))
    s.close()
