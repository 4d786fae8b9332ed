"""The device-ended inner loops of the mixed solves: every refinement step whose
inner tolerance is out of reach takes the iteration cap exactly, whatever the
number of iterations in a pass over the loop's body."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


# the first inner solves ask for 1e-6, the later ones for 0.3 of the reduction that is left, at most 0.1: up to
# five iterations of either preconditioner reach neither at contrast 1e3
@pytest.mark.parametrize("maxit", [1, 3, 4, 5])
@pytest.mark.parametrize("precision,precond", [(vag.VAG_MIXED, vag.VAG_PC_JACOBI), (vag.VAG_MIXED, vag.VAG_PC_AMG),
                                               (vag.VAG_MIXED, vag.VAG_PC_AMG_RS), (vag.VAG_MIXED_F16, vag.VAG_PC_AMG)])
def test_inner_cap_is_exact(precision, precond, maxit):
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, vi.random_dfn_problem(9, 3, 1e3, 5))
    _, info = s.solve(precision=precision, precond=precond, rtol=1e-12, maxit=maxit, raise_on_error=False)
    assert info.outer >= 1 and info.iterations == maxit * info.outer
    s.close()
    ctx.close()
