"""A memory budget that holds a small system's arrays holds its AMG solves: the
hierarchy is counted by its arrays, not by larger pieces that they share."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


# 77 unknowns: the dense inverse takes 47 KiB in FP64 and 24 KiB in FP32, an FP32 copy of the sliced ELL at most
# 12 KiB (96 padded rows of up to 32 entries; two of them in refinement), each of some 20 vectors at most 1 KiB
@pytest.mark.parametrize("precision", [vag.VAG_FP64, vag.VAG_MIXED])
@pytest.mark.parametrize("precond", [vag.VAG_PC_AMG, vag.VAG_PC_AMG_RS])
def test_small_hierarchy_fits_what_its_arrays_take(precision, precond):
    pb = vi.random_dfn_problem(4, 1, 1e2, 5)
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, pb)
    s.solve(rtol=1e-10)
    held = ctx.bytes_in_use()
    s.close()
    ctx.close()
    ctx = vag.Context(0, budget_bytes=held + (128 << 10))
    s = vag.assemble_problem(ctx, pb)
    s.solve(rtol=1e-10)
    _, info = s.solve(precision=precision, precond=precond, rtol=1e-10)
    assert info.status == vag.VAG_OK and ctx.bytes_in_use() <= held + (128 << 10)
    s.close()
    assert ctx.bytes_in_use() == 0
    ctx.close()
