"""Meshes whose node, cell and row counts lie at the edges of the setup scans'
tiles (4096 values): with Lambda_m = I and a fracture normal to the gradient
the pressure is 1 - x exactly, so a wrong offset anywhere in the maps, the
pattern or the hierarchy shows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


# node counts 8, 4095, 4096, 4352, 8192, 9216; cell counts 1, 4096, 8192
@pytest.mark.parametrize("dims", [(1, 1, 1), (14, 12, 20), (15, 15, 15), (16, 15, 15), (16, 16, 16), (31, 31, 7),
                                  (32, 16, 16), (31, 31, 8)])
def test_affine_pressure(dims):
    frac = [(0, dims[0] // 2, 0, dims[1], 0, dims[2])] if dims[0] > 1 else []
    pb = vi.build_problem(dims, frac, jitter=0.2, seed=3)
    exact = 1.0 - pb.xyz[:, 0]
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, pb)
    for precond in (vag.VAG_PC_JACOBI, vag.VAG_PC_AMG, vag.VAG_PC_AMG_RS):
        # (the FP64 rounding floor of the residual is near 1e-12 at this contrast: the last iterate is judged)
        u, _ = s.solve(precond=precond, rtol=1e-12, raise_on_error=False)
        assert np.abs(u[:pb.n_nodes] - exact).max() <= 1e-10
    s.close()
    ctx.close()
