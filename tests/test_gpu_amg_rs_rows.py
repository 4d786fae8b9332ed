"""Rows of the classical hierarchy that few meshes make: equal couplings in
every row of the finest level (the four strongest neighbours are a matter of
position) and restriction rows of more than 32 entries (a coarse level of the
second mesh has rows of 37).  The entries of a restriction row arrive in the
order of atomics, so an unsorted row would change the bits from solve to solve;
the residuals are taken here from the exported system."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402

MESHES = {"equal": lambda: vi.config_plain16(33), "long": lambda: vi.random_dfn_problem(40, 12, 1e4, 3)}


@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("precision", [vag.VAG_FP64, vag.VAG_MIXED])
def test_same_bits_every_time(mesh, precision):
    pb = MESHES[mesh]()
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, pb)
    q = s.export_system()
    A = sp.csr_matrix((q["val"], q["col"], q["rowptr"]), shape=(q["rhs"].size,) * 2)
    got = [s.solve(precision=precision, precond=vag.VAG_PC_AMG_RS, rtol=1e-10) for _ in range(4)]
    for u, info in got:
        assert np.array_equal(u, got[0][0]) and info.iterations == got[0][1].iterations <= 60
    r = q["rhs"] - A @ got[0][0][q["row_dof"]]
    assert np.linalg.norm(r) <= 1.1e-10 * np.linalg.norm(q["rhs"])
    s.close()
    ctx.close()
