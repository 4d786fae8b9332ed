"""The kept graph of transport steps follows the arrays it was captured over:
runs of one system whose rows grow (more wells) and shrink again between long
and short transports give the concentrations of a fresh system, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


def wells(k):
    return dict(ff=np.arange(k, dtype=np.int32), wi=np.full(k, 1e-3), pw=np.full(k, 0.5), q=np.zeros(k),
                cin=np.zeros(k))


def run(s, pb, steps):
    c = pb.c0()
    s.transport(c, pb.phi_m, pb.phi_f, pb.cbar, n_steps=steps, cfl=0.9)
    return c


def test_rows_grow_and_shrink_between_long_runs():
    pb = vi.random_dfn_problem(9, 3, 1e3, 5)
    pb.wells = wells(1)
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, pb)
    s.solve(rtol=1e-12)
    first = run(s, pb, 47)            # captures the steps
    entries = s.info().nnz_transport
    # more rows, few entries, and too few steps for a graph
    s.update_props(pb.lambda_m.ravel(), pb.lambda_f, pb.d_f, pb.mu, wells=wells(40))
    s.solve(rtol=1e-12)
    fluxes = s.export_fluxes()
    s.set_fluxes(*[np.where(np.arange(f.size) < f.size // 3, f.ravel(), 0.0).reshape(f.shape) for f in fluxes])
    run(s, pb, 5)
    assert s.info().nnz_transport < entries // 2
    # as at first
    s.update_props(pb.lambda_m.ravel(), pb.lambda_f, pb.d_f, pb.mu, wells=wells(1))
    s.solve(rtol=1e-12)
    again = run(s, pb, 47)
    s.close()
    ctx.close()
    assert np.abs(first - pb.c0()).max() > 0.01
    np.testing.assert_array_equal(first, again)
