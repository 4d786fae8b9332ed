"""Which loads are taken: a matrix of more than 128 MiB in FP64 holds the packed
columns (seen in the system's bytes), with slices of both kinds where planes are
wide; the FP16 finest level read through them gives the plain arrays' bits; and
the transport maps of the tests lie on the sides of the line that they claim."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


def problem(dims):
    nx, ny, nz = dims
    frac = [(0, nx // 2, 0, ny, 0, nz), (1, ny // 3, 3, nx - 2, 0, nz), (2, nz // 2, 0, nx // 2, 0, ny)]
    return vi.build_problem(dims, frac, jitter=0.2, seed=7, lam_m="lognormal", ratio=1e3)


def slices(rowptr, col):
    """(stored entries of the padded 32-row slices, column span of each slice)"""
    n = rowptr.size - 1
    length = np.diff(rowptr)
    width = np.maximum.reduceat(length, np.arange(0, n, 32))
    lo = np.minimum.reduceat(col, rowptr[:-1])
    hi = np.maximum.reduceat(col, rowptr[:-1])
    at = np.arange(0, n, 32)
    return 32 * int(width.sum()), np.maximum.reduceat(hi, at) - np.minimum.reduceat(lo, at)


def up(b):
    return -(-b // 256) * 256


@pytest.mark.parametrize("dims,packed,wide", [((40, 38, 41), False, False), ((79, 77, 83), True, False),
                                              ((201, 198, 13), True, True)])
def test_packed_columns_are_held_and_read(dims, packed, wide):
    pb = problem(dims)
    held, got = [], []
    for budget in (0, 100 << 30):
        ctx = vag.Context(0, budget_bytes=budget)
        s = vag.assemble_problem(ctx, pb)
        held.append(s.info().device_bytes)
        got.append(s.solve(precision=vag.VAG_MIXED_F16, precond=vag.VAG_PC_AMG, rtol=1e-10, maxit=12,
                           raise_on_error=False)[0])
        if not budget:
            stored, span = slices(*(s.export_system()[k] for k in ("rowptr", "col")))
        s.close()
        ctx.close()
    assert (12 * stored > 128 << 20) == packed
    assert held[0] - held[1] == (up(2 * stored) + up(4 * span.size) if packed else 0)
    if packed:   # rows next to fractures reach face rows; the first and the last plane reach one plane only
        assert (span < 65536).any() and (span >= 65536).any()
    assert (np.median(span) >= 65536) == wide
    np.testing.assert_array_equal(*got)


# the unions of test_gpu_step_loads.py: 12 bytes a stored entry and 24 a row, at most 80 MiB or more; the padding
# of the sorted rows stays below 15 % of the entries
@pytest.mark.parametrize("copies,stays", [(1, True), (7, True), (12, False)])
def test_sides_of_the_transport_line(copies, stays):
    pb = vi.random_dfn_problem(40, 4, 1e3, seed=2)
    ctx = vag.Context(0)
    s = ctx.assemble_batch([vag.problem_arrays(pb)] * copies)
    s.solve(rtol=1e-10, maxit=20000)
    n = s.info().n_cv
    s.transport(np.zeros(n), np.tile(pb.phi_m, copies), np.tile(pb.phi_f, copies), np.tile(pb.cbar, copies), n_steps=1)
    entries = s.info().nnz_transport
    if stays:
        assert 1.15 * 12 * entries + 24 * n <= 80 << 20
    else:
        assert 12 * entries + 24 * n > 80 << 20
    s.close()
    ctx.close()
