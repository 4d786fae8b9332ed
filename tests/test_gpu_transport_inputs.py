"""Porosities and Dirichlet concentrations are copied before a kernel reads
them: device arrays at any byte offset, and pinned host memory passed as device
memory, give the concentrations of plain host arrays, bit for bit."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402
from paper_1602_03641_gb300.vag import vag_transport_info, vag_transport_opts  # noqa: E402


def placed(a, how):
    """(the memory, the address in it of a's doubles)"""
    raw = np.frombuffer(np.ascontiguousarray(a, np.float64).tobytes(), np.uint8)
    if how == "pinned":
        buf = torch.empty(raw.size, dtype=torch.uint8, pin_memory=True)
        buf.copy_(torch.from_numpy(raw.copy()))
        return buf, buf.data_ptr()
    buf = torch.zeros(raw.size + 16, dtype=torch.uint8, device="cuda")
    buf[how:how + raw.size] = torch.from_numpy(raw.copy()).cuda()
    return buf, buf.data_ptr() + how


@pytest.mark.parametrize("how", [0, 4, 1, "pinned"])
def test_any_place_of_the_inputs(how):
    pb = vi.random_dfn_problem(7, 3, 1e3, 5)
    ctx = vag.Context(0)
    s = vag.assemble_problem(ctx, pb)
    s.solve(rtol=1e-12)
    ref = pb.c0()
    s.transport(ref, pb.phi_m, pb.phi_f, pb.cbar, n_steps=23, cfl=0.9)
    c = torch.from_numpy(pb.c0()).cuda()
    keep = [placed(a, how) for a in (pb.phi_m, pb.phi_f, pb.cbar)]
    torch.cuda.synchronize()
    o = vag_transport_opts(keep[0][1], keep[1][1], keep[2][1], 0.5, 0.9, 0.0, 23, vag.VAG_MEM_DEVICE)
    inf = vag_transport_info()
    ctx.check(vag.lib().vag_transport(s.h, C.byref(o), C.c_void_p(c.data_ptr()), C.byref(inf)))
    np.testing.assert_array_equal(c.cpu().numpy(), ref)
    s.close()
    ctx.close()
