"""A transport map that stays in the L2 and one that streams through it are
read by different loads: the same mesh alone (a small map) and among copies of
itself that take the union's map past the line gives the same concentrations,
bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1602_03641_gb300 as vag  # noqa: E402
import vag_inputs as vi  # noqa: E402


# 12 bytes an entry and 24 a row: 0.4 MB and 9 MB alone; 7 copies stay below 80 MiB, 12 exceed it
@pytest.mark.parametrize("n,copies", [(13, 3), (40, 7), (40, 12)])
def test_alone_and_in_a_union(n, copies):
    pb = vi.random_dfn_problem(n, 4, 1e3, seed=2)
    rng = np.random.default_rng(5)
    ctx = vag.Context(0)
    got = []
    start = rng.random(pb.n_nodes + pb.n_ff + pb.n_cells)
    cut = [pb.n_nodes, pb.n_nodes + pb.n_ff]
    for k in (1, copies):
        s = ctx.assemble_batch([vag.problem_arrays(pb)] * k)
        s.solve(rtol=1e-10, maxit=20000)
        c = np.concatenate([np.tile(part, k) for part in np.split(start, cut)])
        s.transport(c, np.tile(pb.phi_m, k), np.tile(pb.phi_f, k), np.tile(pb.cbar, k), n_steps=23, cfl=0.9)
        parts = np.split(c, [k * cut[0], k * cut[1]])
        got.append([p.reshape(k, -1) for p in parts])
        s.close()
    for alone, union in zip(*got):
        np.testing.assert_array_equal(np.broadcast_to(alone, union.shape), union)
    ctx.close()
