"""A context that loads state after state keeps its sphere plan while the grid and the cell stay: the
results are those of a fresh context, whatever changed between the loads."""
import numpy as np
import pytest

from paper_1810_07772_gb300 import gw, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def one_pass(ctx, dims, nv, nc, seed, gcut, cell_L, q, route):
    psi, E = inputs.make_states(0, nv, nc, seed, dims=dims)
    ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).cuda(), E, dims, nv, cell_L=cell_L)
    ctx.set_q(q)
    if route == "gspace":
        g = ctx.build_PG(gcut)
    else:
        ctx.build_P()
        g = ctx.P_to_G(gcut)
    inv = torch.empty((len(g), len(g)), dtype=torch.complex128, device="cuda:0")
    ctx.eps_inv("newton_tc", epsinv_out=inv)
    clos = ctx.corr_closure(gcut, np.array([25.0, 30.0]))
    ctx.sync()
    return g, ctx.view("PG").clone(), inv, clos


def test_sequence_equals_fresh_contexts():
    """Same grid again; another q; another cell; the same points in another shape; another cut and back;
    a smaller and a larger number of states."""
    steps = [((8, 9, 10), 4, 20, 1, 5, 1.0, (0, 0, 0), "rspace"), ((8, 9, 10), 4, 20, 2, 5, 1.0, (0, 0, 0), "gspace"),
             ((8, 9, 10), 4, 20, 3, 5, 1.0, (0.1, 0, 0.2), "rspace"), ((8, 9, 10), 4, 20, 4, 5, 2.5, (0, 0, 0), "gspace"),
             ((10, 9, 8), 4, 20, 5, 5, 2.5, (0, 0, 0), "rspace"), ((10, 9, 8), 2, 7, 6, 9, 2.5, (0, 0, 0), "gspace"),
             ((10, 9, 8), 6, 40, 7, 5, 2.5, (0, 0, 0), "rspace")]
    with gw.Context(0) as ctx:
        for args in steps:
            got = one_pass(ctx, *args)
            with gw.Context(0) as fresh:
                want = one_pass(fresh, *args)
            assert np.array_equal(got[0], want[0])
            for a, b in zip(got[1:], want[1:]):
                assert torch.equal(a, b), args
