"""Pair-density rows transformed in tiles of occupied x unoccupied states: counts that leave ragged tiles,
one-state tiles and odd numbers of tasks, every compiled plane size, both routes of the table form compared."""
import numpy as np
import pytest
import torch

from paper_1810_07772_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,gcut", [(12, 8), (16, 13), (18, 16), (20, 20), (24, 29), (27, 37)])
@pytest.mark.parametrize("nv,nc", [(1, 1), (1, 11), (2, 9), (4, 6), (5, 7), (9, 13)])
def test_tiles_match_the_table_form(n, gcut, nv, nc):
    dims = (n, n, n)
    psi, E = inputs.make_states(0, nv, nc, n + nv + nc, dims=dims)
    out = {}
    with gw.Context(0) as ctx:
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).to(DEV), E, dims, nv)
        for kind in ("two_kernel", "tables"):
            ctx.set_transform_kernel(kind)
            ctx.build_PG(gcut)
            out[kind] = ctx.view("PG").cpu().numpy()
    # the same FP32 sums in the same order; the twiddles differ only in the exact zeros
    d = np.linalg.norm(out["two_kernel"] - out["tables"])
    assert d <= 1e-7 * np.linalg.norm(out["tables"])
