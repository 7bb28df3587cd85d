"""Plane transforms of sizes without a compiled kernel: the two-kernel form against the table form (row-block kernel
or stored pair densities above 4096 rows), both routes, odd and even sides, the smallest plane of the rule and one below
it, few and many columns, and a plane that fits fewer warps."""
import numpy as np
import pytest
import torch

from paper_1810_07772_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dims,gcut,nv,nc", [
    ((13, 14, 13), 9, 3, 9),      # 13 x 14: the smallest plane of the any-size kernel
    ((14, 13, 14), 9, 2, 7),
    ((12, 13, 13), 9, 3, 9),      # below it
    ((9, 22, 17), 1, 2, 3),       # M = 1
    ((10, 25, 23), 14, 2, 5),     # odd sides, rows above 4096
    ((8, 17, 22), 12, 45, 92),    # 4140 pair rows
    ((11, 28, 29), 20, 2, 4),
    ((6, 50, 49), 6, 1, 3),
])
def test_two_kernel_matches_tables(dims, gcut, nv, nc):
    rng = np.random.default_rng(sum(dims))
    nr = int(np.prod(dims))
    psi = (rng.standard_normal((nv + nc, nr)) + 1j * rng.standard_normal((nv + nc, nr))) / np.sqrt(2 * nr)
    E = np.concatenate([np.linspace(-5, -1, nv), np.linspace(1, 9, nc)])
    out = {}
    with gw.Context(0) as ctx:
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).to(DEV), E, dims, nv)
        for kind in ("two_kernel", "tables"):
            ctx.set_transform_kernel(kind)
            ctx.build_P("fp16x3")
            ctx.P_to_G(gcut)
            r = ctx.view("PG").cpu().numpy()
            ctx.build_PG(gcut)
            out[kind] = (r, ctx.view("PG").cpu().numpy())
    for a, b in zip(out["two_kernel"], out["tables"]):
        # FP32 sums of the same terms in two orders: at most 50 terms a stage, three stages twice over
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)
