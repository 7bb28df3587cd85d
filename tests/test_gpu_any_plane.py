"""Plane transforms of sizes without a compiled kernel: the two-kernel form against the table form (row-block kernel
or stored pair densities above 4096 rows), both routes, odd and even sides, the smallest plane of the rule and one below
it, few and many columns, and a plane that fits fewer warps."""
import numpy as np
import pytest
import torch

from paper_1810_07772_gb300 import gw

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def two_kernel_and_tables(dims, gcut, nv, nc):
    """P~ by both routes, each pair by the two-kernel form and by the table form."""
    rng = np.random.default_rng(sum(dims))
    nr = int(np.prod(dims))
    psi = (rng.standard_normal((nv + nc, nr)) + 1j * rng.standard_normal((nv + nc, nr))) / np.sqrt(2 * nr)
    E = np.concatenate([np.linspace(-5, -1, nv), np.linspace(1, 9, nc)])
    out = []
    with gw.Context(0) as ctx:
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).to(DEV), E, dims, nv)
        for kind in ("two_kernel", "tables"):
            ctx.set_transform_kernel(kind)
            ctx.build_P("fp16x3")
            ctx.P_to_G(gcut)
            r = ctx.view("PG").cpu().numpy()
            ctx.build_PG(gcut)
            out.append((r, ctx.view("PG").cpu().numpy()))
    return list(zip(*out))


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
    for a, b in two_kernel_and_tables(dims, gcut, nv, nc):
        # FP32 sums of the same terms in two orders: at most 50 terms a stage, three stages twice over
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)


def _random_states(dims, nv, nc):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(nv + nc)
    psi = torch.randn((nv + nc, int(np.prod(dims))), dtype=torch.complex64, device=DEV, generator=gen)
    return psi / np.sqrt(psi.shape[1]), np.concatenate([np.linspace(-5, -1, nv), np.linspace(1, 9, nc)])


@pytest.mark.parametrize("nv,nc", [(45, 330), (1, 14500)])
def test_slices_of_the_workspace(nv, nc):
    """31 x 23 x 29 with N_g = 3900 takes 14000 rows at once: two slices of P's rows, two of whole occupied states (14850
    pair rows), parts of one state; the closure's pairs with every loaded state start at a later occupied state."""
    dims, gcut = (31, 23, 29), 96
    psi, E = _random_states(dims, nv, nc)
    out = {}
    with gw.Context(0) as ctx:
        ctx.load_states(psi, E, dims, nv)
        del psi
        for kind in ("two_kernel", "tables"):
            ctx.set_transform_kernel(kind)
            r = []
            if nv > 1:
                ctx.build_P("fp16x3")
                ctx.P_to_G(gcut)
                r.append(ctx.view("PG").clone())
            ctx.build_PG(gcut)
            r.append(ctx.view("PG").clone())
            if nv > 1:
                ctx.build_P("fp16x3")
                ctx.P_to_G(gcut)       # takes Q: the closure then transforms every pair itself
                r.append(ctx.corr_closure(gcut, E[-1] + np.arange(1.0, 9.0)) if kind == "two_kernel" else None)
            out[kind] = r
        if nv > 1:
            ctx.set_transform_kernel("fused")
            out["tables"][2] = ctx.corr_closure(gcut, E[-1] + np.arange(1.0, 9.0))
        for a, b in zip(out["two_kernel"], out["tables"]):
            # FP32 sums of the same terms in two orders, then the same 22-bit update
            assert float((a - b).norm()) <= 2e-6 * float(b.norm())


def test_workspace_of_a_long_transform_is_bounded():
    """P_to_G on a grid without a compiled n3: its two row transforms (N_r x N_g each), a few N_g x N_g arrays and
    a workspace of 1 GB, not of all N_r rows."""
    dims, gcut = (31, 23, 29), 96
    nr = int(np.prod(dims))
    psi, E = _random_states(dims, 2, 3)
    with gw.Context(0) as ctx:
        ctx.load_states(psi, E, dims, 2)
        ctx.build_P("fp16x3")
        ctx.sync()
        free = torch.cuda.mem_get_info(0)[0]
        g = ctx.P_to_G(gcut)
        ctx.sync()
        used = free - torch.cuda.mem_get_info(0)[0]
    ng, disk = len(g), len({(m[1], m[2]) for m in g.tolist()})
    assert nr * dims[0] * disk * 8 > 1.4e9
    assert used <= 2 * nr * ng * 8 + 3 * ng * ng * 8 + (1 << 30) + (128 << 20)
