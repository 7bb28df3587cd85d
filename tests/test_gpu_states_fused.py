"""States from plane-wave coefficients made in one kernel over the Miller indices in use: grids of unequal,
odd and largest sides, full and sparse index sets, one plane wave, and a set too wide for a CTA's shared
memory (the axis kernels), against the oracle's phase sums."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_1810_07772_gb300 import gw, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _full(dims):
    return np.indices(dims).reshape(3, -1).T.astype(np.int32)


def _random(dims, n, seed):
    p = np.random.default_rng(seed).choice(int(np.prod(dims)), n, replace=False)
    return np.stack(np.unravel_index(p, dims), axis=1).astype(np.int32)


CASES = [
    ((2, 3, 5), _full((2, 3, 5))),
    ((7, 11, 13), _full((7, 11, 13))),
    ((64, 4, 6), _full((64, 4, 6))),
    ((4, 6, 64), _random((4, 6, 64), 200, 1)),
    ((16, 16, 16), inputs.psi_sphere((16, 16, 16), 20)),
    ((20, 20, 20), inputs.psi_sphere((20, 20, 20), 36)),
    ((9, 8, 33), _random((9, 8, 33), 40, 2)),
    ((12, 10, 8), np.array([[-1, 2, -3]], dtype=np.int32)),
    ((40, 40, 12), np.array([[i, (7 * i) % 40 - 20, i % 12] for i in range(40)], dtype=np.int32)),  # axis kernels
]


@pytest.mark.parametrize("dims,gvec", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else None)
@pytest.mark.parametrize("nb", [2, 5])
def test_states_match_phase_sums(dims, gvec, nb):
    rng = np.random.default_rng(nb)
    coef = (rng.standard_normal((nb, len(gvec))) + 1j * rng.standard_normal((nb, len(gvec)))).astype(np.complex64)
    E = np.concatenate([[-5.0], np.linspace(1.0, 9.0, nb - 1)])
    ref = O.states_from_g(coef, gvec, dims)
    with gw.Context(0) as ctx:
        ctx.load_states_g(torch.from_numpy(coef).to(DEV), gvec, E, dims, 1)
        u = ctx.view("psiT").cpu().numpy().T
    # three FP32 sums of at most 64 terms each, rounding errors of random sign
    assert np.linalg.norm(u - ref) <= 1e-6 * np.linalg.norm(ref)
