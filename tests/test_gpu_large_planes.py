"""Constant-twiddle planes of 30 x 30, 32 x 32 and 36 x 36 points (one CTA per SM) and stage 3 of those lengths, against the
table form: the widest sphere (15 columns), few and many pair rows, an odd number of planes, and n1 alone at the size; and
planes of 15, 21, 25 and 28, whose table form sums in another order."""
import numpy as np
import pytest

from test_gpu_any_plane import two_kernel_and_tables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,gcut,nv,nc", [
    ((15, 30, 30), 49, 2, 5), ((15, 32, 32), 49, 1, 3), ((15, 36, 36), 49, 3, 9),
    ((3, 36, 36), 1, 5, 7), ((5, 30, 30), 4, 9, 21), ((7, 32, 32), 9, 4, 6),
    ((30, 12, 12), 25, 2, 5), ((32, 16, 16), 30, 2, 5), ((36, 18, 18), 30, 2, 5),
])
def test_constant_form_matches_tables(dims, gcut, nv, nc):
    # the same FP32 sums in the same order; the twiddles differ only in the exact zeros
    for a, b in two_kernel_and_tables(dims, gcut, nv, nc):
        assert np.linalg.norm(a - b) <= 1e-7 * np.linalg.norm(b)


@pytest.mark.parametrize("dims,gcut,nv,nc", [((7, 15, 15), 9, 3, 9), ((15, 21, 21), 49, 2, 5), ((9, 25, 25), 16, 5, 7),
                                             ((15, 28, 28), 49, 1, 4), ((21, 15, 15), 36, 2, 5), ((28, 25, 21), 16, 2, 3)])
def test_sizes_without_a_compiled_table_form(dims, gcut, nv, nc):
    # FP32 sums of the same terms in two orders: at most 28 terms a stage, three stages twice over
    for a, b in two_kernel_and_tables(dims, gcut, nv, nc):
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)
