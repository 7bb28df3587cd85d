"""The Cholesky inverse at the edges of its blocks and tiles (32-wide steps, 8 x 16 and 16 x 16 tiles, pairs of blocks
with a short second one), by gw_eps_inv_noalloc: the residual of a well-conditioned matrix, and a bad pivot in
the first block, a later one and the last."""
import numpy as np
import pytest

from paper_1810_07772_gb300 import gw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _matrix(n):
    rng = np.random.default_rng(n)
    B = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) / np.sqrt(4 * n)
    return np.eye(n) + B @ B.conj().T


def _inverse(A):
    eps = torch.from_numpy(A).to(DEV)
    out = torch.empty_like(eps)
    return gw.lib().gw_eps_inv_noalloc(eps.data_ptr(), A.shape[0], out.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream), out.cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 9, 31, 32, 33, 47, 48, 49, 63, 64, 65, 80, 95, 96, 97, 127, 129, 160, 191, 255, 258,
                               300, 419, 512])
def test_residual(n):
    A = _matrix(n)
    st, X = _inverse(A)
    assert st == gw.GW_OK
    # condition number below 10; each of the three stages adds at most n products of unit-sized entries
    assert np.max(np.abs(A @ X - np.eye(n))) <= 1e-14 * max(8, n)
    # mirrored; on the diagonal a y - y a of each term is rounded once, so up to u |Y|^2 per term stays
    d = np.diag(np.diag(X))
    assert np.array_equal(X - d, (X - d).conj().T)
    assert np.max(np.abs(d.imag)) <= 1.2e-16 * np.max(d.real)


@pytest.mark.parametrize("n,bad", [(20, 5), (200, 3), (200, 32), (200, 63), (200, 199)])
def test_bad_pivot_is_reported(n, bad):
    A = _matrix(n)
    A[bad, bad] = -1.0
    assert _inverse(A)[0] == gw.GW_E_NUMERIC
    assert _inverse(_matrix(n))[0] == gw.GW_OK
