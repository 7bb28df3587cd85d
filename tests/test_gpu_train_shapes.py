"""The training step's kernels at the edges of their tiles: one input, one neuron, one row; batches around
16-row chunks and 128-row blocks, widths off the 16- and 32-column groups, the most inputs, and batches on both
sides of the tile-width rule (4864 rows); the gradient against the FP64 oracle, then two Adam steps against the same rule
applied to the library's own gradients."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_1810_07772_gb300 import gw, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _setup(n_in, hid, B):
    rng = np.random.default_rng(n_in + hid + B)
    X = rng.standard_normal((B + 7, n_in)).astype(np.float32)
    T = rng.standard_normal((B + 7, 2)).astype(np.float32)
    rows = rng.permutation(B + 7)[:B].astype(np.int32)
    return X, T, rows, (inputs.mlp_init(n_in, hid, 3) + 0.02 * rng.standard_normal(
        hid * (n_in + 2 * hid + 5) + 2)).astype(np.float32)


@pytest.mark.parametrize("n_in,hid,B", [(1, 1, 1), (12, 16, 15), (17, 40, 16), (64, 130, 129), (5, 33, 1000),
                                        (12, 256, 2048), (12, 256, 5000), (3, 600, 130)])
def test_gradient(n_in, hid, B):
    X, T, rows, th = _setup(n_in, hid, B)
    params = M.unpack(M.to_fp16_weights(th.astype(np.float64), n_in, hid), n_in, hid)
    loss_ref, grads = M.loss_and_grad(params, X[rows].astype(np.float64), T[rows].astype(np.float64))
    g_ref = M.flatten(grads)
    with gw.Mlp(n_in, hid, max_batch=B + 5, device=0) as net:
        net.set_params(th)
        g, loss = net.grad(torch.from_numpy(X).to(DEV), torch.from_numpy(T).to(DEV), torch.from_numpy(rows).to(DEV))
        net.check()
    g = g.cpu().numpy().astype(np.float64)
    # FP32 sums of at most max(B, hid) terms in each of eight product stages, sqrt(5000) u_32 = 4e-6 a stage
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    assert np.linalg.norm(g - g_ref) <= 2e-5 * np.linalg.norm(g_ref)


@pytest.mark.parametrize("n_in,hid,B", [(12, 256, 300), (5, 33, 40)])
def test_two_steps_follow_the_gradients(n_in, hid, B):
    X, T, rows, th = _setup(n_in, hid, B)
    Xd, Td, rd = (torch.from_numpy(a).to(DEV) for a in (X, T, rows))
    lr, b1, b2, eps = 1e-3, 0.9, 0.999, 1e-8
    ref, m, v = th.astype(np.float64), 0.0, 0.0
    with gw.Mlp(n_in, hid, max_batch=B, device=0) as net, gw.Mlp(n_in, hid, max_batch=B, device=0) as other:
        net.set_params(th)
        for t in (1, 2):
            other.set_params(net.get_params())     # the operands packed afresh
            g = other.grad(Xd, Td, rd)[0].cpu().numpy().astype(np.float64)
            m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
            ref = ref - lr * (m / (1 - b1 ** t)) / (np.sqrt(v / (1 - b2 ** t)) + eps)
            net.train_step(Xd, Td, rd, lr)
        got = net.get_params()
        net.check()
    # the step's operands are those the gradient was taken with: equal up to FP32 rounding of the update (an entry
    # whose gradient is near the sums' rounding error may move differently by a fraction of lr)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref - th)
