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


def test_weight_gradients_of_a_large_batch():
    """Each layer's gradient at 8192 rows.  A truncating FP32 sum of n additions of one sign is short by n 2^-24 at
    most and by half of that on average: 1e-6 for 35 chunks with one addition of the sum's size each, beside
    5e-6 of the products before it (three-part splits through three layers).  Six such additions a chunk would
    leave 6.3e-6."""
    n_in, hid, B = 12, 256, 8192
    X, T, rows, th = _setup(n_in, hid, B)
    X[:, 9] = 1.0                                  # terms of one sign
    params = M.unpack(M.to_fp16_weights(th.astype(np.float64), n_in, hid), n_in, hid)
    _, grads = M.loss_and_grad(params, X[rows].astype(np.float64), T[rows].astype(np.float64))
    g_ref = M.flatten(grads)
    with gw.Mlp(n_in, hid, max_batch=B, device=0) as net:
        net.set_params(th)
        g = net.grad(torch.from_numpy(X).to(DEV), torch.from_numpy(T).to(DEV), torch.from_numpy(rows).to(DEV))[0]
        net.check()
    g = g.cpu().numpy().astype(np.float64)
    o = 0
    for n in (hid * n_in, hid, hid * hid, hid, hid * hid, hid, 2 * hid, 2):
        e = np.linalg.norm(g[o:o + n] - g_ref[o:o + n]) / np.linalg.norm(g_ref[o:o + n])
        assert e <= 6e-6, n
        o += n


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


def _order_keys(seed, n):
    """SplitMix64's output of the documented keys of the first pass."""
    u = np.uint64
    z = np.array([seed], dtype=u) * u(0x9E3779B97F4A7C15) + np.array([1], dtype=u) * u(0xD1B54A32D192ED03)
    z = z + np.arange(n, dtype=u)
    z = (z ^ (z >> u(30))) * u(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> u(27))) * u(0x94D049BB133111EB)
    return z ^ (z >> u(31))


@pytest.mark.parametrize("n,seed", [(400000, 7), (1000, 1)])
def test_pass_order_with_equal_upper_halves(n, seed):
    """400000 rows: some twenty pairs of keys share their upper 32 bits, which is all the sort compares; their order
    decides the order of the sums, so the parameters agree bit for bit only if it is that of the whole keys."""
    n_in, hid, batch = 3, 16, n // 4
    keys = _order_keys(seed, n)
    order = np.argsort(keys, kind="stable").astype(np.int32)
    up = keys[order] >> np.uint64(32)
    assert (np.count_nonzero(up[1:] == up[:-1]) > 0) == (n > 100000)
    rng = np.random.default_rng(n)
    X = torch.from_numpy(rng.standard_normal((n, n_in)).astype(np.float32)).to(DEV)
    T = torch.from_numpy(rng.standard_normal((n, 2)).astype(np.float32)).to(DEV)
    rows = torch.from_numpy(order).to(DEV)
    th = inputs.mlp_init(n_in, hid, 3).astype(np.float32)
    with gw.Mlp(n_in, hid, max_batch=batch, device=0) as a, gw.Mlp(n_in, hid, max_batch=batch, device=0) as b:
        a.set_params(th)
        b.set_params(th)
        a.train_corr(X, T, 1, batch, 1e-3, lr_final=1e-3, seed=seed, diag_repeat=1, diag_feature=-1)
        for t in range(4):
            b.train_step(X, T, rows[t * batch:(t + 1) * batch], 1e-3)
        assert np.array_equal(a.get_params(), b.get_params())


def test_two_networks_add_to_one_loss():
    """Two networks on streams of their own add their steps' losses to one accumulator."""
    n_in, hid, B, steps = 5, 33, 40, 300
    X, T, rows, th = _setup(n_in, hid, B)
    Xd, Td, rd = (torch.from_numpy(a).to(DEV) for a in (X, T, rows))
    loss = torch.zeros(1, dtype=torch.float32, device=DEV)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    nets = [gw.Mlp(n_in, hid, max_batch=B, device=0, stream=s) for s in streams]
    for net in nets:
        net.set_params(th)
    one = nets[0].grad(Xd, Td, rd)[1]
    for _ in range(steps):
        for net in nets:
            net.train_step(Xd, Td, rd, 1e-12, loss_accum=loss)   # the parameters stay where they are
    for net in nets:
        net.check()
        net.close()
    # FP32 sum of 2 steps terms of one sign
    assert abs(float(loss.item()) - 2 * steps * one) <= 2 * steps * 2.0 ** -24 * 2 * steps * one
