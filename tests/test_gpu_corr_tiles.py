"""gw_corr_apply and gw_corr_features over 32 x 32 tiles of P~: orders around one and two tiles, with and without the
closure estimate, an odd offset of the feature buffer; and the weight ratio with fewer states than threads."""
import numpy as np
import pytest

from paper_1810_07772_gb300 import gw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("ng", [2, 31, 32, 33, 64, 95])
@pytest.mark.parametrize("with_clos", [False, True])
def test_apply(ng, with_clos):
    rng = np.random.default_rng(ng)
    P = (rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))).astype(np.complex64)
    C = (rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))).astype(np.complex64)
    Y = rng.standard_normal((ng * (ng + 1) // 2, 2)).astype(np.float32)
    scale = np.float32(1.7)
    got = torch.from_numpy(P.copy()).to(DEV)
    gw.corr_apply(got, torch.from_numpy(Y).to(DEV), torch.tensor([scale], device=DEV),
                  torch.from_numpy(C).to(DEV) if with_clos else None)
    ref = P.astype(np.complex128)
    g, h = np.triu_indices(ng)
    d = (Y[:, 0] + 1j * Y[:, 1]).astype(np.complex128) / scale + (C[g, h] if with_clos else 0)
    d = np.where(g == h, d.real, d)
    keep = g > 0
    g, h, d = g[keep], h[keep], d[keep]
    ref[g, h] += d
    off = g != h
    ref[h[off], g[off]] += d[off].conj()
    # two FP32 additions of values below 10
    assert np.max(np.abs(got.cpu().numpy() - ref)) <= 4e-6


@pytest.mark.parametrize("offset", [0, 1])
def test_features_on_unaligned_buffers(offset):
    ng = 33
    rng = np.random.default_rng(5)
    P = (rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))).astype(np.complex64)
    gv = rng.integers(-3, 4, (ng, 3)).astype(np.int32)
    ratio = torch.tensor([0.3], device=DEV)
    Pd, gd = torch.from_numpy(P).to(DEV), torch.from_numpy(gv).to(DEV)
    X, _ = gw.corr_features(Pd, gd, 9, ratio)
    buf, scale = torch.zeros(X.numel() + 4, device=DEV), torch.empty(1, device=DEV)
    st = gw.lib().gw_corr_features(Pd.data_ptr(), ng, gd.data_ptr(), 9, ratio.data_ptr(), None,
                                   buf.data_ptr() + 4 * offset, scale.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
    assert st == gw.GW_OK
    assert torch.equal(buf[offset:offset + X.numel()].view_as(X), X)


@pytest.mark.parametrize("nv,keep,nc", [(1, 1, 2), (3, 5, 9), (7, 300, 5000)])
def test_weight_ratio(nv, keep, nc):
    rng = np.random.default_rng(nc)
    E = np.concatenate([-1 - rng.random(nv), 1 + 5 * rng.random(nc)])
    w = 2.0 / (E[None, nv:] - E[:nv, None])
    ref = w[:, keep:].sum() / w[:, :keep].sum()
    r = torch.empty(1, device=DEV)
    Ed = torch.from_numpy(E).to(DEV)
    assert gw.lib().gw_corr_weight_ratio(Ed.data_ptr(), nv, keep, nc, r.data_ptr(),
                                         torch.cuda.current_stream().cuda_stream) == gw.GW_OK
    assert abs(r.item() - ref) <= 2e-7 * ref      # rounded to FP32 once
