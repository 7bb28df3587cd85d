"""Measured cases: what a user of the library has it do, through its public entry points.

Each case is one pass of a program that keeps its context (and network, batch or matrix) and calls
the library again with the inputs it holds on the device: states and energies for every new
q-point, system or training pass.  The kinds are

* ``rspace``   states -> P(r,r') -> P~(G,G') -> eps^-1: the path of the paper, from latency-bound
               systems to the 36^3 split-precision workload;
* ``gspace``   the same result without P(r,r') (Eq. gpsaceP);
* ``ksum``     a sum over k-points from plane-wave coefficients;
* ``batch``    independent systems of uneven size in one pass;
* ``learned``  the truncated sum plus closure estimate and network, to eps^-1;
* ``infer``, ``train``  the correction network by itself, forward and Adam steps;
* ``zinv``     the tensor-core inverse of a Hermitian positive definite matrix.

Inputs have the distributions of ``inputs.py``: orthonormal complex states (Haar-random, or
energy-ordered plane-wave shells for the learned form) and uniform sorted energies.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1810_07772_gb300 import gw, inputs

HARTREE_EV = 27.211386245988
DEV = "cuda:0"


def _gcut(n):
    """The sphere cut of the repository's workloads: about 5 % of the grid points."""
    return int((n / 4.4) ** 2)


def _system(name, kind, dims, nv, nc, method="newton_tc", precision="fp16x3", target=0.0, gcut=None, **more):
    c = dict(kind=kind, n1=dims[0], n2=dims[1], n3=dims[2], nv=nv, nc=nc,
             gcut=_gcut(min(dims)) if gcut is None else gcut, method=method, precision=precision, target=target, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the small FP64-checkable system (12^3): latency and launches count
        _system("rspace_12", "rspace", (12, 12, 12), 4, 28, gcut=8),
        # a small cell that is not cubic, with an odd axis and an odd number of pairs
        _system("rspace_15x18x20", "rspace", (15, 18, 20), 11, 151),
        # the plain workload: 24^3, 32 occupied and 480 unoccupied states
        _system("rspace_24", "rspace", (24, 24, 24), 32, 480, gcut=29),
        # the split-precision workload: 36^3, BF16 hi + lo operands under its 1e-4 error target
        _system("split_36", "rspace", (36, 36, 36), 64, 1000, gcut=61, precision="bf16x3", target=1e-4),
        # the plain workload by the route that never forms P(r,r')
        _system("gspace_24", "gspace", (24, 24, 24), 32, 480, gcut=29),
        # odd axes without a compiled transform, and the FP64 Cholesky inverse
        _system("gspace_22x25x23_cholesky", "gspace", (22, 25, 23), 13, 170, method="cholesky"),
        # two k-points from a DFT code's plane-wave coefficients, weights 1/2
        _system("ksum_20", "ksum", (20, 20, 20), 16, 200, nk=2, gcut_psi=81),
        # the eight-system batch: grids 16^3 .. 32^3, 8 .. 48 occupied, 100 .. 800 unoccupied
        dict(name="batch_8", kind="batch", grids="16,18,20,24,24,27,30,32", nvs="8,14,19,25,31,37,42,48",
             ncs="100,200,300,400,500,600,700,800"),
        # the learned workload: 200 of 2000 unoccupied states kept, closure estimate and network
        _system("learned_24", "learned", (24, 24, 24), 32, 200, gcut=29, nc_all=2000),
        # the network over the entries of one 24^3 system, and one pass of training over 131,072 rows
        dict(name="infer_239086", kind="infer", rows=239086),
        dict(name="train_131072", kind="train", rows=131072, batch=8192),
        # the inverse alone at the order of the batch's seventh system (odd)
        dict(name="zinv_1357", kind="zinv", n=1357),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rspace", "rspace", "rspace", "gspace", "gspace", "ksum", "batch", "learned", "infer", "train",
                       "zinv"])
    if kind in ("rspace", "gspace", "ksum"):
        cube = rng.random() < 0.5
        n = rng.randint(10, 32)
        dims = (n, n, n) if cube else tuple(min(32, max(10, n + rng.randint(-4, 4))) for _ in range(3))
        nv, nc = _log_int(rng, 2, 48), _log_int(rng, 10, 800)
        method = "cholesky" if rng.random() < 0.2 else "newton_tc"
        if kind == "rspace":
            bf16 = rng.random() < 0.25
            return _system(None, kind, dims, nv, nc, method, "bf16x3" if bf16 else "fp16x3", 1e-4 if bf16 else 0.0)
        if kind == "ksum":
            dims = tuple(min(24, d) for d in dims)
            gpsi = int((0.45 * min(dims)) ** 2)
            npw = len(inputs.psi_sphere(dims, gpsi))
            nc = max(1, min(nc, 300, npw - nv))
            return _system(None, kind, dims, nv, nc, method, nk=rng.randint(2, 4), gcut_psi=gpsi)
        nc = min(nc, 500)
        return _system(None, kind, dims, nv, nc, method)
    if kind == "batch":
        m = rng.randint(2, 6)
        grids = sorted(rng.randint(10, 27) for _ in range(m))
        return dict(kind=kind, grids=",".join(map(str, grids)),
                    nvs=",".join(str(_log_int(rng, 4, 40)) for _ in range(m)),
                    ncs=",".join(str(_log_int(rng, 30, 500)) for _ in range(m)))
    if kind == "learned":
        n = rng.randint(16, 24)
        keep = _log_int(rng, 60, 250)
        return _system(None, kind, (n, n, n), rng.randint(8, 32), keep, nc_all=4 * keep)
    if kind == "infer":
        return dict(kind=kind, rows=_log_int(rng, 200, 2000000))
    if kind == "train":
        batch = rng.choice([1024, 2048, 4096, 8192])
        return dict(kind=kind, rows=batch * rng.randint(6, 20) + rng.randint(0, batch - 1), batch=batch)
    return dict(kind=kind, n=_log_int(rng, 60, 2007))


# ----------------------------------------------------------------------------- inputs


def _dims(case):
    return (case["n1"], case["n2"], case["n3"])


def _orthonormal(rows, cols, seed):
    """[cols][rows] complex64: Haar-random orthonormal vectors (the QR of a complex Gaussian)."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    a = torch.randn((rows, cols), dtype=torch.complex64, device=DEV, generator=gen)
    q, _ = torch.linalg.qr(a, mode="reduced")
    return q.transpose(0, 1).contiguous()


def _energies(nv, nc, seed):
    rng = np.random.default_rng(int(seed))
    return np.concatenate([np.sort(rng.uniform(-10.0, 0.0, nv)), np.sort(rng.uniform(0.5, 20.0, nc))])


def _states(dims, nv, nc, seed):
    return _orthonormal(dims[0] * dims[1] * dims[2], nv + nc, seed), _energies(nv, nc, seed + 7919)


def _batch_systems(case):
    grids, nvs, ncs = ([int(x) for x in case[k].split(",")] for k in ("grids", "nvs", "ncs"))
    return list(zip(grids, nvs, ncs))


def _theta(seed):
    """Network parameters with the small last layer of a trained one (what the closure estimate leaves
    is a few per cent of P~)."""
    th = inputs.mlp_init(gw.N_FEATURES, 256, seed)
    th[-2 * 256 - 2:-2] *= 2e-3
    return th


def _samples(case, seed):
    """Features and targets of the training and inference cases: values of the sizes that
    gw_corr_features gives, a diagonal flag in one row of 345, targets a smooth function of them."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    n = case["rows"]
    X = torch.randn((n, gw.N_FEATURES), device=DEV, generator=gen)
    X[:, :3] = X[:, :3].abs()
    X[:, 7] = (torch.rand(n, device=DEV, generator=gen) < 1.0 / 345).float()
    X[:, 8] = 2.5
    X[:, 9] = 0.0
    T = torch.stack([torch.sin(X[:, 3]) * X[:, 10] - 0.5 * X[:, 7], torch.tanh(X[:, 4] * X[:, 0]) - X[:, 11]], dim=1)
    return X.contiguous(), T.contiguous()


def _hpd(n, seed):
    """I + B B^H with the spread of a dielectric matrix (condition number about 4) and a diagonal
    that varies by a factor of two."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    k = max(1, n // 2)
    B = torch.randn((n, k), dtype=torch.complex128, device=DEV, generator=gen) / math.sqrt(k)
    d = 1.0 + 0.4 * torch.rand(n, dtype=torch.float64, device=DEV, generator=gen)
    A = torch.eye(n, dtype=torch.complex128, device=DEV) + 0.5 * (B @ B.conj().t())
    A = d[:, None] * A * d[None, :]
    return (0.5 * (A + A.conj().t())).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "infer":
        net = gw.Mlp(gw.N_FEATURES, 256, max_batch=8192)
        net.set_params(inputs.mlp_init(gw.N_FEATURES, 256, seed))
        return dict(case=case, net=net, X=_samples(case, seed)[0])
    if kind == "train":
        net = gw.Mlp(gw.N_FEATURES, 256, max_batch=case["batch"])
        X, T = _samples(case, seed)
        theta = torch.from_numpy(inputs.mlp_init(gw.N_FEATURES, 256, seed)).to(DEV)
        return dict(case=case, net=net, X=X, T=T, theta=theta, seed=int(seed))
    if kind == "zinv":
        A = _hpd(case["n"], seed)
        return dict(case=case, ctx=gw.Context(0), A=A, X=torch.empty_like(A))
    if kind == "batch":
        ctxs, gcuts = [], []
        for i, (n, nv, nc) in enumerate(_batch_systems(case)):
            psi, E = _states((n, n, n), nv, nc, 1000 * seed + i)
            ctx = gw.Context(0)
            ctx.load_states(psi, E, (n, n, n), nv)
            ctxs.append(ctx)
            gcuts.append(_gcut(n))
        b = gw.Batch(ctxs, gcuts, "fp16x3")
        b.set_window(3, 256)
        return dict(case=case, batch=b, ctxs=ctxs)
    dims, nv, nc = _dims(case), case["nv"], case["nc"]
    ctx = gw.Context(0)
    s = dict(case=case, ctx=ctx)
    if kind == "ksum":
        s["gvec"] = inputs.psi_sphere(dims, case["gcut_psi"])
        s["k"] = [(_orthonormal(len(s["gvec"]), nv + nc, 1000 * seed + i), _energies(nv, nc, 1000 * seed + i + 7919))
                  for i in range(case["nk"])]
    elif kind == "learned":
        coef, gvec, E = inputs.make_states_g_structured_device(dims, nv, case["nc_all"], seed, DEV)
        ctx.load_states_g(coef[:nv + nc].contiguous(), gvec, E[:nv + nc], dims, nv)
        s["psi"], s["E"] = ctx.view("psiT").t().contiguous(), E
        s["net"] = gw.Mlp(gw.N_FEATURES, 256, max_batch=8192)
        s["net"].set_params(_theta(seed))
    else:
        s["psi"], s["E"] = _states(dims, nv, nc, seed)
    ng = len(inputs.psi_sphere(dims, case["gcut"]))
    s["PG"] = torch.empty((ng, ng), dtype=torch.complex64, device=DEV)
    s["inv"] = torch.empty((ng, ng), dtype=torch.complex128, device=DEV)
    if kind == "learned":
        s["clos"] = torch.empty((ng, ng), dtype=torch.complex64, device=DEV)
    ctx.set_error_target(case["target"])
    return s


# ----------------------------------------------------------------------------- one pass


def _view(ctx, which):
    """The context's own buffer as a tensor that keeps the context: a caller may drop the state first."""
    t = ctx.view(which)
    t.owner = ctx
    return t


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "infer":
        return {"Y": s["net"].infer(s["X"])}
    if kind == "train":
        net = s["net"]
        net.set_params(s["theta"])
        losses = net.train_corr(s["X"], s["T"], 1, case["batch"], 1e-3, seed=s["seed"], diag_repeat=4)
        return {"losses": np.array(losses), "theta": net.get_params()}
    if kind == "zinv":
        return {"X": s["ctx"].zinv_tc(s["A"], s["X"])}
    if kind == "batch":
        s["batch"].run(use_graph=True)
        return {which: [_view(c, which) for c in s["ctxs"]] for which in ("PG", "epsinv")}
    ctx, dims, nv, gcut = s["ctx"], _dims(case), case["nv"], case["gcut"]
    if kind == "rspace":
        ctx.load_states(s["psi"], s["E"], dims, nv)
        ctx.build_P(case["precision"])
        ctx.P_to_G(gcut, PG_out=s["PG"])
        ctx.eps_inv(case["method"], epsinv_out=s["inv"])
        return {"P": _view(ctx, "P"), "PG": s["PG"], "epsinv": s["inv"]}
    if kind == "gspace":
        ctx.load_states(s["psi"], s["E"], dims, nv)
        ctx.build_PG(gcut, case["precision"], PG_out=s["PG"])
        ctx.eps_inv(case["method"], epsinv_out=s["inv"])
        return {"PG": s["PG"], "epsinv": s["inv"]}
    if kind == "ksum":
        for i, (coef, E) in enumerate(s["k"]):
            ctx.load_states_g(coef, s["gvec"], E, dims, nv)
            ctx.set_kweight(1.0 / case["nk"], accumulate=i > 0)
            ctx.build_PG(gcut, case["precision"], PG_out=s["PG"])
        ctx.eps_inv(case["method"], epsinv_out=s["inv"])
        return {"PG": s["PG"], "epsinv": s["inv"]}
    # learned: kept states -> truncated P~, closure estimate, network, eps^-1
    nb = nv + case["nc"]
    ctx.load_states(s["psi"], s["E"][:nb], dims, nv)
    g = ctx.build_PG(gcut, case["precision"])
    PG = _view(ctx, "PG")
    ctx.corr_closure(gcut, s["E"][nb:], out=s["clos"])
    ratio = gw.corr_weight_ratio(s["E"], nv, case["nc"])
    X, scale = gw.corr_features(PG, g, gcut, ratio, s["clos"])
    gw.corr_apply(PG, s["net"].infer(X), scale, s["clos"])
    ctx.eps_inv(case["method"], epsinv_out=s["inv"])
    return {"PG": PG, "clos": s["clos"], "epsinv": s["inv"]}


# ----------------------------------------------------------------------------- what a pass needs


def _nsphere(dims, gcut):
    m = [np.arange(-(n // 2), n - n // 2) ** 2 for n in dims]
    return int(np.count_nonzero(m[0][:, None, None] + m[1][None, :, None] + m[2][None, None, :] <= gcut))


def _rank(nv, nc):
    """Rank that the update of P cannot do without: every pair, or, since the energy denominators
    2 / (E_c - E_v) separate into about a dozen products to FP32 accuracy, a dozen times the states."""
    return min(nv * nc, 12 * (nv + nc))


def _work_system(route, dims, nv, nc, gcut):
    nr, ng, nb, k = dims[0] * dims[1] * dims[2], _nsphere(dims, gcut), nv + nc, nv * nc
    byt = nb * nr * 8.0 + ng * ng * 24.0
    flop = 8.0 * ng ** 3
    if route == "rspace":
        byt += 2 * 8.0 * nr * nr
        flop += 4.0 * _rank(nv, nc) * nr * (nr + 1.0)
    else:
        byt += k * ng * 8.0
        flop += 4.0 * k * ng * (ng + 1.0) + 8.0 * k * nr
    return byt, flop


def work(case):
    kind = case["kind"]
    if kind in ("infer", "train"):
        n = case["rows"]
        fwd = 2.0 * (12 * 256 + 2 * 256 * 256 + 256 * 2)
        return {"bytes": n * 56.0, "flops": n * fwd * (1 if kind == "infer" else 3)}
    if kind == "zinv":
        n = case["n"]
        return {"bytes": 32.0 * n * n, "flops": 8.0 * n ** 3}
    if kind == "batch":
        ws = [_work_system("rspace", (n, n, n), nv, nc, _gcut(n)) for n, nv, nc in _batch_systems(case)]
    else:
        ws = [_work_system(kind, _dims(case), case["nv"], case["nc"], case["gcut"])] * case.get("nk", 1)
    return {"bytes": sum(w[0] for w in ws), "flops": sum(w[1] for w in ws)}


def tolerance(case):
    """About four times what is measured against 64 bits."""
    kind = case["kind"]
    if kind == "infer":
        return {"rel": 1e-3, "max": 0.02}       # FP16 activations, hardware tanh: 2.7e-4
    if kind == "train":
        return {"rel": 2e-5, "max": 0.05}       # FP32 sums through 16 Adam steps: 4e-6, more where a gradient is near 0
    if kind == "zinv":
        return {"rel": 1e-12}                   # 1.4e-13
    if kind == "learned" or case.get("precision") == "bf16x3":
        return {"rel": 2e-5}                    # the network's FP16 activations: 4.6e-6; BF16 hi + lo: 4.8e-6
    return {"rel": 3e-6}                        # FP32 sums of FP16 hi + lo products: 6.6e-7


# ----------------------------------------------------------------------------- the same in 64 bits


def _miller(dims, gcut):
    """The library's sphere: |m|^2 <= gcut ordered by (|m|^2, m1, m2, m3)."""
    g = inputs.psi_sphere(dims, gcut).astype(np.int64)
    m2 = (g * g).sum(axis=1)
    return g[np.lexsort((g[:, 2], g[:, 1], g[:, 0], m2))]


def _flat(dims, m):
    m = np.asarray(m)
    return torch.from_numpy(((m[..., 0] % dims[0]) * dims[1] + m[..., 1] % dims[1]) * dims[2] + m[..., 2] % dims[2]).to(DEV)


def _pair_transforms(psi, v, first, last, idx, dims):
    f = psi[v].conj()[None, :] * psi[first:last]
    return torch.fft.fftn(f.reshape(-1, *dims), dim=(1, 2, 3)).reshape(last - first, -1)[:, idx]


def _pg_exact(psi64, E, nv, dims, gcut):
    psi = psi64.to(torch.complex128)
    idx = _flat(dims, _miller(dims, gcut))
    Eh = torch.from_numpy(np.asarray(E) / HARTREE_EV).to(DEV)
    ng = idx.numel()
    out = torch.zeros((ng, ng), dtype=torch.complex128, device=DEV)
    for v in range(nv):
        M = _pair_transforms(psi, v, nv, psi.shape[0], idx, dims)
        w = 2.0 / (Eh[nv:] - Eh[v])
        out -= (M * w[:, None]).t() @ M.conj()
    return out


def _p_exact(psi64, E, nv):
    """P(r,r') where the direct sum takes a few seconds at FP64 rates, else None."""
    nb, nr = psi64.shape
    if 8.0 * nv * (nb - nv) * nr * nr > 3e12:
        return None
    psi = psi64.to(torch.complex128)
    Eh = torch.from_numpy(np.asarray(E) / HARTREE_EV).to(DEV)
    out = torch.zeros((nr, nr), dtype=torch.complex128, device=DEV)
    for v in range(nv):
        f = psi[v].conj()[None, :] * psi[nv:]
        out -= (f * (2.0 / (Eh[nv:] - Eh[v]))[:, None]).t() @ f.conj()
    return out


def _eps_inv_exact(PG, dims, gcut):
    m2 = torch.from_numpy((_miller(dims, gcut) ** 2).sum(axis=1)).to(DEV).double()
    sv = torch.where(m2 > 0, torch.sqrt(4 * math.pi / ((2 * math.pi) ** 2 * m2.clamp(min=1.0))), torch.zeros_like(m2))
    eps = torch.eye(len(sv), dtype=torch.complex128, device=DEV) - sv[:, None] * PG * sv[None, :]
    return torch.linalg.inv(eps)


def _closure_exact(psi64, E, nv, E_omit, dims, gcut):
    psi = psi64.to(torch.complex128)
    nb, nr = psi.shape
    g = _miller(dims, gcut)
    W = torch.from_numpy((2.0 / ((E[:nv, None] - E_omit[None, :]) / HARTREE_EV)).sum(axis=1)).to(DEV)
    rho = torch.fft.fftn((W[:, None] * psi[:nv].abs() ** 2).sum(0).reshape(dims).to(torch.complex128)).reshape(-1)
    out = rho[_flat(dims, g[:, None, :] - g[None, :, :])]
    idx = _flat(dims, g)
    for v in range(nv):
        M = _pair_transforms(psi, v, 0, nb, idx, dims)
        out = out - W[v] * (M.t() @ M.conj())
    return out / (nr - nb)


def _layers(theta, half):
    """[(W, b)] from the flat vector, the weights rounded to FP16 as the network multiplies them."""
    sizes, out, o = [(256, gw.N_FEATURES), (256, 256), (256, 256), (2, 256)], [], 0
    for r, c in sizes:
        W = theta[o:o + r * c].reshape(r, c)
        out.append((W.half().double() if half else W, theta[o + r * c:o + r * c + r]))
        o += r * c + r
    return out


def _net_exact(theta, X):
    a = X.double()
    layers = _layers(theta.double(), True)
    for W, b in layers[:-1]:
        a = torch.tanh(a @ W.t() + b)
    return a @ layers[-1][0].t() + layers[-1][1]


def _learned_exact(s):
    case = s["case"]
    dims, nv, keep, gcut, E = _dims(case), case["nv"], case["nc"], case["gcut"], s["E"]
    PG = _pg_exact(s["psi"], E[:nv + keep], nv, dims, gcut)
    clos = _closure_exact(s["psi"], E, nv, E[nv + keep:], dims, gcut)
    g = torch.from_numpy(_miller(dims, gcut)).to(DEV).double()
    ng = len(g)
    gi, hi = torch.triu_indices(ng, ng, device=DEV)
    diag = PG.diagonal().real
    sc = 1.0 / diag[1:].abs().mean()
    w = 2.0 / (E[None, nv:] - E[:nv, None])
    ratio = float(w[:, keep:].sum() / w[:, :keep].sum())
    m2, dm = (g * g).sum(1), g[gi] - g[hi]
    p, c = PG[gi, hi], clos[gi, hi]
    head = (gi == 0) | (hi == 0)
    X = torch.stack([m2[gi] / gcut, m2[hi] / gcut, (dm * dm).sum(1) / (4.0 * gcut), sc * p.real, sc * p.imag,
                     sc * diag[gi], sc * diag[hi], (gi == hi).double(), torch.full_like(m2[gi], ratio), head.double(),
                     sc * c.real, sc * c.imag], dim=1)
    Y = _net_exact(torch.from_numpy(s["net"].get_params()).to(DEV), X)
    d = torch.complex(Y[:, 0], Y[:, 1]) / sc + c
    d = torch.where(gi == hi, d.real.to(d.dtype), d)
    d = torch.where(head, torch.zeros_like(d), d)
    D = torch.zeros_like(PG)
    D[hi, gi] = d.conj()
    D[gi, hi] = d
    PG = PG + D
    return {"PG": PG, "clos": clos, "epsinv": _eps_inv_exact(PG, dims, gcut)}


def _order(seed, n):
    """Minibatch order of the first training pass: the pool sorted by SplitMix64-mixed keys."""
    u = np.uint64
    z = np.array([seed], dtype=u) * u(0x9E3779B97F4A7C15) + np.array([1], dtype=u) * u(0xD1B54A32D192ED03)
    z = z + np.arange(n, dtype=u)
    z = (z ^ (z >> u(30))) * u(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> u(27))) * u(0x94D049BB133111EB)
    return np.argsort(z ^ (z >> u(31)), kind="stable")


def _train_exact(s):
    X, T = s["X"].double(), s["T"].double()
    theta, batch = s["theta"].double(), s["case"]["batch"]
    pool = np.arange(X.shape[0])
    pool = np.concatenate([pool] + [np.flatnonzero((s["X"][:, 7] == 1).cpu().numpy())] * 3)
    order = torch.from_numpy(pool[_order(s["seed"], len(pool))]).to(DEV)
    steps = len(pool) // batch
    m, v, total = torch.zeros_like(theta), torch.zeros_like(theta), 0.0
    for t in range(steps):
        rows = order[t * batch:(t + 1) * batch]
        layers, acts = _layers(theta, True), [X[rows]]
        for W, b in layers[:-1]:
            acts.append(torch.tanh(acts[-1] @ W.t() + b))
        r = acts[-1] @ layers[-1][0].t() + layers[-1][1] - T[rows]
        total += 0.5 * float((r * r).sum()) / batch
        delta, grads = r / batch, []
        for i in range(3, -1, -1):
            grads = [(delta.t() @ acts[i]).reshape(-1), delta.sum(0)] + grads
            if i:
                delta = (delta @ layers[i][0]) * (1.0 - acts[i] ** 2)
        g = torch.cat(grads)
        lr = 1e-5 + 0.5 * (1e-3 - 1e-5) * (1.0 + math.cos(math.pi * t / steps))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        theta = theta - lr * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
    return {"losses": np.array([total / steps]), "theta": theta}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = {"PG": [], "epsinv": []}
        for i, (n, nv, nc) in enumerate(_batch_systems(case)):
            psi, E = _states((n, n, n), nv, nc, 1000 * seed + i)
            PG = _pg_exact(psi, E, nv, (n, n, n), _gcut(n))
            out["PG"].append(PG)
            out["epsinv"].append(_eps_inv_exact(PG, (n, n, n), _gcut(n)))
        return out
    s = prepare(case, seed)
    if kind == "infer":
        return {"Y": _net_exact(torch.from_numpy(s["net"].get_params()).to(DEV), s["X"])}
    if kind == "train":
        return _train_exact(s)
    if kind == "zinv":
        return {"X": torch.linalg.inv(s["A"])}
    if kind == "learned":
        return _learned_exact(s)
    dims, nv, gcut = _dims(case), case["nv"], case["gcut"]
    if kind == "ksum":
        PG = 0.0
        idx = _flat(dims, s["gvec"])
        for coef, E in s["k"]:
            box = torch.zeros((coef.shape[0], dims[0] * dims[1] * dims[2]), dtype=torch.complex128, device=DEV)
            box[:, idx] = coef.to(torch.complex128)
            psi = torch.fft.ifftn(box.reshape(-1, *dims), dim=(1, 2, 3)).reshape(coef.shape[0], -1)
            psi = psi * math.sqrt(dims[0] * dims[1] * dims[2])
            PG = PG + _pg_exact(psi, E, nv, dims, gcut) / case["nk"]
        return {"PG": PG, "epsinv": _eps_inv_exact(PG, dims, gcut)}
    PG = _pg_exact(s["psi"], s["E"], nv, dims, gcut)
    out = {"PG": PG, "epsinv": _eps_inv_exact(PG, dims, gcut)}
    if kind == "rspace":
        out["P"] = _p_exact(s["psi"], s["E"], nv)
    return out
