"""The separable form of the 16-bit rank-k update (gw_build_P where T (nv + nc) states are fewer than
nv nc pairs) against the FP64 sum of Eq. (Pstatic), at the edges of its tiles and chunks.

Bars as in test_gpu_parity: FP16X3 1e-6 relative at the default window, 2e-6 at any window; BF16X3
1e-5 (the 8 + 8-bit split: 4.5e-6 measured in the pair form, which the separable form must not exceed by
more than its spread)."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_1810_07772_gb300 import gw, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def build(dims, nv, nc, psi, E, prec="fp16x3", window=None, kind="single", by_pairs=False):
    nr = int(np.prod(dims))
    with gw.Context(0) as ctx:
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).cuda(), E, dims, nv)
        ctx.set_herk_kernel(kind, by_pairs)
        if window:
            ctx.set_herk_window(*window)
        P = torch.empty((nr, nr), dtype=torch.complex64, device="cuda:0")
        ctx.build_P(prec, P_out=P)
        ctx.sync()
        return P, ctx.update_form()


# exact multiples of 128 rows and 16 states; one state beyond a chunk on both sides; ragged rows with
# a 1-row last block; several occupied chunks; fewer tiles than SMs and more
CASES = [((8, 8, 8), 16, 208, 1), ((7, 9, 11), 33, 97, 2), ((3, 11, 27), 33, 160, 3), ((9, 10, 11), 70, 81, 4),
         ((16, 16, 13), 24, 200, 5)]


@pytest.mark.parametrize("dims,nv,nc,seed", CASES)
@pytest.mark.parametrize("window", [None, (1, 1), (5, 256), (6, 256), (64, 4096)])
def test_matches_fp64(dims, nv, nc, seed, window):
    psi, E = inputs.make_states(0, nv, nc, seed, dims=dims)
    P, form = build(dims, nv, nc, psi, E, window=window)
    assert form["terms"] > 1 and form["chunks"] == form["terms"] * (-(-nv // 16) + -(-nc // 16))
    ref = O.P_rspace(psi, E, nv)
    P = P.cpu().numpy()
    assert rel(P, ref) <= (1e-6 if window is None else 2e-6)
    assert np.array_equal(P, P.conj().T) and not np.diag(P).imag.any()


@pytest.mark.parametrize("window", [None, (16, 256)])
def test_bf16(window):
    dims, nv, nc = (7, 9, 11), 33, 97
    psi, E = inputs.make_states(0, nv, nc, 2, dims=dims)
    P, form = build(dims, nv, nc, psi, E, "bf16x3", window)
    assert form["terms"] > 1 and rel(P.cpu().numpy(), O.P_rspace(psi, E, nv)) <= 1e-5


def test_energies_in_any_order_and_degenerate():
    """Unsorted energies and shells of equal ones; the states' amplitudes differ by orders of magnitude
    (unnormalised input), which the per-set power-of-two scales must carry."""
    dims, nv, nc = (7, 9, 11), 20, 110
    rng = np.random.default_rng(9)
    psi, _ = inputs.make_states(0, nv, nc, 6, dims=dims)
    psi = psi * np.concatenate([np.full(nv, 1e-7), np.full(nc, 300.0)])[:, None]
    E = np.concatenate([np.round(rng.uniform(-8, 0, nv)), 0.5 + np.round(rng.uniform(0, 12, nc))])
    P, form = build(dims, nv, nc, psi, E)
    assert form["terms"] > 1 and rel(P.cpu().numpy(), O.P_rspace(psi, E, nv)) <= 1e-6


@pytest.mark.parametrize("prec,bar", [("fp16x3", 1e-6), ("bf16x3", 1e-5)])
@pytest.mark.parametrize("ev,ec", [(60, -60), (-60, 60), (-100, 100), (100, -100), (30, 30), (-20, -30), (0, 55), (-55, 0)])
def test_states_of_any_scale(prec, bar, ev, ec):
    """Occupied states times 2^ev, unoccupied ones times 2^ec: P is 2^(2 ev + 2 ec) times that of the unit states,
    an FP32 value, and only powers of two change on the way."""
    dims, nv, nc = (7, 9, 11), 20, 110
    psi, E = inputs.make_states(0, nv, nc, 6, dims=dims)
    scale = np.concatenate([np.full(nv, 2.0 ** ev), np.full(nc, 2.0 ** ec)])[:, None]
    P, form = build(dims, nv, nc, psi.astype(np.complex64).astype(np.complex128) * scale, E, prec)
    assert form["terms"] > 1
    P = P.cpu().numpy().astype(np.complex128) * 2.0 ** (-2 * ev - 2 * ec)
    assert rel(P, O.P_rspace(psi, E, nv)) <= bar


def _smooth_states(kind, dims, nv, nc, seed):
    """(psi complex64 on the device, E): Haar-random, band-structured or plane waves in order of |m|."""
    if kind == "haar":
        psi, E = inputs.make_states(0, nv, nc, seed, dims=dims)
        return torch.from_numpy(psi.astype(np.complex64)).cuda(), E
    if kind == "bands":
        coef, gvec, E = inputs.make_states_g_structured_device(dims, nv, nc, seed, "cuda:0")
        with gw.Context(0) as ctx:
            ctx.load_states_g(coef, gvec, E, dims, nv)
            return ctx.view("psiT").t().contiguous(), E
    m = np.stack(np.meshgrid(*[np.arange(-(d // 2) + 1, d // 2) for d in dims], indexing="ij"), -1).reshape(-1, 3)
    m2 = (m ** 2).sum(1)
    order = np.argsort(m2, kind="stable")[:nv + nc]
    m, m2 = m[order], m2[order].astype(float)
    E = np.concatenate([-10 + 9 * m2[:nv] / m2[nv - 1], 0.5 + 19.5 * (m2[nv:] - m2[nv]) / (m2[-1] - m2[nv])])
    x = [np.exp(2j * np.pi * np.outer(m[:, a], np.arange(d)) / d) for a, d in enumerate(dims)]
    psi = np.einsum("pa,pb,pc->pabc", *x).reshape(nv + nc, -1) / np.sqrt(np.prod(dims))
    return torch.from_numpy(psi.astype(np.complex64)).cuda(), E


@pytest.mark.parametrize("kind,dims,nv,nc", [("haar", (12, 12, 12), 40, 1600), ("bands", (14, 14, 14), 16, 1040),
                                             ("plane", (16, 16, 16), 19, 600)])
@pytest.mark.parametrize("prec", ["fp16x3", "bf16x3"])
def test_no_less_precise_than_by_pairs(kind, dims, nv, nc, prec):
    """Windows up to 64 chunks that are really that long, and smooth states, whose sums near the diagonal have
    terms of one sign: the whole of P, its diagonal, its elements next to it and the far ones, against an
    FP64 sum, beside the pair form's errors at the same window.  The whole within 5 % of the pair form's
    (rounding of the last bit); a class of elements within a quarter of the larger of its own and the
    whole's (the loss that is added back is a mean over states)."""
    psi, E = _smooth_states(kind, dims, nv, nc, 3)
    p64, Eh = psi.to(torch.complex128), torch.from_numpy(E / 27.211386245988).cuda()
    ref = 0.0
    for v in range(nv):
        f = p64[v].conj()[None, :] * p64[nv:]
        ref = ref - (f * (2.0 / (Eh[nv:] - Eh[v]))[:, None]).t() @ f.conj()
    x = torch.from_numpy(np.stack(np.unravel_index(np.arange(int(np.prod(dims))), dims), -1)).cuda()
    d2 = 0
    for a, n in enumerate(dims):
        q = (x[:, None, a] - x[None, :, a]).abs()
        d2 = d2 + torch.minimum(q, n - q) ** 2
    classes = [d2 >= 0, d2 == 0, d2 == 1, (d2 >= 2) & (d2 <= 9), d2 > 9]

    def errors(ctx, by_pairs):
        ctx.set_herk_kernel("single", by_pairs)
        ctx.build_P(prec)
        ctx.sync()
        assert (ctx.update_form()["terms"] > 0) == (not by_pairs)
        P = ctx.view("P").to(torch.complex128)
        return [float((P[k] - ref[k]).norm() / ref[k].norm()) for k in classes]

    with gw.Context(0) as ctx:
        ctx.load_states(psi, E, dims, nv)
        for W in (2, 3, 16, 64):
            ctx.set_herk_window(W, 256)
            sep, pair = errors(ctx, False), errors(ctx, True)
            assert sep[0] <= 1.05 * pair[0], (W, sep, pair)
            for s, p in zip(sep[1:], pair[1:]):
                assert s <= 1.25 * max(p, pair[0]), (W, sep, pair)


def test_by_pairs():
    """GW_HERK_BY_PAIRS takes the other kernel: FP32 sums of the same numbers in another order, each within
    1e-6 of FP64; the factors are there after the separable form only, and a bad value is refused."""
    dims, nv, nc = (8, 8, 8), 16, 208
    psi, E = inputs.make_states(0, nv, nc, 1, dims=dims)
    a, fa = build(dims, nv, nc, psi, E)
    b, fb = build(dims, nv, nc, psi, E, by_pairs=True)
    assert fa["terms"] > 1 and fb == {"terms": 0, "chunks": nv * nc // 16}
    assert not torch.equal(a, b) and rel(a.cpu().numpy(), b.cpu().numpy()) <= 2e-6
    with gw.Context(0) as ctx:
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).cuda(), E, dims, nv)
        ctx.build_P("fp16x3")
        ctx.set_herk_kernel("single", by_pairs=True)
        assert ctx.update_form()["terms"] == fa["terms"]  # the form of the last update, not of the next
        ctx.build_P("fp16x3")
        assert ctx.update_form()["terms"] == 0
        with pytest.raises(gw.GwError) as e:
            ctx.set_herk_kernel(4)
        assert e.value.status == gw.GW_E_INVALID


@pytest.mark.parametrize("kind,npl", [("single", 4), ("pair", 6)])
def test_kernel_setting_and_pair_densities_afterwards(kind, npl):
    """GW_HERK_PAIR leaves the kernel of the separable form as it is (128 x 128 tiles are reported); GW_BUF_F
    still holds the pair densities, in the layout of the setting, when it is asked for."""
    from test_gpu_parity import _decode_16
    dims, nv, nc = (8, 8, 8), 16, 208
    psi, E = inputs.make_states(0, nv, nc, 1, dims=dims)
    with gw.Context(0) as ctx:
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).cuda(), E, dims, nv)
        ctx.set_herk_kernel(kind)
        ctx.build_P("fp16x3")
        assert ctx.update_form()["terms"] > 1 and ctx.stats()["herk_tiles"] == 10
        ptr, nbytes = ctx.buffer("F")
        torch.cuda.synchronize()
        F = torch.as_tensor(gw.DeviceView(ptr, (nbytes,), "|u1"), device="cuda:0").cpu().numpy()
        e = int(ctx.stats()["fp16_scale_exp"])
        f, _ = _decode_16(F, ctx.dims8()[7], 512, nv * nc, bf16=False, npl=npl)
    assert rel(f / 2.0 ** e, O.pair_density(psi, E, nv).T) < 1e-6


@pytest.mark.parametrize("by_pairs", [False, True])
def test_pair_densities_after_another_operand_found_no_room(by_pairs):
    """A TF32 build that runs out of memory leaves the earlier P; GW_BUF_F then holds that update's operand, padded
    to 16 pairs (8021 pairs: 8032, where the TF32 operand has 8024)."""
    from test_gpu_parity import _decode_16
    dims, nv, nc = (16, 16, 16), 13, 617
    psi, E = inputs.make_states(16, nv, nc, 3)
    with gw.Context(0) as ctx:
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).cuda(), E, dims, nv)
        ctx.set_herk_kernel("single", by_pairs)
        ctx.build_P("fp16x3")
        ctx.sync()
        P = ctx.view("P").clone()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        # 400 MB are left, with the operand that the pair form holds
        left = (400 << 20) - (ctx.buffer("F")[1] if by_pairs else 0)
        fill = torch.empty(torch.cuda.mem_get_info(0)[0] - left, dtype=torch.uint8, device="cuda:0")
        with pytest.raises(gw.GwError) as e:
            ctx.build_P("tf32x3")                # 526 MB; the 16-bit operand takes 263
        assert e.value.status == gw.GW_E_NOMEM
        ptr, nbytes = ctx.buffer("F")
        torch.cuda.synchronize()
        assert nbytes == 8032 * 4096 * 8
        del fill
        torch.cuda.empty_cache()
        assert torch.equal(ctx.view("P"), P)
        F = torch.as_tensor(gw.DeviceView(ptr, (nbytes,), "|u1"), device="cuda:0").cpu().numpy()
        e = int(ctx.stats()["fp16_scale_exp"])
        f, _ = _decode_16(F, 4096, 4096, nv * nc, bf16=False)
    assert rel(f / 2.0 ** e, O.pair_density(psi, E, nv).T) < 1e-6


def test_update_after_a_larger_grid_found_no_room():
    """P(r,r') of 58^3 points (305 GB) finds no room, and the earlier buffer is gone; a smaller grid leaves one too
    small for the first states, which are then loaded again: the update goes to the buffer that is there."""
    systems = {n: inputs.make_states(n, nv, nc, 7) for n, nv, nc in ((16, 24, 200), (8, 2, 3))}
    with gw.Context(0) as ctx:
        def build(n, nv, precision):
            psi, E = systems[n]
            ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).cuda(), E, (n, n, n), nv)
            ctx.build_P(precision)
            ctx.sync()
            return ctx.view("P").clone()

        first = build(16, 24, "fp16x3")
        assert ctx.buffer("factors")[1] > 0
        ctx.load_states(torch.zeros(2, 58 ** 3, dtype=torch.complex64, device="cuda:0"), np.array([-1.0, 1.0]), (58,) * 3, 1)
        with pytest.raises(gw.GwError) as e:
            ctx.build_P("fp32_simt")
        assert e.value.status == gw.GW_E_NOMEM
        build(8, 2, "fp32_simt")
        assert torch.equal(build(16, 24, "fp16x3"), first)


def test_batch_of_both_forms_equals_single_instances():
    """One launch over a separable, a pair-form and another separable instance, replayed from the graph
    and after a change of window: bit for bit the single-instance P~."""
    systems = [((9, 10, 11), 24, 200, 5, 71), ((8, 10, 12), 3, 30, 6, 73), ((12, 12, 12), 33, 97, 8, 72)]
    loaded = []
    for dims, nv, nc, gcut, seed in systems:
        psi, E = inputs.make_states(0, nv, nc, seed, dims=dims)
        loaded.append((torch.from_numpy(psi.astype(np.complex64)).cuda(), E))

    def single(W):
        out = []
        for (dims, nv, nc, gcut, _), (psi, E) in zip(systems, loaded):
            with gw.Context(0) as ctx:
                ctx.load_states(psi, E, dims, nv)
                ctx.set_herk_window(W, 256)
                ctx.build_P("fp16x3")
                form = ctx.update_form()["terms"]
                ctx.P_to_G(gcut)
                out.append((ctx.view("PG").clone(), form))
        return out

    ctxs = []
    for (dims, nv, nc, gcut, _), (psi, E) in zip(systems, loaded):
        ctx = gw.Context(0)
        ctx.load_states(psi, E, dims, nv)
        ctxs.append(ctx)
    with gw.Batch(ctxs, [s[3] for s in systems]) as b:
        for W in (2, 7):
            b.set_window(W, 256)
            ref = single(W)
            assert [f > 0 for _, f in ref] == [True, False, True]
            for _ in range(3):
                b.run(use_graph=True)
                for c, (PG, _) in zip(ctxs, ref):
                    assert torch.equal(c.view("PG"), PG)
    for c in ctxs:
        c.close()


def test_batch_set_up_behind_queued_work():
    """Contexts on a stream of their own with work queued on it: the factors are there when the autotuner starts
    on the batch's stream."""
    dims, nv, nc, gcut = (9, 10, 11), 24, 200, 5
    loaded = [inputs.make_states(0, nv, nc, seed, dims=dims) for seed in (81, 82)]
    s = torch.cuda.Stream()
    refs, ctxs = [], []
    for psi, E in loaded:
        refs.append(build(dims, nv, nc, psi, E, window=(2, 256))[0])
        ctx = gw.Context(0, stream=s)
        ctx.load_states(torch.from_numpy(psi.astype(np.complex64)).cuda(), E, dims, nv)
        ctxs.append(ctx)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(200_000_000)     # about 0.1 s
    with gw.Batch(ctxs, [gcut] * 2) as b:
        b.autotune(target_error=1e-3)
        got = [c.view("P").clone() for c in ctxs]
    for P, ref in zip(got, refs):
        assert rel(P.cpu().numpy(), ref.cpu().numpy()) <= 1e-4
    for c in ctxs:
        c.close()


def test_batch_after_reloading_its_contexts():
    """Other states and energies of the same shape (graph captured before), then another shape, then a context
    used by itself with another cut and a wider operand: the next passes equal fresh single instances."""
    def single(dims, nv, psi, E, gcut):
        with gw.Context(0) as ctx:
            ctx.load_states(psi, E, dims, nv)
            ctx.set_herk_window(2, 256)
            ctx.build_P("fp16x3")
            ctx.P_to_G(gcut)
            return ctx.view("PG").clone()

    def states(dims, nv, nc, seed, gap):
        psi, E = inputs.make_states(0, nv, nc, seed, dims=dims)
        E = np.concatenate([E[:nv], E[nv:] + gap])
        return torch.from_numpy(psi.astype(np.complex64)).cuda(), E

    gcut = 5
    shapes = [((9, 10, 11), 24, 200), ((8, 10, 12), 3, 30)]
    loads = [[states(*sh, 90 + i + 10 * q, gap) for i, sh in enumerate(shapes)] for q, gap in ((0, 0.0), (1, 7.0))]
    ctxs = [gw.Context(0) for _ in shapes]
    for c, sh, (psi, E) in zip(ctxs, shapes, loads[0]):
        c.load_states(psi, E, sh[0], sh[1])
    with gw.Batch(ctxs, [gcut] * 2) as b:
        b.set_window(2, 256)

        def check(data, shp):
            for _ in range(3):
                b.run(use_graph=True)
                for c, sh, (psi, E) in zip(ctxs, shp, data):
                    assert torch.equal(c.view("PG"), single(sh[0], sh[1], psi, E, gcut))

        check(loads[0], shapes)
        for c, sh, (psi, E) in zip(ctxs, shapes, loads[1]):
            c.load_states(psi, E, sh[0], sh[1])
        check(loads[1], shapes)
        other = ((12, 12, 12), 33, 97)
        data = [states(*other, 120, 1.0), loads[1][1]]
        ctxs[0].load_states(*data[0], other[0], other[1])
        check(data, [other, shapes[1]])
        ctxs[1].build_P("tf32x3")
        ctxs[1].P_to_G(3)
        check(data, [other, shapes[1]])
    for c in ctxs:
        c.close()


def test_form_follows_the_window():
    """42 x 42 states: separable with windows of three chunks, by pairs with one (three windows a term cost more
    than the pairs save); a batch changes over with its window, bit for bit as a single instance."""
    dims, nv, nc, gcut = (8, 9, 8), 42, 42, 5
    psi, E = inputs.make_states(0, nv, nc, 4, dims=dims)
    psi = torch.from_numpy(psi.astype(np.complex64)).cuda()
    want = {}
    with gw.Context(0) as ctx:
        ctx.load_states(psi, E, dims, nv)
        for W in (1, 3):
            ctx.set_herk_window(W, 256)
            ctx.build_P("fp16x3")
            assert (ctx.update_form()["terms"] > 0) == (W == 3)
            ctx.P_to_G(gcut)
            want[W] = ctx.view("PG").clone()
        with gw.Batch([ctx], [gcut]) as b:
            for W in (3, 1, 3):
                b.set_window(W, 256)
                for _ in range(3):
                    b.run(use_graph=True)
                    assert torch.equal(ctx.view("PG"), want[W])


def test_captured_update_follows_later_loads():
    """gw_build_P and gw_P_to_G captured on a caller's stream: each replay takes the states and energies loaded
    last, with fewer or more terms than at the capture, as a fresh context gives them; the third set's energies
    crowd at the gap, so that a fresh context takes it pair by pair and the replay with all 16 terms."""
    dims, nv, nc, gcut = (8, 8, 8), 16, 208, 5
    nr = 512
    loads = []
    for seed, gap, power in ((1, 0.5, 1), (2, 30.0, 1), (3, 1e-3, 4), (1, 0.5, 1)):
        psi, _ = inputs.make_states(0, nv, nc, seed, dims=dims)
        E = np.concatenate([-10 * np.linspace(0, 1, nv) ** power, gap + 20 * np.linspace(0, 1, nc) ** power])
        loads.append((torch.from_numpy(psi.astype(np.complex64)).cuda(), E))
    want, terms = [], []
    for psi, E in loads:
        with gw.Context(0) as ctx:
            ctx.load_states(psi, E, dims, nv)
            ctx.build_P("fp16x3")
            terms.append(ctx.update_form()["terms"])
            ctx.P_to_G(gcut)
            want.append((ctx.view("P").clone(), ctx.view("PG").clone()))
    assert 0 < terms[1] < terms[0] and terms[2] == 0
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        ctx = gw.Context(0, stream=s)
        ctx.load_states(*loads[0], dims, nv)
        ctx.build_P("fp16x3")
        g = ctx.P_to_G(gcut)
        ctx.sync()
        P = torch.empty((nr, nr), dtype=torch.complex64, device="cuda:0")
        PG = torch.empty((len(g), len(g)), dtype=torch.complex64, device="cuda:0")
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        graph.capture_begin()
        ctx.build_P("fp16x3", P_out=P)
        ctx.P_to_G(gcut, PG_out=PG)
        graph.capture_end()
        for (psi, E), (Pw, PGw) in zip(loads, want):
            ctx.load_states(psi, E, dims, nv)
            graph.replay()
            s.synchronize()
            ctx.sync()
            if E[nv] < 0.01:
                assert rel(P.cpu().numpy(), Pw.cpu().numpy()) <= 2e-6
                assert rel(PG.cpu().numpy(), PGw.cpu().numpy()) <= 2e-6
            else:
                assert torch.equal(P, Pw) and torch.equal(PG, PGw)
        # energies without factors (weights beyond the range of FP32 scales): the replay says so, once
        ctx.load_states(loads[0][0], loads[0][1] * 1e-45, dims, nv)
        graph.replay()
        with pytest.raises(gw.GwError) as e:
            ctx.sync()
        assert e.value.status == gw.GW_E_INVALID and "separable" in str(e.value)
        ctx.load_states(*loads[-1], dims, nv)
        graph.replay()
        ctx.sync()
        assert torch.equal(P, want[-1][0])
        ctx.build_P("fp16x3")                     # and the calls by themselves as before
        assert ctx.update_form()["terms"] == terms[-1] and torch.equal(ctx.view("P"), want[-1][0])
        ctx.close()
