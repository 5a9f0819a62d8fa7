"""GPU parity of the hand-written adjoint (fptc_decode_backward) and of the
autograd wrapper against the FP64 oracle gradient, for the MSE loss to the
original signal.  The oracle gradient itself is pinned by central finite
differences in test_oracle_pipeline.py."""
import numpy as np
import pytest

import oracle
import siggen

from gpu_util import encode_workload, gpu_decode, make_plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRAD_COEFF_REL_L2 = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_01086_gb300 import build
    build()


def _signals_on_device(plan, wl):
    """Original signals laid out like the decoder output (0 in the gaps)."""
    x = torch.zeros(plan.info["out_extent"], dtype=torch.float32)
    for i in range(wl.n_streams):
        s = plan.segments[i]
        a = int(s["out_offset"])
        x[a:a + int(s["n_samples"])] = torch.from_numpy(siggen.signal(int(wl.domains[i]), int(wl.seeds[i]),
                                                                      int(wl.lengths[i])))
    return x.to(plan.device)


def _oracle_grads(plan, b, lv_h, gx_h, scale=None):
    n_dom = len(b.domains)
    gA = np.zeros((n_dom, 3))
    absA = np.zeros((n_dom, 3))
    gC = []
    for i in range(b.n_streams):
        d = b.domains[b.domain_idx[i]]
        if scale is not None:
            d = oracle.Domain(d.N, d.E, d.B1, d.B2, d.mu, d.alpha1, tuple(scale[b.domain_idx[i]]), d.lmax, d.code_len)
        S = int(b.lengths[i])
        L = d.windows(S) * d.E
        a = int(plan.level_offsets[i])
        o = int(plan.segments[i]["out_offset"])
        lv = lv_h[a:a + L]
        c, g = oracle.backward_stream(lv, S, d, gx_h[o:o + S])
        gA[b.domain_idx[i]] += g
        gC.append(c)
        # sum of |terms| bounds the rounding error of the FP32 products
        unit = np.array([[oracle.dequantize_unit(d, z, Lv) for Lv in range(256)] for z in (0, 1)])
        zones = np.array([d.zone(k) for k in range(d.E)])
        cc = c.reshape(-1, d.E)
        ll = lv.reshape(-1, d.E)
        for z in (0, 1):
            m = zones == z
            absA[b.domain_idx[i], z] += np.abs(cc[:, m] * unit[z][ll[:, m]]).sum()
    return gA, absA, gC


def _check(plan, b, gsc, gco, gA, absA, gC):
    g = gsc.cpu().numpy()
    # FP32 products g_C * unit: each term carries ~N+2 roundings of 2^-24; FP64 reduction
    tol = 1e-6 * np.abs(gA) + 40 * 2.0 ** -24 * absA
    assert np.all(np.abs(g - gA) <= tol), (g, gA, tol)
    if gco is not None:
        h = gco.cpu().numpy()
        for i, c in enumerate(gC):
            a = int(plan.level_offsets[i])
            seg = h[a:a + c.size].astype(np.float64)
            nr = np.linalg.norm(c)
            assert np.linalg.norm(seg - c) <= GRAD_COEFF_REL_L2 * max(nr, 1e-30), i


@pytest.mark.parametrize("name", ["power", "mixed"])
def test_backward_matches_oracle(name):
    wl = siggen.power_1024x65536(n=12, S=20000) if name == "power" else \
        siggen.mixed_10000_logu(n=16, lo=33, hi=60000)
    b = encode_workload(wl)
    plan = make_plan(b)
    w, s, out, lv = gpu_decode(plan, b)
    x = _signals_on_device(plan, wl)
    M = wl.n_samples
    gx = (2.0 / M) * (out - x)
    mask = torch.zeros_like(gx, dtype=torch.bool)
    for sg in plan.segments:
        mask[int(sg["out_offset"]):int(sg["out_offset"]) + int(sg["n_samples"])] = True
    gx = torch.where(mask, gx, torch.zeros_like(gx)).contiguous()
    gco = torch.empty(plan.info["n_levels_total"], dtype=torch.float32, device=plan.device)
    gsc, _ = plan.backward(gx, levels=lv, grad_coeffs=gco)
    # the same with the levels decoded again from the words
    gco2 = torch.empty_like(gco)
    gsc2, _ = plan.backward(gx, words=w, symlen=s, grad_coeffs=gco2)
    torch.cuda.synchronize()
    assert torch.equal(gco, gco2)
    assert torch.allclose(gsc, gsc2, rtol=1e-12, atol=0)
    gA, absA, gC = _oracle_grads(plan, b, lv.cpu().numpy(), gx.double().cpu().numpy())
    _check(plan, b, gsc, gco, gA, absA, gC)
    assert plan.device_status()[0] == 0


def test_autograd_function():
    from paper_2605_01086_gb300 import decode_differentiable
    wl = siggen.power_1024x65536(n=6, S=30000)
    b = encode_workload(wl)
    plan = make_plan(b)
    w, s = plan.to_device(b.words, b.symlen)
    x = _signals_on_device(plan, wl)
    base = np.array([d.A for d in b.domains])
    scale = torch.tensor(base * 1.1, dtype=torch.float64, device=plan.device, requires_grad=True)
    probe = torch.zeros(plan.info["n_levels_total"], device=plan.device, requires_grad=True)
    out = decode_differentiable(plan, w, s, scale, probe)
    n = int(plan.segments[-1]["out_offset"] + plan.segments[-1]["n_samples"])
    mask = torch.zeros(out.numel(), dtype=torch.bool, device=plan.device)
    for sg in plan.segments:
        mask[int(sg["out_offset"]):int(sg["out_offset"]) + int(sg["n_samples"])] = True
    loss = ((out - x)[mask] ** 2).mean()
    loss.backward()
    assert scale.grad is not None and probe.grad is not None
    # oracle with the same g_x
    gx = torch.where(mask, (2.0 / int(mask.sum())) * (out.detach() - x), torch.zeros_like(x))
    lv = torch.empty(plan.info["n_levels_total"], dtype=torch.uint8, device=plan.device)
    plan.decode(w, s, out=torch.empty_like(out), levels=lv)
    sc32 = (base * 1.1).astype(np.float32).astype(np.float64)
    gA, absA, gC = _oracle_grads(plan, b, lv.cpu().numpy(), gx.double().cpu().numpy(), scale=sc32)
    _check(plan, b, scale.grad, probe.grad, gA, absA, gC)
    assert n <= out.numel()


def test_backward_zone_switched_off():
    # A_1 = 0 at run time: zone 1 reconstructs 0 and has no gradient
    wl = siggen.power_1024x65536(n=3, S=5000)
    b = encode_workload(wl)
    plan = make_plan(b)
    w, s = plan.to_device(b.words, b.symlen)
    sc = torch.tensor(np.array([[d.A[0], 0.0, 0.0] for d in b.domains], np.float32).ravel(), device=plan.device)
    out = plan.decode(w, s, scale=sc)
    gx = torch.ones_like(out) * 1e-3
    gsc, _ = plan.backward(gx, words=w, symlen=s, scale=sc)
    torch.cuda.synchronize()
    g = gsc.cpu().numpy()
    assert np.all(g[:, 1] == 0.0) and np.all(g[:, 2] == 0.0) and np.any(g[:, 0] != 0.0)


@pytest.mark.parametrize("mode", ["levels", "redecode"])
def test_backward_other_shapes_matches_oracle(mode):
    """The adjoint on a plan of other window shapes (N = 64, 128, 16, 32 with E = N/2, N/2, N/2,
    N/4 in one batch; decoded by the shape kernel, differentiated by the block adjoint), from saved
    levels and decoding them again, against the oracle gradient."""
    shapes = [(64, 32), (128, 64), (16, 8), (32, 8)]
    doms = [oracle.trained_domain(i, N=N, E=E, B1=2, B2=E) for i, (N, E) in enumerate(shapes)]
    wl = siggen.mixed_10000_logu(n=12, lo=100, hi=40000)
    b = encode_workload(wl, domains=doms)
    plan = make_plan(b)
    assert plan.info["kernel"] == 3
    w, s, out, lv = gpu_decode(plan, b)
    x = _signals_on_device(plan, wl)
    gx = (2.0 / wl.n_samples) * (out - x)
    mask = torch.zeros_like(gx, dtype=torch.bool)
    for sg in plan.segments:
        mask[int(sg["out_offset"]):int(sg["out_offset"]) + int(sg["n_samples"])] = True
    gx = torch.where(mask, gx, torch.zeros_like(gx)).contiguous()
    gco = torch.empty(plan.info["n_levels_total"], dtype=torch.float32, device=plan.device)
    if mode == "levels":
        gsc, _ = plan.backward(gx, levels=lv, grad_coeffs=gco)
    else:
        gsc, _ = plan.backward(gx, words=w, symlen=s, grad_coeffs=gco)
    torch.cuda.synchronize()
    assert plan.device_status()[0] == 0
    gA, absA, gC = _oracle_grads(plan, b, lv.cpu().numpy(), gx.double().cpu().numpy())
    g = gsc.cpu().numpy()
    # FP32 products of up to N = 128 terms per coefficient, FP64 reduction
    tol = 1e-6 * np.abs(gA) + 136 * 2.0 ** -24 * absA
    assert np.all(np.abs(g - gA) <= tol), (g, gA, tol)
    h = gco.cpu().numpy()
    for i, c in enumerate(gC):
        a = int(plan.level_offsets[i])
        assert np.linalg.norm(h[a:a + c.size] - c) <= GRAD_COEFF_REL_L2 * max(np.linalg.norm(c), 1e-30), i


def test_backward_after_autotune():
    """The adjoint of a plan whose autotuner tried warp-tile candidates and may
    have settled on a block kernel (a single stream of 65,536 samples, where the
    block-tile kernel tends to win): the adjoint serves the configuration the
    autotuner left, and agrees with a plan configured once."""
    wl = siggen.Workload("one", 3, np.zeros(1, np.int32), np.array([siggen.stream_seed(3, 0)], np.uint64),
                         np.array([65536], np.uint64))
    b = encode_workload(wl)
    outs = []
    for tune in (True, False):
        plan = make_plan(b, out_align=32)
        w, s = plan.to_device(b.words, b.symlen)
        out = plan.empty_out().zero_()
        if tune:
            plan.autotune(w, s, out, trials=2)
        n_lev = plan.info["n_levels_total"]
        lv = torch.empty(n_lev, dtype=torch.uint8, device=plan.device)
        gco = torch.empty(n_lev, dtype=torch.float32, device=plan.device)
        plan.decode(w, s, out=out, levels=lv)
        gsc, _ = plan.backward(out, levels=lv, grad_coeffs=gco)
        torch.cuda.synchronize()
        assert plan.device_status()[0] == 0
        outs.append((gsc.cpu().numpy(), gco.cpu().numpy().astype(np.float64)))
    (g1, c1), (g2, c2) = outs
    np.testing.assert_allclose(g1, g2, rtol=1e-6, atol=1e-9)
    assert np.linalg.norm(c1 - c2) <= 1e-6 * np.linalg.norm(c2)


@pytest.mark.parametrize("N,E,B1,B2", [(4, 3, 1, 2), (5, 5, 2, 5), (16, 16, 2, 16), (24, 12, 0, 12), (33, 17, 2, 16),
                                       (64, 32, 2, 32), (64, 64, 5, 60), (100, 50, 2, 50), (127, 127, 2, 127),
                                       (128, 64, 2, 64)])
def test_backward_from_levels_any_shape(N, E, B1, B2):
    """The adjoint from saved levels for other shapes: streams that end anywhere in
    a group of windows, outputs and levels at any alignment, a domain with its
    first zone off, against the FP64 oracle.

    Bounds: dL/dC[k] of a window is a sum over n of g[n] B[k][n] by folding (one
    rounding), at most ceil(N / 2) / 2 + 2 multiply-adds in a row and one addition,
    with cosines off by 2^-25: within (N / 2 + 5) 2^-24 of S = sum |g[n]|.  dL/dA_z
    adds those times unit_z (at most 1) over the bins, unit_z rounded to 2^-24, the
    sum itself compensated: within sum (N / 2 + 5) 2^-24 S over the zone's bins, and
    2^-24 of sum |terms|."""
    from gpu_util import crafted_batch
    cl = np.full(256, 8, np.uint8)
    doms = [oracle.Domain(N, E, B1, B2, 30.0, 0.02, (0.0 if k else 3.0, 1.5, 0.0), 8, cl) for k in range(2)]
    rng = np.random.default_rng(N * 10 + E)
    lens = [1, N, 7 * N + 1, 16 * N, 33 * N + N // 2, 5000, 64 * N]
    idx = [i % 2 for i in range(len(lens))]
    levels = [rng.integers(0, 256, size=doms[j].windows(S) * E).astype(np.uint8) for S, j in zip(lens, idx)]
    b = crafted_batch(doms, levels, lens, idx)
    for align in (32, 1):
        plan = make_plan(b, out_align=align, out_base=0 if align == 32 else 3)
        _, _, out, lv = gpu_decode(plan, b)
        gx = torch.randn(plan.info["out_extent"], generator=torch.Generator().manual_seed(3)).to(plan.device)
        gco = torch.empty(plan.info["n_levels_total"], device=plan.device)
        gsc, _ = plan.backward(gx, levels=lv, grad_coeffs=gco)
        torch.cuda.synchronize()
        gh = gx.double().cpu().numpy()
        gA, absA, gC = _oracle_grads(plan, b, lv.cpu().numpy(), gh)
        got = gco.double().cpu().numpy()
        slack = 2.0 ** -24 * absA
        for i, S in enumerate(lens):
            a, o = int(plan.level_offsets[i]), int(plan.segments[i]["out_offset"])
            W = doms[idx[i]].windows(S)
            g = np.zeros(W * N)
            g[:S] = np.abs(gh[o:o + S])
            bound = (N / 2 + 5) * 2.0 ** -24 * g.reshape(W, N).sum(1)
            c = gC[i].reshape(W, E)
            assert np.all(np.abs(got[a:a + W * E].reshape(W, E) - c) <= bound[:, None]), i
            slack[idx[i], 0] += bound.sum() * B1
            slack[idx[i], 1] += bound.sum() * (B2 - B1)
        g = gsc.cpu().numpy()
        for d in range(2):
            for z in range(2):
                want = 0.0 if (z == 0 and d == 1) else gA[d, z]
                assert abs(g[d, z] - want) <= slack[d, z], (d, z, g[d, z], want)


def _two_routes(doms, lens, idx, seed, gx=None):
    """dL/dC and dL/dA from the saved levels and with the levels decoded again (the
    block kernel, where the domains are not N = 32, E = 16), and what they were made of."""
    from gpu_util import crafted_batch
    rng = np.random.default_rng(seed)
    levels = [rng.integers(0, 256, size=doms[j].windows(S) * doms[j].E).astype(np.uint8) for S, j in zip(lens, idx)]
    b = crafted_batch(doms, levels, lens, idx)
    plan = make_plan(b, out_align=4)
    w, s, _, lv = gpu_decode(plan, b)
    if gx is None:
        gx = torch.randn(plan.info["out_extent"], generator=torch.Generator().manual_seed(seed))
    gx = gx.to(plan.device)
    gco = torch.full((plan.info["n_levels_total"],), float("nan"), device=plan.device)
    gco2 = torch.full_like(gco, float("nan"))
    gsc, _ = plan.backward(gx, levels=lv, grad_coeffs=gco)
    gsc2, _ = plan.backward(gx, words=w, symlen=s, grad_coeffs=gco2)
    assert plan.device_status()[0] == 0
    return plan, gx.cpu().numpy(), gsc.cpu().numpy(), gco.cpu().numpy(), gsc2.cpu().numpy(), gco2.cpu().numpy()


@pytest.mark.parametrize("N,E", [(4, 4), (16, 8), (24, 12), (64, 64), (81, 41), (127, 64), (128, 128)])
@pytest.mark.parametrize("n", [1, 3, 12])
def test_backward_batch_sizes(N, E, n):
    """Batches of a few tiles (split into parts, most warps idle) and of more than the
    chip holds at once, of one domain, several (a CTA loads the tables of those its
    segments have) and more than the warp-tile kernel takes: both routes agree.

    Either route's coefficient is a sum of at most N products: within (N + 5) 2^-24
    of sum |g| of its window (|basis| <= 1), and the scale gradients within the sum
    of that over their bins (|unit| <= 1) and (4 + 2048) 2^-24 of the sum of
    |g_C unit| <= sum |g| E (the block kernel's partial sums are FP32 over at most
    2048 products a thread)."""
    cl = np.full(256, 8, np.uint8)
    doms = [oracle.Domain(N, E, min(2, E - 1), E - (d % 2), 30.0, 0.02, (3.0, 1.5, 0.0), 8, cl) for d in range(n)]
    for lens in ([1, N, 7 * N + 1, 16 * N, 33 * N + N // 2, 5000],
                 [30000 + 11 * i for i in range(max(n, 40))]):
        idx = [i % n for i in range(len(lens))] if len(lens) >= n else [(3 * i) % n for i in range(len(lens))]
        plan, g, sa, ca, sb, cb = _two_routes(doms, lens, idx, N + n)
        slack = np.zeros((n, 3))
        for i, S in enumerate(lens):
            a, o = int(plan.level_offsets[i]), int(plan.segments[i]["out_offset"])
            W = doms[idx[i]].windows(S)
            x = np.zeros(W * N)
            x[:S] = np.abs(g[o:o + S].astype(np.float64))
            x = x.reshape(W, N).sum(1)
            bound = 2 * (N + 5) * 2.0 ** -24 * x
            d = np.abs(ca[a:a + W * E].astype(np.float64) - cb[a:a + W * E]).reshape(W, E)
            assert np.all(d <= bound[:, None]), (i, d.max())  # a NaN is no bound's
            slack[idx[i]] += (bound.sum() + 2052 * 2.0 ** -24 * x.sum()) * E
        assert np.all(np.abs(sa - sb) <= slack)
        assert np.all(sa[np.unique(idx), 1] != 0)


@pytest.mark.parametrize("N,E,n", [(64, 64, 8), (128, 64, 4)])
def test_small_batches_of_many_domains_are_quick(N, E, n):
    """From saved levels a few short streams of several domains take no longer than
    with the levels decoded again, which is the same work and more (they took
    twice as long while every block loaded every domain's tables)."""
    from gpu_util import crafted_batch
    cl = np.full(256, 8, np.uint8)
    doms = [oracle.Domain(N, E, 2, E, 30.0, 0.02, (3.0, 1.5, 0.0), 8, cl) for _ in range(n)]
    lens = [5000] * n
    rng = np.random.default_rng(1)
    levels = [rng.integers(0, 256, size=doms[i].windows(S) * E).astype(np.uint8) for i, S in enumerate(lens)]
    b = crafted_batch(doms, levels, lens, list(range(n)))
    plan = make_plan(b)
    w, s, _, lv = gpu_decode(plan, b)
    g = torch.randn(plan.info["out_extent"], device=plan.device)
    gc = torch.empty(plan.info["n_levels_total"], device=plan.device)

    def quickest(call):
        times = []
        for _ in range(20):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call()
            z.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(z))
        return min(times)

    saved = quickest(lambda: plan.backward(g, levels=lv, grad_coeffs=gc))
    again = quickest(lambda: plan.backward(g, words=w, symlen=s, grad_coeffs=gc))
    assert saved <= 1.2 * again, (saved, again)


@pytest.mark.parametrize("N,E", [(64, 32), (24, 12), (81, 41), (5, 5), (127, 127)])
def test_backward_infinite_and_nan_gradients(N, E):
    """Infinities and NaN in the incoming gradient (either half of a window, both
    mirrored samples, the middle one of an odd N): dL/dC and dL/dA are infinite, of
    the same sign, and NaN where the block kernel's sums are."""
    cl = np.full(256, 8, np.uint8)
    inf, nan = float("inf"), float("nan")
    places = [[(0, inf)], [(N - 1, -inf)], [(N // 2, inf)], [((N - 1) // 2, nan)], [(1, inf), (N - 2, inf)],
              [(1, inf), (N - 2, -inf)], [(2, nan)], [(N // 2 + 1, -inf)], []]
    doms = [oracle.Domain(N, E, 1, E, 30.0, 0.02, (3.0, 1.5, 0.0), 8, cl) for _ in range(len(places))]
    lens = [40 * N] * len(places)
    off = np.zeros(len(places) + 1, np.int64)
    off[1:] = np.cumsum([-(-S // 4) * 4 for S in lens])
    gx = torch.randn(int(off[-1]), generator=torch.Generator().manual_seed(N))
    for i, at in enumerate(places):
        for n, v in at:
            gx[off[i] + 17 * N + n] = v
    plan, _, sa, ca, sb, cb = _two_routes(doms, lens, list(range(len(places))), N, gx)
    assert [int(x["out_offset"]) for x in plan.segments] == list(off[:-1])
    assert np.isinf(sb[:, 0]).any() and np.isnan(sb).any() and np.isfinite(sb[-1]).all()
    for a, b in ((ca, cb), (sa, sb)):
        np.testing.assert_array_equal(np.isnan(a), np.isnan(b))
        np.testing.assert_array_equal(np.where(np.isinf(a), a, 0.0), np.where(np.isinf(b), b, 0.0))
