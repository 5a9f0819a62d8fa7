"""GPU parity of the warp-tile kernel for window shapes other than N = 32,
E = 16 (any N in [4, 128] for every domain of a plan, power-of-two or not,
several N in one batch, any E <= N per domain; Table 1 ranges), and of the
tensor-core transform for the shapes with E >= 32: levels bit-exact and samples within the
FP32 bound against the FP64 oracle, for random levels over every bin, ragged
lengths (partial windows, partial tiles, partial output steps), outputs at
128-byte boundaries (TMA stores) and at odd offsets (per-lane stores), several
kept-bin counts and window sizes in one batch, trained tables on synthetic signals, and tiles
chained across a segment the index rejects."""
import numpy as np
import pytest

import oracle
import siggen

from gpu_util import FP32_REL_L2, compare_with_oracle, crafted_batch, encode_workload, gpu_decode, make_plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WARP_TILE = 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_01086_gb300 import build
    build()


def _random_batch(N, Es, seed, lens_of=None):
    """Uniform 8-bit codes (every level a codeword), random levels; per domain
    (same N, kept bins Es[d]) streams of ragged lengths."""
    cl = np.full(256, 8, np.uint8)
    doms = [oracle.Domain(N, E, min(2, E), max(1, E - (d % 2)), 30.0 + d, 0.02, (3.0 + d, 1.0 + 0.5 * d, 0.0), 8, cl)
            for d, E in enumerate(Es)]
    rng = np.random.default_rng(seed)
    lens, dom_idx, levels = [], [], []
    for d, dom in enumerate(doms):
        T = min(2048 // dom.E, 8192 // N)
        base = lens_of(N, T) if lens_of else [1, N - 1, N, N + 1, 1024 + 5, T * N, T * N + 3, 3 * T * N - N // 2,
                                               40000 + 17 * d]
        for S in base:
            lens.append(S)
            dom_idx.append(d)
            levels.append(rng.integers(0, 256, size=dom.windows(S) * dom.E).astype(np.uint8))
    return crafted_batch(doms, levels, lens, dom_idx)


@pytest.mark.parametrize("N,Es", [(4, [1]), (4, [3, 4]), (8, [8]), (8, [3, 6]), (16, [8, 16]), (16, [5]),
                                  (32, [8]), (32, [32, 12]), (64, [16, 32]), (64, [7]), (128, [32, 64]),
                                  (128, [128, 1]),
                                  # window sizes that are not a power of two (run-time-N transform)
                                  (5, [5]), (6, [3, 6]), (12, [5]), (24, [12, 24]), (48, [24, 7]), (100, [50, 33]),
                                  (127, [64, 127])])
@pytest.mark.parametrize("align", [32, 1])
def test_shape_random_levels(N, Es, align):
    b = _random_batch(N, Es, seed=N * 100 + sum(Es) + align)
    plan = make_plan(b, out_align=align, out_base=0 if align == 32 else 3, kernel="warp_tile")
    assert plan.info["kernel"] == WARP_TILE
    _, _, out, lv = gpu_decode(plan, b, out_fill=float("nan"))
    compare_with_oracle(plan, b, out, lv)
    # nothing outside the segments is written
    h = out.cpu().numpy()
    mask = np.ones(h.size, bool)
    for sg in plan.segments:
        mask[int(sg["out_offset"]):int(sg["out_offset"]) + int(sg["n_samples"])] = False
    assert np.all(np.isnan(h[mask]))
    assert plan.device_status()[0] == 0


@pytest.mark.parametrize("threads", [256, 512, 768])
def test_shape_thread_counts(threads):
    b = _random_batch(64, [32, 16], seed=7)
    plan = make_plan(b, out_align=32, kernel="warp_tile", threads=threads)
    assert plan.info["threads"] == threads
    _, _, out, lv = gpu_decode(plan, b)
    compare_with_oracle(plan, b, out, lv)


@pytest.mark.parametrize("N,Es", [(64, [32, 7]), (24, [12, 5]), (128, [128, 64])])
def test_shape_tuned_and_three_kernel(N, Es):
    """A tuned plan's options make a plan again, and the three-kernel schedule's tiles
    (several of the shape kernel's steps) cover ragged streams: both within the
    bounds of every other plan."""
    from paper_2605_01086_gb300.tune_cache import plan_kwargs
    b = _random_batch(N, Es, seed=11)
    plan = make_plan(b, out_align=32)
    w, s = plan.to_device(b.words, b.symlen)
    best, _ = plan.autotune(w, s, plan.empty_out(), trials=1)
    for p in (plan, make_plan(b, out_align=32, **plan_kwargs(best)),
              make_plan(b, out_align=32, schedule="three_kernel")):
        _, _, out, lv = gpu_decode(p, b)
        compare_with_oracle(p, b, out, lv)


def test_shape_default_choice():
    """Plans whose domains all have a power-of-two N get the warp-tile kernel by
    default, several N in one plan included, window sizes that are not a power
    of two too."""
    b = _random_batch(16, [8], seed=3)
    assert make_plan(b).info["kernel"] == WARP_TILE
    cl = np.full(256, 8, np.uint8)
    for n2, want in ((64, WARP_TILE), (24, WARP_TILE), (100, WARP_TILE)):
        doms = [oracle.Domain(16, 8, 2, 8, 30.0, 0.02, (3.0, 1.0, 0.0), 8, cl),
                oracle.Domain(n2, 8, 2, 8, 30.0, 0.02, (3.0, 1.0, 0.0), 8, cl)]
        lv = [np.full(d.windows(1000) * d.E, 128, np.uint8) for d in doms]
        assert make_plan(crafted_batch(doms, lv, [1000, 1000], [0, 1])).info["kernel"] == want


@pytest.mark.parametrize("align", [32, 1])
def test_shape_mixed_window_sizes(align):
    """Domains of N = 4, 16, 32 (E = 16 and E = 8), 64, 128, 24 and 100 in one batch,
    streams interleaved in the output: each tile takes its domain's transform."""
    cl = np.full(256, 8, np.uint8)
    shapes = [(4, 4, 1, 3), (16, 8, 2, 8), (32, 16, 2, 16), (32, 8, 2, 6), (64, 24, 3, 20), (128, 64, 2, 64),
              (24, 12, 2, 12), (100, 50, 2, 40)]
    doms = [oracle.Domain(N, E, B1, B2, 25.0 + i, 0.03, (2.0 + i, 1.0 + 0.25 * i, 0.0), 8, cl)
            for i, (N, E, B1, B2) in enumerate(shapes)]
    rng = np.random.default_rng(99 + align)
    lens, idx, levels = [], [], []
    for r in range(5):
        for d, dom in enumerate(doms):
            S = int(rng.integers(1, 60000)) if r else dom.N * 300 + d
            lens.append(S)
            idx.append(d)
            levels.append(rng.integers(0, 256, size=dom.windows(S) * dom.E).astype(np.uint8))
    b = crafted_batch(doms, levels, lens, idx)
    plan = make_plan(b, out_align=align, out_base=0 if align == 32 else 1)
    assert plan.info["kernel"] == WARP_TILE
    _, _, out, lv = gpu_decode(plan, b)
    compare_with_oracle(plan, b, out, lv)
    assert plan.device_status()[0] == 0


@pytest.mark.parametrize("N,E", [(64, 32), (16, 8), (128, 64)])
def test_shape_trained_signals(N, E):
    """Tables trained on the synthetic domains at another shape, signals of all four domains."""
    doms = [oracle.trained_domain(i, N=N, E=E, B1=2, B2=E) for i in range(4)]
    wl = siggen.mixed_10000_logu(n=24, lo=100, hi=200000)
    b = encode_workload(wl, domains=doms)
    plan = make_plan(b, out_align=32)
    assert plan.info["kernel"] == WARP_TILE
    _, _, out, lv = gpu_decode(plan, b)
    compare_with_oracle(plan, b, out, lv)


def test_shape_chain_across_rejected_segment():
    """Several tiles per warp, a segment with a wrong symbol count in between:
    it is flagged and skipped, the others decode exactly."""
    from paper_2605_01086_gb300 import _lib
    b = _random_batch(64, [32], seed=11, lens_of=lambda N, T: [T * N * 62 + 5] * 40)
    bad = 17
    b.symlen[int(b.word_off[bad]) + 9] -= 1
    plan = make_plan(b, out_align=32, kernel="warp_tile", threads=256, ctas_per_sm=1)
    assert plan.info["n_tiles"] >= 2 * plan.info["grid"] * 8
    w, s = plan.to_device(b.words, b.symlen)
    out = plan.empty_out().fill_(float("nan"))
    lv = torch.empty(plan.info["n_levels_total"], dtype=torch.uint8, device=plan.device)
    plan.decode(w, s, out=out, levels=lv)
    st, flags, first = plan.device_status()
    assert st == _lib.CORRUPT_STREAM and flags & _lib.FLAG_SYMBOL_COUNT and first == bad
    compare_with_oracle(plan, b, out, lv, idx=[i for i in range(b.n_streams) if i != bad])


TC_TOL = {"tf32": 1e-3, "bf16x3": 2e-5, "tf32x3": 1e-5}  # as for N = 32, E = 16 (tests/test_gpu_tc.py)


@pytest.mark.parametrize("mode", ["tf32", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("N,E", [(32, 32), (64, 32), (128, 32), (128, 64)])
@pytest.mark.parametrize("align", ["window", "odd"])
def test_tensor_core_shapes(N, E, mode, align):
    """The tensor-core transform for shapes with E >= 32 (decode_tcs.cu): two
    domains of the same (N, E) with different scales and zone bounds (one with a
    zone-2 bin), ragged lengths; outputs on window boundaries (3-D TMA stores of
    whole steps) and at odd offsets (lane stores); levels bit-exact, samples
    within the form's bound, nothing written outside the segments."""
    b = _random_batch(N, [E, E], seed=N * 7 + E + len(mode))
    plan = make_plan(b, out_align=N if align == "window" else 1, out_base=0 if align == "window" else 3, idct=mode)
    assert plan.info["kernel"] == 4
    _, _, out, lv = gpu_decode(plan, b, out_fill=float("nan"))
    # TF32 bounds each sample's error by ~2^-10 sum_k |C_k B_kn|, not by the sample: a
    # stream of a few samples whose sums cancel can exceed the stream-level bound
    short = np.flatnonzero(b.lengths < 1024)
    longer = np.flatnonzero(b.lengths >= 1024)
    worst = compare_with_oracle(plan, b, out, lv, idx=longer, tol=TC_TOL[mode])
    compare_with_oracle(plan, b, out, lv, idx=short, tol=TC_TOL[mode] * (50 if mode == "tf32" else 1))
    h = out.cpu().numpy()
    mask = np.ones(h.size, bool)
    for sg in plan.segments:
        mask[int(sg["out_offset"]):int(sg["out_offset"]) + int(sg["n_samples"])] = False
    assert np.all(np.isnan(h[mask]))
    assert plan.device_status()[0] == 0
    print(N, E, mode, align, "worst rel L2", worst)


def test_tensor_core_shape_trained_signals():
    """(64, 32) on trained tables and EEG-like signals, against the FP32 kernel's output too."""
    wl = siggen.Workload("tcs", 11, np.zeros(6, np.int32),
                         np.array([siggen.stream_seed(11, i) for i in range(6)], np.uint64),
                         np.array([64 * 1000 + 3, 65536, 1, 200000, 64 * 64, 12345], np.uint64))
    ts = siggen.training_set(0)
    flat, offs = siggen.signals(ts.domains, ts.seeds, ts.lengths)
    dom = oracle.train_domain(flat, offs, ts.lengths, oracle.Domain(64, 32, 2, 32, 50.0, 0.004, (0.0, 0.0, 0.0), 12),
                              99.9)
    b = encode_workload(wl, domains=[dom])
    plan = make_plan(b, out_align=64, idct="tf32x3")
    assert plan.info["kernel"] == 4
    _, _, out, lv = gpu_decode(plan, b, out_fill=0.0)   # the gaps between segments compare equal
    compare_with_oracle(plan, b, out, lv, tol=TC_TOL["tf32x3"])
    ref = make_plan(b, out_align=64, kernel="warp_tile")
    _, _, out32, _ = gpu_decode(ref, b, out_fill=0.0)
    rel = float(torch.linalg.vector_norm((out - out32).double()) / torch.linalg.vector_norm(out32.double()))
    assert rel < 1e-6


@pytest.mark.parametrize("N,E,B1", [(16, 4, 0), (16, 5, 5), (32, 9, 3), (32, 32, 2), (64, 16, 2), (64, 17, 1),
                                    (64, 33, 4), (64, 64, 2), (128, 32, 0), (128, 33, 2), (128, 64, 3),
                                    (128, 65, 2)])
@pytest.mark.parametrize("align", [32, 4])
def test_shape_transform_forms(N, E, B1, align):
    """Bin counts on both sides of where the compiled transforms change, first
    zones other than Table 1's, streams that end inside an output step and whose
    outputs start at any chunk of a window row of the output.

    Bound: a sample is a sum over the bins of c_k cos(.), |c_k| <= A_z <= 2.  A
    coefficient carries the roundings of unit_z and of A_z unit_z, its cosine one
    of half that size, and the sum at most E / 2 multiply-adds in a row and one
    addition per halving of N (7 at most): within (2 + 1 + E / 2 + 7) 2^-24 of
    sum |c_k| <= 2 E.  (Streams of one sample are among them: relative to the
    sample itself there is no bound.)"""
    cl = np.full(256, 8, np.uint8)
    doms = [oracle.Domain(N, E, B1, E, 40.0, 0.01, (2.0, 1.5, 0.0), 8, cl),
            oracle.Domain(32, 16, 2, 16, 50.0, 0.004, (1.0, 1.0, 0.0), 8, cl)]
    rng = np.random.default_rng(N * 1000 + E)
    lens, idx, levels = [], [], []
    for S in [1, N, 32 * N, 32 * N + 33, 64 * N, 65 * N - 1, 100 * N + 7, 20000]:
        for d in (0, 1):
            lens.append(S)
            idx.append(d)
            levels.append(rng.integers(0, 256, size=doms[d].windows(S) * doms[d].E).astype(np.uint8))
    b = crafted_batch(doms, levels, lens, idx)
    plan = make_plan(b, out_align=align, kernel="warp_tile")
    _, _, out, lv = gpu_decode(plan, b, out_fill=float("nan"))
    h = out.cpu().numpy()
    xs, off, olv, lv_off = oracle.decode_many(b, np.arange(b.n_streams), want_levels=True)
    lv = lv.cpu().numpy()
    for i, S in enumerate(lens):
        d = doms[idx[i]]
        o, a = int(plan.segments[i]["out_offset"]), int(plan.level_offsets[i])
        L = d.windows(S) * d.E
        np.testing.assert_array_equal(lv[a:a + L], olv[int(lv_off[i]):int(lv_off[i]) + L])
        err = np.abs(h[o:o + S].astype(np.float64) - xs[int(off[i]):int(off[i]) + S]).max()
        assert err <= (10 + d.E / 2) * 2.0 ** -24 * 2 * d.E, (i, err)
    mask = np.ones(h.size, bool)
    for sg in plan.segments:
        mask[int(sg["out_offset"]):int(sg["out_offset"]) + int(sg["n_samples"])] = False
    assert np.all(np.isnan(h[mask]))
    assert plan.device_status()[0] == 0


@pytest.mark.parametrize("N,E", [(32, 16), (16, 8), (64, 32), (128, 128), (100, 50), (127, 127), (5, 5)])
def test_long_and_short_words(N, E):
    """Words of 64 one-bit codewords (a pass of 64 words holds 4096 symbols, more
    than a warp's stage: the words that fit are decoded, the rest in the next
    pass) beside words of a few long codewords, changing within a stream and from
    stream to stream, in ranges that start and end anywhere in a word.  Levels
    equal the oracle's bit for bit, samples within the FP32 bound."""
    cl = np.zeros(256, np.uint8)
    cl[128] = 1
    cl[np.r_[0:32, 200:232]] = 7
    d = oracle.Domain(N, E, min(2, E), E, 50.0, 0.004, (3.0, 2.0, 0.0), 8, cl)
    long_codes = np.r_[0:32, 200:232]
    rng = np.random.default_rng(N + E)
    lens, levels = [], []
    for i, W in enumerate([1, 3, 64, 1000, 4097, 300, 20000 // E]):
        x = np.full(W * E, 128, np.uint8)
        at = 0
        while at < x.size:  # runs of either kind
            n = int(rng.integers(1, 9000))
            if i % 3 != 1 and rng.random() < 0.5:
                x[at:at + n] = rng.choice(long_codes, size=x[at:at + n].size)
            at += n
        x[:E] = rng.choice(long_codes, size=E)  # no stream of zeros alone
        lens.append(W * N)
        levels.append(x)
    b = crafted_batch([d], levels, lens, [0] * len(lens))
    for ctas in (0, 1):
        plan = make_plan(b, out_align=32, kernel="warp_tile", ctas_per_sm=ctas)
        _, _, out, lv = gpu_decode(plan, b, out_fill=float("nan"))
        assert plan.device_status()[0] == 0
        compare_with_oracle(plan, b, out, lv)


@pytest.mark.parametrize("N,Es", [(12, [5, 8]), (24, [9, 24]), (48, [7, 40]), (52, [13, 48]), (72, [8, 71]), (81, [41, 8]),
                                  (84, [40, 81]), (85, [85, 48]), (88, [88, 33]), (96, [95, 16]), (100, [50, 33]),
                                  (127, [64, 127])])
@pytest.mark.parametrize("align", [32, 1])
def test_pair_form_thread_counts(N, Es, align):
    """The pair form with one to eight groups of eight pairs a window, with two output
    tiles per warp (four windows a lane) and with one (two windows a lane: 768
    threads, and other counts where two tiles do not fit): every window of a step,
    every pair of it, bins of either parity last."""
    b = _random_batch(N, Es, seed=N + align)
    for threads in (0, 256, 512, 768):
        plan = make_plan(b, out_align=align, out_base=0 if align == 32 else 3, kernel="warp_tile", threads=threads)
        _, _, out, lv = gpu_decode(plan, b, out_fill=float("nan"))
        compare_with_oracle(plan, b, out, lv)
        assert plan.device_status()[0] == 0


@pytest.mark.parametrize("N,E,n", [(84, 40, 3), (84, 40, 4), (81, 41, 3), (100, 50, 3), (127, 127, 2)])
def test_pair_form_of_many_domains(N, E, n):
    """Plans whose tables leave the default no room for two output tiles per warp."""
    b = _random_batch(N, [E] * n, seed=N + n)
    for d in b.domains:
        d.lmax = 12  # decode tables of 8 KB a domain, the same codewords
    plan = make_plan(b, out_align=32)
    assert plan.info["kernel"] == WARP_TILE
    _, _, out, lv = gpu_decode(plan, b, out_fill=float("nan"))
    compare_with_oracle(plan, b, out, lv)
    assert plan.device_status()[0] == 0
