"""The work that is timed: decodes, differentiable steps and encodes as a user's program calls them.

A case names one call of the public API and the batch it works on:

  op       decode  ``Plan.decode``                      compressed batch -> float32 samples
           train   ``decode_differentiable`` + gradient -> samples, dL/dC, dL/dA
           encode  ``Encoder.encode``                   float32 samples -> words, symbol counts, word counts
  idct     the plan's precision form (fp32, tf32, bf16x3, tf32x3)
  kinds    signal kinds of the batch, one domain (tables trained for it) each
  shapes   (window size N)x(kept bins E) of each domain: one for all, or one per kind
  streams, lo, hi   how many signals and their lengths (log-uniform in [lo, hi], a function of these three alone)

Streams are synthetic: sums of tones, coloured noise and decaying events with
the spectra of EEG channels, seismic traces, power-grid telemetry and
meteorological series, on which the trained codes come out at 4 to 8 bits a
level.  Tables are trained once per (kind, shape) on signals of their own seed.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2605_01086_gb300 import Plan, codec
from paper_2605_01086_gb300.decoder import decode_differentiable
from paper_2605_01086_gb300.encoder import Encoder

KINDS = ("eeg", "seismic", "power", "met")
ALL = ",".join(KINDS)
MU, ALPHA1, LMAX, PERCENTILE = 50.0, 0.004, 12, 99.9
SAMPLES_MAX = 120_000_000  # of a drawn case
LEVEL_BITS = {"eeg": 7.0, "seismic": 4.5, "power": 6.5, "met": 6.5}  # about, of the trained codes


def listed():
    def case(name, op, kinds, shapes, streams, lo, hi, idct="fp32"):
        return {"name": name, "op": op, "idct": idct, "kinds": kinds, "shapes": shapes, "streams": streams, "lo": lo,
                "hi": hi}
    return [
        # one EEG channel on request: launches and a warp's serial chain are all there is
        case("decode_stream", "decode", "eeg", "32x16", 1, 65536, 65536),
        # a seismic archive read back: very many short traces, one tile each
        case("decode_traces", "decode", "seismic", "32x16", 16384, 4096, 4096),
        # the main load of a decode server: every domain and length in one batch
        case("decode_mixed", "decode", ALL, "32x16", 1200, 4096, 524288),
        # the same from a server that takes the tensor-core form
        case("decode_mixed_bf16x3", "decode", ALL, "32x16", 800, 4096, 262144, "bf16x3"),
        # larger windows: E = 32 of N = 64
        case("decode_n64_e32", "decode", "eeg", "64x32", 1024, 65536, 65536),
        # a window that is not a power of two (100 samples: a second at 100 Hz), ragged lengths
        case("decode_n100_e50", "decode", "seismic", "100x50", 512, 60007, 70001),
        # domains that each chose their own window and rate, in one batch
        case("decode_shapes", "decode", ALL, "64x16,16x8,128x32,32x8", 600, 4096, 262144),
        # fitting the decoder's scales or an upstream model through the decoder
        case("train_power", "train", "power", "32x16", 1024, 65536, 65536),
        # the same with a larger window
        case("train_n64_e32", "train", "eeg", "64x32", 256, 65536, 65536),
        # one channel acquired and compressed at once
        case("encode_stream", "encode", "eeg", "32x16", 1, 65536, 65536),
        # server-side (re-)encoding of a mixed batch
        case("encode_mixed", "encode", ALL, "32x16", 800, 4096, 524288),
        # the same for a larger window
        case("encode_n64_e32", "encode", "eeg", "64x32", 256, 65536, 65536),
    ]


def draw(rng):
    op = rng.choice(("decode", "decode", "decode", "train", "encode"))
    table = ["32x16", "32x16", "32x16", "16x8", "32x8", "32x32", "64x16", "64x32", "128x32", "128x64", "24x12", "48x24",
             "100x50"]
    kinds = list(KINDS) if rng.random() < 0.4 else [rng.choice(KINDS)]
    if len(kinds) > 1 and rng.random() < 0.3:
        shapes = ",".join(rng.choice(table) for _ in kinds)
    else:
        shapes = rng.choice(table)
    idct = "fp32"
    if op == "decode" and shapes in ("32x16", "32x32", "64x32", "128x32", "128x64") and rng.random() < 0.3:
        idct = rng.choice(("tf32", "bf16x3", "tf32x3"))
    lo = int(round(math.exp(rng.uniform(math.log(100), math.log(65536)))))
    hi = int(round(lo * math.exp(rng.uniform(0.0, math.log(64)))))
    mean = lo if hi == lo else (hi - lo) / math.log(hi / lo)
    # the shapes without a kernel of their own cost several times more a sample
    cap = SAMPLES_MAX if shapes == "32x16" else SAMPLES_MAX // 8
    streams = int(round(math.exp(rng.uniform(0.0, math.log(max(2.0, min(20000.0, cap / mean)))))))
    case = {"op": op, "idct": idct, "kinds": ",".join(kinds), "shapes": shapes, "streams": max(1, streams), "lo": lo,
            "hi": hi}
    while int(_lengths(case).sum()) > cap and case["streams"] > 1:
        case["streams"] = max(1, case["streams"] * 3 // 4)
    return case


# ---- the batch of a case ------------------------------------------------------

def _lengths(case):
    n, lo, hi = case["streams"], case["lo"], case["hi"]
    r = random.Random(f"{n}/{lo}/{hi}")
    return np.array([int(round(math.exp(r.uniform(math.log(lo), math.log(hi))))) if hi > lo else lo
                     for _ in range(n)], np.int64)


def _domain_index(case):
    return np.arange(case["streams"], dtype=np.int64) % len(case["kinds"].split(","))


def _shapes(case):
    kinds, shapes = case["kinds"].split(","), case["shapes"].split(",")
    shapes = shapes * len(kinds) if len(shapes) == 1 else shapes
    return [(k, *map(int, s.split("x"))) for k, s in zip(kinds, shapes)]


# per kind: offset, two tones (amplitude, least and most cycles a sample), the
# noise's white, short-range and slow parts, events (amplitude over the
# background, samples between them, decay in samples)
_TABLE = {
    #          offset  a1    f1lo    f1hi    a2    f2lo     f2hi   white  fir   slow  event  gap   decay
    "eeg":     (0.0, 12.0, 0.032, 0.050, 9.0, 0.006, 0.016, 1.2, 5.0, 14.0, 0.0, 4000, 200),
    "seismic": (0.0, 0.02, 0.001, 0.003, 0.01, 0.05, 0.10, 0.01, 0.10, 0.06, 12.0, 9000, 450),
    "power":   (0.0, 1.0, 0.0078, 0.0079, 0.04, 0.039, 0.040, 0.004, 0.008, 0.03, 0.6, 7000, 120),
    "met":     (15.0, 9.0, 0.00069, 0.0007, 2.0, 0.0027, 0.0029, 0.15, 0.2, 2.0, 0.0, 5000, 300),
}


def _signals(kinds, lengths, seed):
    """The streams back to back, float32 on the GPU."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(seed))
    n, total = len(lengths), int(lengths.sum())
    tab = torch.tensor([_TABLE[k] for k in kinds], dtype=torch.float64, device=dev)
    u = torch.rand(n, 6, dtype=torch.float64, device=dev, generator=g)
    gain = 0.6 + 0.8 * u[:, 0]
    f1 = tab[:, 2] + (tab[:, 3] - tab[:, 2]) * u[:, 1]
    f2 = tab[:, 5] + (tab[:, 6] - tab[:, 5]) * u[:, 2]
    start = torch.zeros(n, dtype=torch.int64, device=dev)
    ln = torch.from_numpy(lengths).to(dev)
    start[1:] = torch.cumsum(ln, 0)[:-1]
    ends = start + ln
    x = torch.empty(total, dtype=torch.float32, device=dev)
    step, taps, slow = 1 << 24, 8, 32
    for a in range(0, total, step):
        b = min(total, a + step)
        i = torch.arange(a, b, device=dev)
        s = torch.searchsorted(ends, i, right=True)
        t = (i - start[s]).double()
        white = torch.randn(b - a + taps, device=dev, generator=g)
        fir = sum(0.75 ** j * white[j:j + b - a] for j in range(taps)) * 0.6
        coarse = torch.randn((b - a) // slow + 2, device=dev, generator=g)
        q, r = (i - a) // slow, ((i - a) % slow).float() / slow
        drift = coarse[q] * (1 - r) + coarse[q + 1] * r
        tk = tab.float()[s]
        since = torch.remainder(t + 1000.0 * u[s, 5] * tab[s, 11], tab[s, 11]).float()
        env = 1.0 + tk[:, 10] * torch.exp(-since / tk[:, 12])
        tone = tk[:, 1] * torch.sin(2 * math.pi * torch.frac(f1[s] * t + u[s, 3])).float() \
            + tk[:, 4] * torch.sin(2 * math.pi * torch.frac(f2[s] * t + u[s, 4])).float()
        noise = tk[:, 7] * white[:b - a] + tk[:, 8] * fir + tk[:, 9] * drift
        x[a:b] = tk[:, 0] + gain[s].float() * (tone + env * noise)
    return x


@functools.lru_cache(maxsize=None)
def _trained(kind, N, E):
    lengths = np.full(16, 16384, np.int64)
    x = _signals([kind] * len(lengths), lengths, 900_000 + KINDS.index(kind)).cpu().numpy()
    return codec.train_domain(x, np.arange(len(lengths)) * 16384, lengths, N, E, min(2, E), E, MU, ALPHA1, LMAX,
                              PERCENTILE)


def _compressed(domains, lengths, di, x):
    """The batch's words and symbol counts on the GPU, stream after stream, with its segment table."""
    enc = Encoder(domains, lengths, di)
    words, symlen, n_words = enc.encode(x)
    nw = n_words.cpu().numpy()[:len(lengths)]
    off = np.concatenate([[0], np.cumsum(nw)[:-1]]).astype(np.int64)
    shift = torch.from_numpy(enc.room_offsets.astype(np.int64) - off).cuda()
    idx = torch.repeat_interleave(shift, torch.from_numpy(nw).cuda()) + torch.arange(int(nw.sum()), device="cuda")
    words, symlen = words[idx].contiguous(), symlen[idx].contiguous()
    enc.close()
    segs = codec.segments_array(off, nw, lengths, codec.packed_out_offsets(lengths), di)
    return words, symlen, segs


def prepare(case, seed):
    lengths, di = _lengths(case), _domain_index(case)
    shapes = _shapes(case)
    domains = [_trained(*s) for s in shapes]
    x = _signals([shapes[d][0] for d in di], lengths, seed)
    st = {"op": case["op"]}
    if case["op"] == "encode":
        st["encoder"] = Encoder(domains, lengths, di)
        st["x"] = x
        st["buffers"] = st["encoder"].buffers()
        return st
    st["words"], st["symlen"], segs = _compressed(domains, lengths, di, x)
    st["plan"] = plan = Plan(domains, segs, idct=case["idct"])
    if case["op"] == "decode":
        # a buffer kept between calls; the padding between streams stays zero
        st["out"] = torch.zeros(plan.info["out_extent"], dtype=torch.float32, device=plan.device)
        return st
    g = torch.Generator(device=plan.device).manual_seed(int(seed) + 1)
    st["scale"] = torch.tensor([d.scale for d in domains], dtype=torch.float32, device=plan.device, requires_grad=True)
    st["probe"] = torch.zeros(plan.info["n_levels_total"], device=plan.device, requires_grad=True)
    st["grad"] = torch.randn(plan.info["out_extent"], device=plan.device, generator=g)
    st["gap"] = None
    if int(lengths.sum()) != plan.info["out_extent"]:  # padding between streams, which no call writes
        st["gap"] = torch.ones(plan.info["out_extent"], dtype=torch.bool, device=plan.device)
        for a, b in zip(segs["out_offset"].astype(np.int64), lengths):
            st["gap"][int(a):int(a + b)] = False
    return st


def run(state):
    if state["op"] == "encode":
        return state["encoder"].encode(state["x"], *state["buffers"])
    plan = state["plan"]
    if state["op"] == "decode":
        return plan.decode(state["words"], state["symlen"], out=state["out"])
    out = decode_differentiable(plan, state["words"], state["symlen"], state["scale"], state["probe"])
    g_scale, g_coeffs = torch.autograd.grad(out, (state["scale"], state["probe"]), state["grad"])
    out = out.detach()
    if state["gap"] is not None:
        out = out.masked_fill(state["gap"], 0.0)
    return out, g_scale, g_coeffs


def work(case):
    """Compressed words are 8 bytes and a symbol count each, about 61 of their 64 bits used."""
    lengths, di = _lengths(case), _domain_index(case)
    shapes = _shapes(case)
    samples = int(lengths.sum())
    levels = words = macs = 0
    for S, d in zip(lengths, di):
        kind, N, E = shapes[d]
        W = -(-int(S) // N)
        levels += W * E
        words += int(W * E * LEVEL_BITS[kind] / 61) + 1
        macs += W * E * N
    if case["op"] == "train":
        # words read; samples written; gradient read; coefficient gradients written
        return {"bytes": 9 * words + 8 * samples + 4 * levels, "flops": 4 * macs}
    return {"bytes": 9 * words + 4 * samples, "flops": 2 * macs}


# ---- the same in 64 bits ------------------------------------------------------

def _levels(domains, segs, words, symlen):
    """Every stream's levels back to back (streams in order), from canonical codes."""
    dev = words.device
    size = 1 << LMAX
    sym = torch.zeros(len(domains), size, dtype=torch.int64)
    length = torch.zeros(len(domains), size, dtype=torch.int64)
    for d, dom in enumerate(domains):
        at = 0  # canonical order fills the table of prefixes from 0 up
        for s in sorted((int(v), i) for i, v in enumerate(dom.code_len) if v):
            end = at + (1 << (LMAX - s[0]))
            sym[d, at:end], length[d, at:end] = s[1], s[0]
            at = end
    sym, length = sym.flatten().to(dev), length.flatten().to(dev)
    nw = torch.from_numpy(segs["n_words"].astype(np.int64)).to(dev)
    dom_w = torch.repeat_interleave(torch.from_numpy(segs["domain"].astype(np.int64)).to(dev), nw) * size
    n = symlen.long()
    pos = torch.cumsum(n, 0) - n
    levels = torch.zeros(int(n.sum()), dtype=torch.uint8, device=dev)
    w = words.clone()
    for j in range(int(n.max())):
        live = n > j
        e = dom_w + ((w >> (64 - LMAX)) & (size - 1))
        levels[pos[live] + j] = sym[e[live]].to(torch.uint8)
        w = w << length[e]
    return levels


def _unit(dev):
    """Reconstruction at scale 1 of zones 0 (mu-law) and 1 (deadzone lattice)."""
    u = np.zeros((2, 256))
    for L in range(256):
        if L > 128:
            u[0, L] = ((1 + MU) ** ((L - 128) / 127.0) - 1) / MU
            u[1, L] = ALPHA1 + (L - 129) / 126.0 * (1 - ALPHA1)
        elif L < 128:
            u[0, L] = -((1 + MU) ** ((128 - L) / 128.0) - 1) / MU
            u[1, L] = -(ALPHA1 + (127 - L) / 127.0 * (1 - ALPHA1))
    return torch.from_numpy(u).to(dev)


def exact(case, seed):
    if case["op"] == "encode":
        return None  # words and counts: whole numbers
    st = prepare(case, seed)
    plan = st["plan"]
    dev, segs, domains = plan.device, plan.segments, plan.domains
    levels = _levels(domains, segs, st["words"], st["symlen"])
    out = torch.zeros(plan.info["out_extent"], dtype=torch.float64, device=dev)
    train = case["op"] == "train"
    g_coeffs = torch.zeros(levels.numel(), dtype=torch.float64, device=dev) if train else None
    g_scale = torch.zeros(len(domains), 3, dtype=torch.float64, device=dev)
    unit = _unit(dev)
    S = segs["n_samples"].astype(np.int64)
    per = np.array([-(-int(s) // domains[d].N) for s, d in zip(S, segs["domain"])], np.int64)
    lev_off = np.concatenate([[0], np.cumsum(per * np.array([domains[d].E for d in segs["domain"]]))])[:-1]
    for d, dom in enumerate(domains):
        mine = np.nonzero(segs["domain"] == d)[0]
        k = torch.arange(dom.E, device=dev)
        nn = torch.arange(dom.N, device=dev)
        basis = torch.cos(math.pi * (2 * nn[None, :] + 1).double() * k[:, None].double() / (2 * dom.N))
        basis[0] = 0.5
        zone1 = (k >= dom.B1).long()
        a = torch.tensor([np.float32(v) for v in dom.scale[:2]], dtype=torch.float64, device=dev)
        scale = a[zone1] * (k < dom.B2)
        for c in range(0, len(mine), 4096):
            ids = mine[c:c + 4096]
            t = lambda v: torch.from_numpy(np.ascontiguousarray(v[ids].astype(np.int64))).to(dev)  # noqa: E731
            pw = t(per)
            first = torch.cumsum(pw, 0) - pw
            win = torch.arange(int(pw.sum()), device=dev) - torch.repeat_interleave(first, pw)
            li = (torch.repeat_interleave(t(lev_off), pw) + win * dom.E)[:, None] + k
            v = unit[zone1, levels[li].long()]
            si = (win * dom.N)[:, None] + nn
            ok = si < torch.repeat_interleave(t(S), pw)[:, None]
            si += torch.repeat_interleave(t(segs["out_offset"]), pw)[:, None]
            out[si[ok]] = ((v * scale) @ basis)[ok]
            if train:
                gx = torch.where(ok, st["grad"][torch.where(ok, si, 0)].double(), 0.0)
                gc = gx @ basis.T
                g_coeffs[li] = gc
                m = (gc * v * (k < dom.B2)).sum(0)
                g_scale[d, 0] += m[:dom.B1].sum()
                g_scale[d, 1] += m[dom.B1:].sum()
            del li, v, si, ok
    return [out, g_scale, g_coeffs] if train else out
