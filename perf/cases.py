"""The calls this library is measured on.

Every case is one call of a public entry point on data shaped like the
library's workload presets (paper_2301_09310_gb300/synth.py): small and large
batches, short and long reads, equal-length tables, both-direction seeds, the
BWA-MEM-compatible variant and the host-buffer call.  A case is a dict of
plain values:

    call      "extend", "seeds", "bwa" or "host": the entry point
    preset    the workload preset the pairs are drawn from, or "equal" for
              equal-length pairs whose band is the whole table
    pairs     pairs (reads, for "seeds") per call
    length    equal-length pairs: bases per sequence; seeds: bases per read;
              else 0 (the preset's own lengths)
    w, zdrop  band half-width and z-drop cutoff (0: off)
    unrelated share of pairs whose query and target are unrelated
    alphabet  "codes", "ascii" or "packed4"
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

import paper_2301_09310_gb300 as xt
from paper_2301_09310_gb300 import synth

_SEED_LEN = 19        # exact-match seed of a read, bases
_SEEDS_PER_READ = 2
_SEED_MARGIN = 100    # target bases before and after the read's own window
_ALPHABETS = {"codes": xt.XT_ALPHABET_CODES, "ascii": xt.XT_ALPHABET_ASCII,
              "packed4": xt.XT_ALPHABET_PACKED4}


def _case(name, call, preset, pairs, length=0, w=100, zdrop=100, unrelated=0.05,
          alphabet="codes"):
    return {"name": name, "call": call, "preset": preset, "pairs": pairs, "length": length,
            "w": w, "zdrop": zdrop, "unrelated": unrelated, "alphabet": alphabet}


def listed():
    return [
        # one read pair file's worth of 100-base extensions: the smallest call,
        # where launches and the host's part decide
        _case("tiny_1k", "extend", "c1_tiny", 1000, unrelated=0.0),
        # the kernel comparison of the method: 5,000 equal-length pairs, whole
        # tables, z-drop off; short and medium length
        _case("equal_64", "extend", "equal", 5000, length=64, w=64, zdrop=0, unrelated=0.0),
        _case("equal_1024", "extend", "equal", 5000, length=1024, w=1024, zdrop=0, unrelated=0.0),
        # one lane of 150-base reads: what is left of each read past its seed
        _case("short_1m", "extend", "c2_short", 1_000_000),
        # the benchmark's batch: reads of 100, 150 and 250 bases mixed
        _case("mixed_4m", "extend", "c3_mixed", 4_000_000),
        # long reads, a whole chunk of them and a small batch
        _case("long_250k", "extend", "c4_long", 250_000, w=500, zdrop=400, unrelated=0.0),
        _case("long_3k", "extend", "c4_long", 3_001, w=500, zdrop=400, unrelated=0.0),
        # batches the server forms from a request stream at low and at high load
        _case("stream_55k", "extend", "c5_stream", 55_001),
        _case("stream_885k", "extend", "c5_stream", 885_003),
        # raw 150-base reads, two seeds each, extended to both sides
        _case("seeds_200k", "seeds", "c2_short", 100_000, length=150, unrelated=0.0,
              alphabet="ascii"),
        # the same kind of batch under the BWA-MEM-compatible definition
        _case("bwa_500k", "bwa", "c3_mixed", 500_000),
        # an aligner whose batches live in pinned host memory
        _case("host_2m", "host", "c3_mixed", 2_200_000),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["reads", "reads", "stream", "long", "equal", "seeds", "bwa", "host"])
    unrelated = rng.choice([0.0, 0.05, 0.1])
    if kind == "long":
        w = log_int(200, 500)
        return _drawn("extend", "c4_long", log_int(1000, 250_000), w=w, zdrop=rng.choice([0, 400]),
                      unrelated=0.0)
    if kind == "equal":
        length = log_int(64, 4096)
        return _drawn("extend", "equal", log_int(1000, 5000), length=length, w=length, zdrop=0,
                      unrelated=0.0)
    w, zdrop = log_int(50, 200), rng.choice([0, 100, 100])
    alphabet = rng.choice(["codes", "codes", "ascii", "packed4"])
    reads = rng.choice(["c2_short", "c3_mixed"])
    if kind == "seeds":
        return _drawn("seeds", "c2_short", log_int(1000, 500_000), length=rng.randint(80, 250),
                      w=w, zdrop=zdrop, unrelated=0.0, alphabet=alphabet)
    if kind == "bwa":
        return _drawn("bwa", reads, log_int(1000, 2_000_000), w=w, zdrop=zdrop,
                      unrelated=unrelated, alphabet=alphabet)
    if kind == "host":
        return _drawn("host", reads, log_int(20_000, 3_000_000), unrelated=unrelated,
                      alphabet=alphabet)
    preset = "c5_stream" if kind == "stream" else reads
    top = 2_000_000 if kind == "stream" else 4_000_000
    return _drawn("extend", preset, log_int(1000, top), w=w, zdrop=zdrop, unrelated=unrelated,
                  alphabet=alphabet)


def _drawn(call, preset, pairs, **kw):
    c = _case("", call, preset, pairs, **kw)
    del c["name"]
    return c


def _workload(case, seed):
    if case["preset"] == "equal":
        wl = synth.x2_workload(case["length"], case["pairs"])
    else:
        wl = synth.WORKLOADS[case["preset"]]
        if case["call"] == "seeds":
            wl = replace(wl, len_kind=0, qlen_fixed=case["length"], tlen_extra=_SEED_MARGIN)
    sc = replace(wl.scoring, w=case["w"], zdrop=case["zdrop"])
    return replace(wl, n_pairs=case["pairs"], seed=seed, p_unrelated=case["unrelated"], scoring=sc)


def _letters(codes, alphabet):
    """Base codes as the call's alphabet has them (a host array)."""
    if alphabet == "ascii":
        return np.frombuffer(b"ACGTN", np.uint8)[np.minimum(codes, 4)]
    if alphabet == "packed4":
        return xt.pack4(codes)
    return codes


def _seeds(wl, b, seed):
    """Two seeds a read; the read's target window gets _SEED_MARGIN bases in front."""
    rng = np.random.default_rng(seed)
    n, read = b.n, wl.qlen_fixed
    window = int(b.t_len[0]) + _SEED_MARGIN
    t = rng.integers(0, 4, (n, window), dtype=np.uint8)
    t[:, _SEED_MARGIN:] = b.t_seq.reshape(n, window - _SEED_MARGIN)
    of = np.repeat(np.arange(n, dtype=np.int64), _SEEDS_PER_READ)
    q_beg = rng.integers(0, read - _SEED_LEN + 1, of.size, dtype=np.int32)
    full = lambda v: np.full(of.size, v, np.int32)  # noqa: E731
    return {"q_seq": b.q_seq, "q_off": of * read, "q_len": full(read), "t_seq": t.reshape(-1),
            "t_off": of * window, "t_len": full(window), "q_beg": q_beg,
            "t_beg": q_beg + _SEED_MARGIN, "seed_len": full(_SEED_LEN),
            "h0": full(_SEED_LEN * wl.scoring.match)}


def _arrays(case, seed):
    """(workload, the call's host arrays in its argument order)."""
    wl = _workload(case, seed)
    b = synth.generate(wl)
    if case["call"] == "seeds":
        a = _seeds(wl, b, seed)
    else:
        a = {"q_seq": b.q_seq, "q_off": b.q_off, "q_len": b.q_len, "t_seq": b.t_seq,
             "t_off": b.t_off, "t_len": b.t_len, "h0": b.h0}
    for name in ("q_seq", "t_seq"):
        a[name] = _letters(a[name], case["alphabet"])
    return wl, a


def prepare(case, seed):
    wl, a = _arrays(case, seed)
    ctx = xt.Context(0)
    ctx.set_alphabet(_ALPHABETS[case["alphabet"]])
    scoring = wl.scoring
    if case["call"] == "bwa":
        scoring = synth.BwaScoringParams.from_scoring(scoring)
    if case["call"] == "host":
        keep = [torch.from_numpy(np.ascontiguousarray(v)).pin_memory() for v in a.values()]
        args = [t.numpy() for t in keep]
        n = a["q_len"].size
        out = torch.empty((n, 7), dtype=torch.int32, pin_memory=True)
        cells = torch.empty(n, dtype=torch.int64, pin_memory=True)
        return {"call": "host", "ctx": ctx, "scoring": scoring, "args": args, "keep": keep,
                "results": (out, cells)}
    args = [torch.from_numpy(np.array(v)).cuda() for v in a.values()]
    return {"call": case["call"], "ctx": ctx, "scoring": scoring, "args": args}


def run(state):
    ctx, args, sc = state["ctx"], state["args"], state["scoring"]
    if state["call"] == "seeds":
        return ctx.extend_seeds(*args, sc)
    if state["call"] == "bwa":
        return ctx.extend_bwa(*args, sc)
    if state["call"] == "host":
        out, cells = state["results"]
        ctx.extend_host(*args, sc, out=out.numpy(), cells=cells.numpy())
        return out, cells
    return ctx.extend(*args, sc)


def work(case):
    """Bytes: every sequence, offset, length and seed score read once, every
    result and cell count written once.  Operations: ten integer operations
    (one cell update) for every query base, which any alignment has to score;
    how many cells off the alignment's path have to be evaluated depends on
    the data."""
    wl = _workload(case, 1)
    n = case["pairs"]
    ql, tl, _ = synth.shapes(wl, min(n, 100_000))
    q, t = float(np.mean(ql)) * n, float(np.mean(tl)) * n
    per_pair = 8 + 8 + 4 + 4 + 4 + 28 + 8
    if case["call"] == "seeds":
        t += _SEED_MARGIN * n
        seeds = n * _SEEDS_PER_READ
        extra = (8 + 8 + 6 * 4 + 2 * (28 + 8)) * seeds
        ops = 10.0 * (q - _SEED_LEN * n) * _SEEDS_PER_READ
    else:
        extra = per_pair * n
        ops = 10.0 * q
    letters = (q + t) * (0.5 if case["alphabet"] == "packed4" else 1.0)
    return {"bytes": letters + extra, "flops": ops}


def exact(case, seed):
    """The definition in 64-bit torch, row by row, for batches small enough."""
    if case["call"] != "extend":
        return None
    wl = _workload(case, seed)
    ql, tl, _ = synth.shapes(wl)
    n, qmax = case["pairs"], int(ql.max())
    rows = min(int(tl.max()), qmax + wl.scoring.w)
    if n * qmax * rows > 1_000_000_000 or rows > 1000:
        return None
    return _definition(synth.generate(wl), wl.scoring, qmax, rows)


def _definition(b, sc, qmax, rows):
    dev = torch.device("cuda")
    T = lambda a: torch.from_numpy(a.astype(np.int64)).to(dev)  # noqa: E731
    n = b.n
    ql, tl, h0 = T(b.q_len), T(b.t_len), T(b.h0)
    qs, ts = T(b.q_seq), T(b.t_seq)
    cols = torch.arange(qmax, device=dev)
    at = T(b.q_off)[:, None] + cols[None, :]
    q = torch.where(cols[None, :] < ql[:, None], qs[at.clamp(max=qs.numel() - 1)],
                    torch.full_like(at, 4)).clamp(max=4)
    alpha, beta = sc.gap_open + sc.gap_extend, sc.gap_extend
    zero = torch.zeros((), dtype=torch.int64, device=dev)
    # row -1: the insertion run from the seed, inside the band
    up_h = torch.where((cols + 1 <= sc.w)[None, :], (h0[:, None] - alpha - beta * cols).clamp(min=0),
                       zero)
    up_f = torch.zeros_like(up_h)
    corner = h0.clone()                         # H(i-1, -1)
    best, bi, bj = h0.clone(), torch.full_like(h0, -1), torch.full_like(h0, -1)
    max_off, gscore, gtle = torch.zeros_like(h0), torch.full_like(h0, -1), torch.zeros_like(h0)
    last = torch.full_like(h0, -1)
    stop = torch.zeros(n, dtype=torch.bool, device=dev)
    t_off = T(b.t_off)
    for i in range(rows):
        live_row = (i < tl) & ~stop
        tb = ts[(t_off + i).clamp(max=ts.numel() - 1)].clamp(max=4)
        s = torch.where(q == tb[:, None], sc.match, sc.mismatch)
        s = torch.where((q == 4) | (tb[:, None] == 4), sc.n_score, s)
        diag = torch.cat([corner[:, None], up_h[:, :-1]], 1)
        m = torch.where(diag > 0, diag + s, zero)
        f = torch.maximum(up_f - beta, up_h - alpha).clamp(min=0)
        left = (h0 - alpha - beta * i).clamp(min=0) if i + 1 <= sc.w else torch.zeros_like(h0)
        band = ((cols - i).abs() <= sc.w)[None, :] & (cols[None, :] < ql[:, None])
        x = torch.where(band, torch.maximum(m, f).clamp(min=0), zero)
        # E(i, j) = max over k < j of x(k) - alpha - beta (j - 1 - k), the boundary k = -1 too
        chain = torch.cat([left[:, None] - beta, x[:, :-1] + beta * cols[:-1]], 1)
        e = torch.cummax(chain, 1).values - alpha - beta * (cols - 1)
        h = torch.where(band, torch.maximum(x, e), zero)
        f = torch.where(band, f, zero)
        # row maximum with its largest column
        key = torch.where(band, h * (qmax + 1) + cols + 1, zero).max(1).values
        mi, mj = key // (qmax + 1), key % (qmax + 1) - 1
        last = torch.where(live_row & (mi > 0), i, last)
        end_in = (ql - 1 - i).abs() <= sc.w
        g = h.gather(1, (ql - 1)[:, None])[:, 0]
        better = live_row & end_in & (g > 0) & (g > gscore)
        gscore, gtle = torch.where(better, g, gscore), torch.where(better, i + 1, gtle)
        up = live_row & (mi > best)
        drop = best - mi - ((i - bi) - (mj - bj)).abs() * beta
        if sc.zdrop > 0:
            stop = stop | (live_row & ~up & (drop > sc.zdrop))
        best = torch.where(up, mi, best)
        bi, bj = torch.where(up, i, bi), torch.where(up, mj, bj)
        max_off = torch.where(up, torch.maximum(max_off, (mj - i).abs()), max_off)
        up_h, up_f, corner = h, f, left
    k = torch.arange(rows, device=dev)
    width = (torch.minimum(ql[:, None], k + sc.w + 1) - (k - sc.w).clamp(min=0)).clamp(min=0)
    cells = torch.where(k[None, :] <= last[:, None], width, zero).sum(1)
    out = torch.stack([best, bj + 1, bi + 1, gscore, gtle, max_off, torch.zeros_like(best)], 1)
    return out, cells
