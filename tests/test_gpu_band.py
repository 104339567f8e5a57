"""The band engine: every pair equals the CPU oracle (integer DP: the tolerance
is zero) at the band widths where its lane and slot counts change, with long
and short targets, ends inside and past the band, z-drop stops, seeds whose
boundary gap holds the row maximum, and scores up to its 16-bit limit."""
import random

import numpy as np
import pytest

from paper_2301_09310_gb300 import synth
from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, batch_from_lists, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = xt.Context(0)
    yield c
    c.close()


def long_batch(seed, n, top=1400, h0_top=300):
    rng = random.Random(seed)
    qs, ts, hs = [], [], []
    for _ in range(n):
        ql = rng.choice([511, 512, 513, rng.randint(511, 700), rng.randint(511, top)])
        kind = rng.random()
        if kind < 0.2:
            unit = [rng.randint(0, 3) for _ in range(rng.randint(1, 7))]
            base = (unit * 3000)[:3000]
        else:
            base = [rng.randint(0, 3) for _ in range(3000)]
        sub, gap = rng.choice([0, 0.02, 0.06]), rng.choice([0, 0.02, 0.05])
        q, p = [], 0
        while len(q) < ql:
            r = rng.random()
            if r < sub:
                q.append(rng.randint(0, 3))
                p += 1
            elif r < sub + gap / 2:
                q.extend(rng.randint(0, 3) for _ in range(rng.randint(1, 8)))
            elif r < sub + gap:
                p += rng.randint(1, 8)
            elif r < sub + gap + 0.003:
                q.append(rng.choice([4, 9, 255]))
                p += 1
            else:
                q.append(base[p % 3000])
                p += 1
        q = q[:ql]
        if rng.random() < 0.15:  # the alignment breaks off: a z-drop, or a dead end
            k = rng.randint(0, ql - 1)
            q[k:] = [rng.randint(0, 3) for _ in range(ql - k)]
        tl = max(1, ql + rng.choice([0, 0, -ql // 2, -100, 30, 200, 1200]))
        qs.append(q)
        ts.append(base[:tl])
        hs.append(rng.choice([1, 5, 30, rng.randint(1, h0_top)]))
    return batch_from_lists(qs, ts, hs)


SCORINGS = [ScoringParams(w=w, zdrop=z) for w, z in
            ((8, 0), (31, 50), (32, 100), (63, 0), (64, 100), (100, 100), (103, 0), (104, 40),
             (127, 100), (128, 100), (207, 0), (208, 100), (255, 60), (256, 100), (415, 0),
             (416, 100), (500, 400), (511, 0), (512, 100))]
SCORINGS += [
    ScoringParams(2, -3, 2, 2, 50, 20, -2),
    ScoringParams(3, 0, 1, 0, 120, 0, 0),            # free gap extension
    ScoringParams(5, -4, 0, 3, 90, 60, 0),           # no opening penalty
    ScoringParams(1, -9, 12, 1, 300, 0, -9),
    ScoringParams(1, -60, 60, 1, 100, 200, -60),     # keys at the edge of their range
    ScoringParams(10, -4, 6, 1, 100, 0, -1),         # scores near and past the 16-bit limit
]


@pytest.mark.parametrize("si", range(len(SCORINGS)))
def test_band_engine(ctx, si):
    sc = SCORINGS[si]
    b = long_batch(70 + si, 150, top=1400 if sc.w < 300 else 2600)
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), f"{sc}")


def test_band_engine_high_seeds(ctx):
    # seed scores far above what the query can add: the boundary gaps stay
    # above the rows for long, and the rows' keys start far from 0
    sc = ScoringParams(w=100, zdrop=100)
    b = long_batch(7, 300, h0_top=15000)
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), "high seeds")


def test_band_engine_long_reads(ctx):
    wl = synth.WORKLOADS["c4_long"]
    b = synth.generate(wl, n=96, first=1234)
    assert_same(run_gpu(ctx, b, wl.scoring), run_oracle(b, wl.scoring), "long reads")
