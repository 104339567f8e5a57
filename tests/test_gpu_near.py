"""The passes that settle near-matching pairs without their whole band: every
pair equals the CPU oracle (integer DP: the tolerance is zero), on inputs where
the bounds are close -- repeats, whose off-diagonal paths nearly match too,
edits near the ends, short targets -- and on scorings that move each bound."""
import random

import numpy as np
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, batch_from_lists, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

SCORINGS = [
    ScoringParams(),
    ScoringParams(w=15, zdrop=0),                 # the narrow band is the whole band
    ScoringParams(w=14),                          # and wider than it
    ScoringParams(w=60, zdrop=9),                 # stops close to the bound
    ScoringParams(2, -3, 2, 2, 50, 20, -2),
    ScoringParams(3, 0, 1, 0, 40, 0, 0),          # free gap extension
    ScoringParams(1, -1, 1, 1, 40, 8, -1),        # gaps as cheap as mismatches
    ScoringParams(5, -4, 0, 3, 40, 30, 0),        # no opening penalty
    ScoringParams(1, -9, 126, 1, 41, 0, -9),      # alpha 127, and past it
    ScoringParams(1, -9, 127, 1, 41, 0, -9),
    ScoringParams(2, -8, 12, 1, 100, 100, -127),
    ScoringParams(1, -4, 0, 0, 30, 100, -1),      # gaps cost nothing
]


@pytest.fixture(scope="module")
def ctx():
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = xt.Context(0)
    yield c
    c.close()


def near_batch(seed, n):
    rng = random.Random(seed)
    qs, ts, hs = [], [], []
    for _ in range(n):
        ql = rng.choice([rng.randint(1, 18), rng.randint(1, 70), rng.randint(20, 140),
                         rng.choice([6, 7, 8, 9, 15, 16, 30, 31, 62, 63, 254, 255, 509, 510, 511])])
        kind = rng.random()
        if kind < 0.3:
            unit = [rng.randint(0, 3) for _ in range(rng.randint(1, 5))]
            base = (unit * 800)[:800]
        elif kind < 0.5:
            base = [rng.choice([0, 0, 0, 1]) for _ in range(800)]
        else:
            base = [rng.randint(0, 3) for _ in range(800)]
        t = base[:max(0, ql + rng.choice([0, 0, -1, 1, rng.randint(0, 20), rng.randint(0, 200)]))]
        sub, gap = rng.choice([0, 0.01, 0.02, 0.05]), rng.choice([0, 0, 0.01, 0.03])
        q, p = [], 0
        while len(q) < ql:
            r = rng.random()
            if r < sub:
                q.append(rng.randint(0, 3))
                p += 1
            elif r < sub + gap / 2:
                q.extend(rng.randint(0, 3) for _ in range(rng.randint(1, 6)))
            elif r < sub + gap:
                p += rng.randint(1, 6)
            elif r < sub + gap + 0.003:
                q.append(rng.choice([4, 5, 9, 255]))  # any byte >= 4 is N
                p += 1
            else:
                q.append(base[p % 800])
                p += 1
        if rng.random() < 0.2:  # a mismatch in one of the last bases
            k = ql - 1 - min(ql - 1, rng.randint(0, 4))
            q[k] = (q[k] + 1) % 4
        qs.append(q[:ql])
        ts.append(t)
        hs.append(rng.choice([1, 5, 19, 30, 60, rng.randint(1, 300)]))
    return batch_from_lists(qs, ts, hs)


@pytest.mark.parametrize("si", range(len(SCORINGS)))
def test_near_pairs(ctx, si):
    b = near_batch(900 + si, 6000)
    assert_same(run_gpu(ctx, b, SCORINGS[si]), run_oracle(b, SCORINGS[si]), f"{SCORINGS[si]}")


@pytest.mark.parametrize("n", [4095, 4096, 4097, 4351])
def test_near_small_batches(ctx, n):
    # around the smallest batch, partly filled warps and blocks, and buffers that start off a word
    import torch
    b = near_batch(50 + n, n)
    want = run_oracle(b, SCORINGS[0])
    for shift in range(3):
        pad = np.full(shift, 2, np.uint8)
        T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        q, t = T(np.concatenate([pad, b.q_seq]))[shift:], T(np.concatenate([pad, b.t_seq]))[shift:]
        out, cells = ctx.extend(q, T(b.q_off), T(b.q_len), t, T(b.t_off), T(b.t_len), T(b.h0),
                                SCORINGS[0])
        torch.cuda.synchronize()
        assert_same((out.cpu().numpy(), cells.cpu().numpy()), want, f"n={n} shift={shift}")
