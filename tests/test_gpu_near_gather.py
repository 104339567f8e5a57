"""What the near pass leaves goes back to the queue: batches whose pairs crowd into
one length or a few (most of them left by the near pass) equal the CPU oracle, and
one length costs no more than sixteen neighbouring ones."""
import random
from dataclasses import replace

import numpy as np
import pytest

from paper_2301_09310_gb300 import synth
from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, batch_from_lists, run_gpu, run_oracle, to_dev

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


def reads(seed, n, lengths, sub):
    rng = random.Random(seed)
    qs, ts, hs = [], [], []
    for _ in range(n):
        ql = rng.choice(lengths)
        t = [rng.randint(0, 3) for _ in range(ql + 100)]
        rate = rng.choice(sub)
        q = [(b + rng.randint(1, 3)) % 4 if rng.random() < rate else b for b in t[:ql]]
        qs.append(q)
        ts.append(t)
        hs.append(rng.randint(19, 60))
    return batch_from_lists(qs, ts, hs)


@pytest.mark.parametrize("lengths", [(150,), (510,), (1,), (511, 40), (30, 31, 126, 127, 254, 255),
                                     tuple(range(1, 511))], ids=lambda t: f"{t[0]}x{len(t)}")
@pytest.mark.parametrize("sub", [(0.03,), (0.0, 0.02), (0.2,)], ids=str)
def test_left_pairs_by_length(ctx, lengths, sub):
    sc = ScoringParams()
    b = reads(len(lengths), 400, lengths, sub)
    want, cells = run_oracle(b, sc)
    idx = np.random.default_rng(1).integers(0, b.n, 30000)
    many = type(b)(b.q_seq, b.q_off[idx], b.q_len[idx], b.t_seq, b.t_off[idx], b.t_len[idx], b.h0[idx])
    assert_same(run_gpu(ctx, many, sc), (want[idx], cells[idx]), f"{lengths[:4]} {sub}")


def test_one_length_costs_like_sixteen(ctx):
    # most of these pairs are left by the near pass; the batches differ in length by 5%
    import torch
    wl = replace(synth.WORKLOADS["c2_short"], len_kind=0, qlen_fixed=150, p_sub=0.04, p_unrelated=0.0)
    n = 500_000
    b = synth.generate(replace(wl, n_pairs=n), n=n)
    spread = replace_lengths(b, 135 + np.arange(n, dtype=np.int32) % 16)
    ms = []
    for x in (b, spread):
        args = to_dev(x, torch.device("cuda", ctx.device))
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for rep in range(6):
            t0.record()
            ctx.extend(*args, wl.scoring)
            t1.record()
            torch.cuda.synchronize()
            if rep:
                best = min(best, t0.elapsed_time(t1))
        ms.append(best)
    assert ms[0] < 1.5 * ms[1], ms


def replace_lengths(b, q_len):
    return type(b)(b.q_seq, b.q_off, np.minimum(b.q_len, q_len), b.t_seq, b.t_off, b.t_len, b.h0)
