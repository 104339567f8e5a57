"""Pairs the near pass cannot settle beside many it can (so that it runs on all of
them): every pair equals the CPU oracle (integer DP: the tolerance is zero)."""
import random

import numpy as np
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, batch_from_lists, run_gpu, run_oracle
from tests.test_gpu_near import SCORINGS, near_batch

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


def promising(seed, n):
    """Reads whose first mismatches lie in their last bases: the diagonal pass gives
    them up late, and the narrow band settles them."""
    rng = random.Random(seed)
    qs, ts, hs = [], [], []
    for _ in range(n):
        ql = rng.randint(90, 250)
        t = [rng.randint(0, 3) for _ in range(ql + 15)]
        q = t[:ql]
        for _ in range(3):
            k = rng.randint(ql - 12, ql - 4)
            q[k] = (t[k] + 1) % 4
        qs.append(q)
        ts.append(t)
        hs.append(60)
    return batch_from_lists(qs, ts, hs)


def join(a, b):
    return type(a)(np.concatenate([a.q_seq, b.q_seq]), np.concatenate([a.q_off, b.q_off + a.q_seq.size]),
                   np.concatenate([a.q_len, b.q_len]), np.concatenate([a.t_seq, b.t_seq]),
                   np.concatenate([a.t_off, b.t_off + a.t_seq.size]),
                   np.concatenate([a.t_len, b.t_len]), np.concatenate([a.h0, b.h0]))


@pytest.mark.parametrize("si", range(len(SCORINGS)))
def test_hard_pairs_among_promising_ones(ctx, si):
    sc = SCORINGS[si]
    b = join(near_batch(300 + si, 3000), promising(si, 300))
    want, cells = run_oracle(b, sc)
    rng = np.random.default_rng(si)
    idx = rng.permutation(np.concatenate([np.arange(b.n), rng.integers(3000, b.n, 24000)]))
    many = type(b)(b.q_seq, b.q_off[idx], b.q_len[idx], b.t_seq, b.t_off[idx], b.t_len[idx], b.h0[idx])
    assert_same(run_gpu(ctx, many, sc), (want[idx], cells[idx]), f"{sc}")
