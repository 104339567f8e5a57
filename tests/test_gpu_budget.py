"""Memory budgets: what near passes leave needs a buffer of its own, held only while a
budget has room for it; a call that fits without it is accepted and gives the same
results.  The budgets are those of 5 bytes a pair (calls in capacity classes of powers
of two) and fixed counters."""
import numpy as np
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, run_gpu, run_oracle
from tests.test_gpu_band_near import batch
from tests.test_gpu_near_promise import join, promising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xt():
    import torch
    import paper_2301_09310_gb300 as mod
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return mod


def tiled(b, n, seed):
    idx = np.random.default_rng(seed).integers(0, b.n, n)
    return idx, type(b)(b.q_seq, b.q_off[idx], b.q_len[idx], b.t_seq, b.t_off[idx], b.t_len[idx], b.h0[idx])


@pytest.mark.parametrize("spare", [0, 1 << 19, 1 << 20, 4 << 20])
def test_near_pairs_within_a_budget(xt, spare):
    # a band whose rings lie in shared memory: the workspace is all the call needs
    sc = ScoringParams(w=20)
    b = join(promising(3, 300), batch(3, 200, (20, 60, 120, 200, 250)))
    want, cells = run_oracle(b, sc)
    n = 1 << 18
    idx, many = tiled(b, n, 1)
    ctx = xt.Context(0, mem_budget_bytes=5 * n + (190 << 10) + spare)
    for rep in range(2):
        assert_same(run_gpu(ctx, many, sc), (want[idx], cells[idx]), f"spare {spare}")
    ctx.close()


def test_buffer_given_back_to_a_larger_call(xt):
    sc = ScoringParams(w=20)
    b = join(promising(5, 300), batch(5, 200, (20, 60, 120, 200, 250)))
    want, cells = run_oracle(b, sc)
    n = 1 << 18
    # room for the first call with its buffer, or the second without
    ctx = xt.Context(0, mem_budget_bytes=10 * n + (190 << 10))
    for size in (n, 2 * n, n):
        idx, many = tiled(b, size, size)
        assert_same(run_gpu(ctx, many, sc), (want[idx], cells[idx]), f"{size}")
    ctx.close()


def test_narrow_band_first_within_a_budget(xt):
    sc = ScoringParams(w=600)
    b = batch(7, 300, (511, 700, 1023, 2000))
    want = run_oracle(b, sc)
    ctx = xt.Context(0, mem_budget_bytes=5 * 1024 + (190 << 10))
    for rep in range(2):
        assert_same(run_gpu(ctx, b, sc), want, "w = 600")
    ctx.close()
