"""Every lane and slot count of the band engine, at the bands and batch sizes that take
it (tests/test_plan.py holds the plan to them), and row keys at the edge of their range:
every pair equals the CPU oracle (integer DP: the tolerance is zero)."""
import numpy as np
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.band_shapes import KEY_EDGES, SHAPES
from tests.gpu_util import assert_same, run_gpu, run_oracle
from tests.test_gpu_band_near import batch

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


def one_bucket(seed, n):
    """n pairs of 511-513 bases whose scores reach 512, over 150 different ones."""
    b = batch(seed, 400, (511, 512, 513), h0_top=300)
    ok = np.nonzero(b.h0 + np.minimum(b.q_len, b.t_len) >= 512)[0][:150]
    idx = np.random.default_rng(seed).choice(ok, n)
    return idx, b, type(b)(b.q_seq, b.q_off[idx], b.q_len[idx], b.t_seq, b.t_off[idx], b.t_len[idx],
                           b.h0[idx])


def check(ctx, seed, n, sc):
    idx, b, many = one_bucket(seed, n)
    want, cells = run_oracle(b, sc)
    assert_same(run_gpu(ctx, many, sc), (want[idx], cells[idx]), f"{sc} n={n}")


@pytest.mark.parametrize("w,n,P,K", SHAPES)
@pytest.mark.parametrize("zdrop", [0, 60])
def test_shape(ctx, w, n, P, K, zdrop):
    check(ctx, w + n, n, ScoringParams(w=w, zdrop=zdrop))


@pytest.mark.parametrize("sc,n,fits", KEY_EDGES, ids=str)
def test_row_keys_at_the_edge(ctx, sc, n, fits):
    check(ctx, n + sc.w, n, sc)
