"""The BWA-compatible extension with two pairs per lane (batches of many queries
of 33-256 bases): every pair equals the CPU oracle (integer DP: the tolerance is
zero) -- lengths at the edges of the row buffers and chunks, bands that cut live
columns off, scores on both sides of a byte, short and long targets, z-drop."""
import random

import numpy as np
import pytest

from paper_2301_09310_gb300.synth import BwaScoringParams

from tests.gpu_util import assert_same
from tests.test_gpu_band_near import batch
from tests.test_gpu_bwa import run_gpu_bwa, run_oracle_bwa

pytestmark = pytest.mark.gpu

COPIES = 1 << 18  # enough pairs for every lane class


@pytest.fixture(scope="module")
def ctx():
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = xt.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("sc", [
    BwaScoringParams(), BwaScoringParams(w=5, zdrop=0), BwaScoringParams(w=33, zdrop=20),
    BwaScoringParams(o_del=2, e_del=3, o_ins=5, e_ins=1, w=40, zdrop=20, end_bonus=0),
    BwaScoringParams(match=2, mismatch=-3, o_del=0, e_del=2, o_ins=1, e_ins=4, w=200, zdrop=0,
                     end_bonus=100, n_score=-2),
    BwaScoringParams(match=5, mismatch=-4, o_del=3, o_ins=3, w=100, zdrop=50, n_score=0),
], ids=str)
def test_two_pairs_per_lane(ctx, sc):
    lengths = (32, 33, 40, 63, 64, 65, 71, 72, 73, 95, 96, 120, 127, 128, 129, 136, 200, 247, 248, 249, 255, 256, 257)
    b = batch(sc.w + sc.match, 1500, lengths, h0_top=random.Random(sc.w).choice([40, 150, 300]))
    want, want_cells = run_oracle_bwa(b, sc)
    # many pairs over the same sequences, in an order that mixes them in the warps
    rng = np.random.default_rng(5)
    short = np.nonzero((b.q_len > 32) & (b.q_len <= 64))[0]
    idx = np.concatenate([rng.integers(0, b.n, COPIES), rng.choice(short, COPIES)])
    many = type(b)(b.q_seq, b.q_off[idx], b.q_len[idx], b.t_seq, b.t_off[idx], b.t_len[idx],
                   b.h0[idx])
    assert_same(run_gpu_bwa(ctx, many, sc), (want[idx], want_cells[idx]), f"{sc}")
