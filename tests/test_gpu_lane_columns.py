"""The one-lane engine sweeps only the columns that can be alive and stops past
the query's end: every pair equals the CPU oracle (integer DP: the tolerance is
zero), on scorings that move the live columns' limits (cheap and dear gaps, free
extension, high matches), with warps that mix short-lived and long-lived pairs."""
import random

import pytest

from paper_2301_09310_gb300.synth import ScoringParams

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
    c.set_schedule(1, 8)
    yield c
    c.close()


@pytest.mark.parametrize("sc", [
    ScoringParams(), ScoringParams(w=300, zdrop=0), ScoringParams(w=20, zdrop=10),
    ScoringParams(1, -4, 0, 1, 200, 0, -1), ScoringParams(1, -4, 126, 1, 200, 100, -1),
    ScoringParams(2, -3, 2, 2, 100, 30, -2), ScoringParams(3, 0, 1, 0, 100, 0, 0),
    ScoringParams(1, -9, 3, 40, 100, 0, -9), ScoringParams(1, -1, 1, 1, 250, 0, -1),
], ids=str)
def test_live_columns(ctx, sc):
    lengths = (1, 2, 15, 16, 17, 31, 33, 62, 63, 100, 126, 130, 200, 254, 300)
    b = batch(random.Random(sc.w).randint(1, 999), 600, lengths, h0_top=60)
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), f"{sc}")
