"""The one-lane engine's looks for live columns and rows, on both sides of the bands
where they are switched on (gap_extend x w of 24 and 80) and where gaps extend for
nothing: every pair equals the CPU oracle (integer DP: the tolerance is zero)."""
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, run_gpu, run_oracle
from tests.test_gpu_band_near import batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [4, 8, 16])
@pytest.mark.parametrize("sc", [
    ScoringParams(w=23), ScoringParams(w=24), ScoringParams(w=79, zdrop=20), ScoringParams(w=80),
    ScoringParams(1, -4, 6, 3, 26, 0, -1), ScoringParams(1, -4, 2, 3, 27, 100, -1),
    ScoringParams(2, -3, 1, 23, 1, 0, -2), ScoringParams(2, -3, 1, 40, 2, 30, -2),
    ScoringParams(1, -4, 6, 0, 200, 0, -1), ScoringParams(1, -4, 500, 1000, 70, 0, -1),
], ids=str)
def test_live_looks(sc, rows):
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = xt.Context(0)
    ctx.set_schedule(1, rows)
    lengths = (1, 2, 15, 16, 17, 31, 33, 62, 63, 100, 126, 130, 200, 254, 300, 511, 700)
    b = batch(sc.w + sc.gap_extend, 500, lengths, h0_top=60)
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), f"{sc} {rows}")
    ctx.close()
