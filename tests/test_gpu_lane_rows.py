"""The one-lane engine's look for live rows alone (gap_extend x w from 24 to 47) and
with live columns (from 48): every pair equals the CPU oracle (integer DP: the
tolerance is zero)."""
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, run_gpu, run_oracle
from tests.test_gpu_band_near import batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sc", [
    ScoringParams(w=47), ScoringParams(w=48, zdrop=0), ScoringParams(2, -3, 3, 4, 11, 60, -1),
    ScoringParams(1, -4, 0, 4, 12, 0, -1), ScoringParams(1, -1, 1, 1, 40, 20, 0),
], ids=str)
def test_live_rows(sc):
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = xt.Context(0)
    ctx.set_schedule(1, 8)
    b = batch(sc.w, 700, (1, 15, 16, 17, 33, 62, 63, 100, 126, 130, 254, 300, 511), h0_top=60)
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), f"{sc}")
    ctx.close()
