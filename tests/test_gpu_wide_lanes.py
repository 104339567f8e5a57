"""Pairs the band engine could take, on lanes: short queries under wide bands in large
batches.  Every pair equals the CPU oracle (integer DP: the tolerance is zero)."""
import numpy as np
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, run_gpu, run_oracle
from tests.test_gpu_band_near import batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [255, 256, 500])
def test_wide_bands_short_queries(w):
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = ScoringParams(5, -4, 8, 2, w, 60, -1)
    b = batch(w, 300, (110, 126, 127, 150, 254, 255, 400, 510, 511), h0_top=300)
    want, cells = run_oracle(b, sc)
    idx = np.random.default_rng(w).integers(0, b.n, 200_000)
    many = type(b)(b.q_seq, b.q_off[idx], b.q_len[idx], b.t_seq, b.t_off[idx], b.t_len[idx], b.h0[idx])
    ctx = xt.Context(0)
    assert_same(run_gpu(ctx, many, sc), (want[idx], cells[idx]), f"{sc}")
    ctx.close()
