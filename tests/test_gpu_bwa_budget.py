"""BWA-compatible calls within a memory budget of 5 bytes a pair and 32 KB of counters."""
import pytest

from paper_2301_09310_gb300.synth import BwaScoringParams

from tests.gpu_util import assert_same
from tests.test_gpu_band_near import batch
from tests.test_gpu_bwa import run_gpu_bwa, run_oracle_bwa

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xt():
    import torch
    import paper_2301_09310_gb300 as mod
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return mod


@pytest.mark.parametrize("spare", [0, 32 << 10])
def test_bwa_within_a_budget(xt, spare):
    sc = BwaScoringParams()
    b = batch(9, 1000, (1, 30, 33, 64, 65, 128, 129, 200, 256, 257, 600))
    want = run_oracle_bwa(b, sc)
    ctx = xt.Context(0, mem_budget_bytes=1024 + 4096 + 33024 + spare)
    assert_same(run_gpu_bwa(ctx, b, sc), want, "bwa")
    ctx.close()
