"""Launch accounting and DP timing take in the pass that settles pairs on their
diagonal."""
import numpy as np
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import batch_from_lists, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,passes", [(8192, 1), (1000, 0)])
def test_diagonal_pass_is_counted_and_timed(n, passes):
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(2)
    t = [rng.integers(0, 4, 150).tolist() for _ in range(50)]
    b = batch_from_lists([t[k % 50][:100] for k in range(n)], [t[k % 50] for k in range(n)], [30] * n)
    ctx = xt.Context(0)
    args = to_dev(b, torch.device("cuda", 0))
    for timing in (False, True):
        ctx.set_timing(timing)
        ctx.stats()
        for rep in range(3):
            ctx.extend(*args, ScoringParams(w=40))
        st = ctx.stats()
        engines = st["dp_launches"] - 3 * passes
        # every pair is its diagonal: the pass settles all of them, or an engine runs
        assert engines == 0 if passes else engines >= 3
        assert st["calls"] == 3 and st["launches"] == 12 + st["dp_launches"]
        assert st["timed_calls"] == (3 if timing else 0)
        assert (st["dp_ms"] > 0.003) == timing  # 1 us a pass at the least
    ctx.close()
