"""A begun call keeps the schedule it was begun under: overrides and bucket schedules
set between xt_extend_batch_begin and _finish neither fail it nor change its results."""
import numpy as np
import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, run_oracle, to_dev
from tests.test_gpu_band_near import batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sc", [ScoringParams(), ScoringParams(w=600), ScoringParams(3, -4, 5, 2, 100, 0, -1)],
                         ids=str)
@pytest.mark.parametrize("before,after", [((0, 8), (32, 8)), ((0, 8), (1, 8)), ((16, 8), (0, 8)),
                                          ((1, 4), (32, 4))], ids=str)
def test_schedule_set_between_begin_and_finish(sc, before, after):
    import torch
    import paper_2301_09310_gb300 as xt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = batch(sc.w, 800, (1, 33, 100, 200, 400, 600, 900, 1500), h0_top=500)
    ctx = xt.Context(0)
    q, qo, ql, t, to, tl, h0 = args = to_dev(b, torch.device("cuda", 0))
    out = torch.zeros((b.n, 7), dtype=torch.int32, device="cuda")
    cells = torch.zeros(b.n, dtype=torch.int64, device="cuda")
    ctx.set_schedule(*before)
    st = xt.xt_extend_batch_begin(ctx.handle, q.data_ptr(), q.numel(), qo.data_ptr(), ql.data_ptr(),
                                  t.data_ptr(), t.numel(), to.data_ptr(), tl.data_ptr(), h0.data_ptr(),
                                  b.n, xt._scoring(sc), out.data_ptr(), cells.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
    assert st == xt.XT_OK
    ctx.set_schedule(*after)
    ctx.set_bucket_schedule(sc.w, 9, 16, 8)
    assert xt.xt_extend_batch_finish(ctx.handle) == xt.XT_OK, xt.xt_ctx_last_error(ctx.handle)
    torch.cuda.synchronize()
    want = run_oracle(b, sc)
    assert_same((out.cpu().numpy(), cells.cpu().numpy()), want, f"{sc}")
    out2, cells2 = ctx.extend(*args, sc)  # and the next call follows the new one
    torch.cuda.synchronize()
    assert_same((out2.cpu().numpy(), cells2.cpu().numpy()), want, f"{sc} after")
    ctx.close()
