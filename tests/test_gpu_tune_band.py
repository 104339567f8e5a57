"""The autotuner times the band engine too: results under its table equal the CPU
oracle, the table keeps the choice, and a tuned context is not left behind by the
built-in rule."""
import json

import pytest

from paper_2301_09310_gb300 import synth
from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, run_gpu, run_oracle, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xt():
    import torch
    import paper_2301_09310_gb300 as mod
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return mod


@pytest.fixture(scope="module")
def table(xt, tmp_path_factory):
    path = str(tmp_path_factory.mktemp("tune") / "tuning.json")
    ctx = xt.Context(0)
    ctx.autotune(ScoringParams(), j_max=11, cells_per_trial=1e9, table_path=path)
    ctx.close()
    return path


def test_the_table_keeps_the_band_engine(xt, table):
    e = json.load(open(table))["entries"][0]
    by_j = {b["j"]: b for b in e["buckets"]}
    # a few thousand queries of 511 bases and longer: 510 GCUPS on bands, 271 on groups
    assert by_j[10]["band_s"] == 1 and by_j[11]["band_s"] == 1
    assert all(b["P"] >= 1 and b["Ps"] >= 1 for b in e["buckets"])


@pytest.mark.parametrize("n", [3000, 40000])
@pytest.mark.parametrize("sc", [ScoringParams(), ScoringParams(5, -4, 8, 2, 100, 100, -1)], ids=str)
def test_results_under_the_table(xt, table, n, sc):
    b = synth.generate(synth.WORKLOADS["c5_stream"], n=n, first=77)
    ctx = xt.Context(0)
    ctx.load_tuning(table)
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), f"{sc} n={n}")
    ctx.close()


def test_a_tuned_stream_keeps_up(xt, table):
    # the tuner and the built-in rule choose among the same engines; half as much again
    # is for choices its synthetic trials of single buckets get wrong
    import torch
    wl = synth.WORKLOADS["c5_stream"]
    args = to_dev(synth.generate(wl, n=20000), torch.device("cuda", 0))
    ms = []
    for tuned in (True, False):
        ctx = xt.Context(0)
        if tuned:
            ctx.load_tuning(table)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for rep in range(8):
            t0.record()
            ctx.extend(*args, wl.scoring)
            t1.record()
            torch.cuda.synchronize()
            if rep > 1:
                best = min(best, t0.elapsed_time(t1))
        ms.append(best)
        ctx.close()
    assert ms[0] < 1.5 * ms[1], ms
