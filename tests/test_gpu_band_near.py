"""The narrow band tried first where the whole band is too wide for the band
engine, and the band engine on small batches of short queries: every pair equals
the CPU oracle (integer DP: the tolerance is zero).  Lengths at the edges of the
buckets, whose narrow bands differ, losses on both sides of the bounds, repeats
whose off-diagonal paths nearly match, short and long targets, z-drop stops."""
import random

import pytest

from paper_2301_09310_gb300.synth import ScoringParams

from tests.gpu_util import assert_same, batch_from_lists, run_gpu, run_oracle

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


def batch(seed, n, lengths, h0_top=40):
    rng = random.Random(seed)
    qs, ts, hs = [], [], []
    for _ in range(n):
        ql = rng.choice(lengths)
        if rng.random() < 0.2:
            unit = [rng.randint(0, 3) for _ in range(rng.choice([1, 3, 60, 200]))]
            base = (unit * 4000)[:4000]
        else:
            base = [rng.randint(0, 3) for _ in range(4000)]
        q, p = [], 0
        sub = rng.choice([0, 0.005, 0.02, 0.03, 0.05])
        gap, top = rng.choice([(0, 1), (0.001, 3), (0.004, 8), (0.002, 150)])
        while len(q) < ql:
            r = rng.random()
            if r < sub:
                q.append(rng.choice([0, 1, 2, 3, 3, 4]))
                p += 1
            elif r < sub + gap / 2:
                q.extend(rng.randint(0, 3) for _ in range(rng.randint(1, top)))
            elif r < sub + gap:
                p += rng.randint(1, top)
            else:
                q.append(base[p % 4000])
                p += 1
        q = q[:ql]
        if rng.random() < 0.1:
            k = rng.randint(0, ql - 1)
            q[k:] = [rng.randint(0, 3) for _ in range(ql - k)]
        tl = max(1, ql + rng.choice([0, 0, 0, -1, 1, -ql // 3, 40, 127, 128, 129, 600]))
        qs.append(q)
        ts.append(base[:tl])
        hs.append(rng.choice([1, 20, rng.randint(1, h0_top)]))
    return batch_from_lists(qs, ts, hs)


@pytest.mark.parametrize("sc", [
    ScoringParams(w=4000, zdrop=0), ScoringParams(w=700, zdrop=100), ScoringParams(w=512, zdrop=30),
    ScoringParams(2, -3, 2, 2, 900, 0, -2), ScoringParams(3, 0, 1, 0, 600, 0, 0),
    ScoringParams(1, -1, 1, 1, 2000, 0, -1), ScoringParams(5, -4, 0, 3, 1000, 60, 0),
], ids=str)
@pytest.mark.parametrize("lengths", [(511, 512, 700, 1021, 1022), (1023, 1024, 2045),
                                     (2047, 2500)], ids=str)
def test_narrow_band_first(ctx, sc, lengths):
    b = batch(lengths[0] + sc.w, 120, lengths)
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), f"{sc} {lengths}")


@pytest.mark.parametrize("sc", [
    ScoringParams(), ScoringParams(w=8), ScoringParams(w=31, zdrop=5), ScoringParams(w=63, zdrop=0),
    ScoringParams(w=127), ScoringParams(w=128, zdrop=20), ScoringParams(w=224), ScoringParams(w=511),
    ScoringParams(2, -3, 2, 2, 60, 20, -2), ScoringParams(3, 0, 1, 0, 100, 0, 0),
    ScoringParams(1, -4, 127, 0, 40, 100, -1),
], ids=str)
@pytest.mark.parametrize("n", [1, 150, 5000])
def test_small_batches_of_short_queries(ctx, sc, n):
    b = batch(n + sc.w, n, (1, 2, 7, 8, 30, 31, 62, 63, 90, 126, 127, 200, 254, 255, 400, 510, 511))
    assert_same(run_gpu(ctx, b, sc), run_oracle(b, sc), f"{sc} {n}")
