"""The launch plan of a batched call, from pair counts alone (the planner is host
code: no GPU needed)."""
import json
import os
import subprocess

import pytest

from paper_2301_09310_gb300 import build
from paper_2301_09310_gb300.synth import ScoringParams

PACKED, NARROW, WIDE, HUGE, NEAR, BAND = range(6)


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    lib = build.build()
    exe = str(tmp_path_factory.mktemp("plan") / "plan_probe")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "plan_probe.cu")
    subprocess.run([build.nvcc(), *build.ARCH_FLAGS, "-O1", "-std=c++17", f"-I{build.INCLUDE}",
                    f"-I{build.CSRC}", src, "-o", exe, lib, "-Xlinker", "-rpath", "-Xlinker",
                    os.path.dirname(lib)], check=True, capture_output=True)

    def run(cases):
        text = []
        for c in cases:
            sc, counts, tuned = c.get("sc", ScoringParams()), c["counts"], c.get("tuned", ())
            n = c.get("n", sum(counts.values()))
            text.append(f"{sc.w} {sc.match} {sc.mismatch} {sc.gap_open} {sc.gap_extend} {sc.zdrop} "
                        f"{sc.n_score} {n} {c.get('hopeful', 0)} {c.get('budget', 0)} {int(c.get('near_ok', True))} {len(tuned)} "
                        f"{len(counts)}")
            text += [" ".join(map(str, t)) for t in tuned]
            text += [f"{cls} {j} {v}" for (cls, j), v in counts.items()]
        r = subprocess.run([exe], input="\n".join(text) + "\n", capture_output=True, text=True, check=True)
        out = [json.loads(line) for line in r.stdout.splitlines()]
        assert len(out) == len(cases)
        return out

    return run


def reads(n, share_near, hope, long_share=0.4):
    """n pairs of up to 254 bases the diagonal pass left, so many of them near pairs."""
    near, rest = int(n * share_near), int(n * (1 - share_near))
    return {"counts": {(NEAR, 8): int(near * long_share), (NEAR, 7): near - int(near * long_share),
                       (PACKED, 7): rest // 2, (PACKED, 6): rest - rest // 2},
            "hopeful": int(near * hope), "n": n}


@pytest.mark.parametrize("n", [30_000, 130_000, 900_000])
def test_near_pass_only_where_reads_promise_it(plan, n):
    none, noisy, good = plan([reads(n, 0.5, 0.0), reads(n, 0.5, 0.05), reads(n, 0.7, 0.57)])
    assert none["near_pairs"] == 0 and noisy["near_pairs"] == 0
    assert good["near_pairs"] == int(n * 0.7)


def test_near_pass_not_before_lanes_within_one_wave(plan):
    # one length bucket, a single wave of lanes: the pass would only delay them ...
    lanes, sooner, waves = plan([
        {"counts": {(NEAR, 7): 37_000}, "hopeful": 20_000, "n": 55_000},
        # ... unless what it leaves goes to a sooner engine, or there are more waves
        {"counts": {(NEAR, 8): 45_000}, "hopeful": 21_400, "n": 55_000},
        {"counts": {(NEAR, 7): 200_000}, "hopeful": 110_000, "n": 300_000}])
    assert lanes["near_pairs"] == 0
    assert sooner["near_pairs"] == 45_000 and sooner["launches"][0]["engine"] == "band"
    assert waves["near_pairs"] == 200_000


def test_ctas_for_the_pairs_the_near_pass_leaves(plan):
    few, many = plan([reads(200_000, 0.7, 0.6), reads(200_000, 0.7, 0.25)])
    for a, b in zip(few["launches"], many["launches"]):
        assert a["engine"] == b["engine"]
        if a["engine"] == "band":
            assert b["grid"] > 1.3 * a["grid"]


def full_plan(rng, flags, j_top):
    """Counts in every class and bucket that classify could fill, of sizes that keep
    neighbouring buckets' launches apart."""
    counts = {}
    for j in range(5, j_top + 1):
        f = flags[j]
        classes = [WIDE] if not f & 4 and not f & 1 else [HUGE]
        if j <= 17 and not f & 1:
            classes.append(NARROW)
            if f & 2:
                classes += [PACKED] + ([NEAR] if j <= 9 else [])
        if j <= 17 and f & 16:
            classes.append(BAND)
        for cls in classes:
            if rng.random() < 0.97:
                counts[cls, j] = rng.choice([1, 50, 3000, 8191, 8192, 9000, 40_000, 100_000])
    return counts


def test_every_class_and_bucket_gets_its_launch(plan):
    import random
    rng = random.Random(3)
    scs = [ScoringParams(w=w) for w in (5, 20, 60, 100, 300, 511, 512, 700, 1000, 1900, 4000)]
    schedules = [(1, 4), (1, 8), (1, 16), (2, 8), (4, 4), (8, 8), (16, 4), (32, 8), (32, 4)]
    shapes = []
    for k in range(800):
        tuned = []
        if k % 3 == 0:
            tuned = [(j, s, *rng.choice(schedules)) for j in range(5, 22) for s in (0, 1)
                     if rng.random() < 0.5 and j <= 9]
        shapes.append({"sc": rng.choice(scs), "counts": {(WIDE, 5): 1}, "n": rng.choice([50_000, 1 << 20]),
                       "tuned": tuned})
    flags = [p["flags"] for p in plan(shapes)]
    for c, f in zip(shapes, flags):
        c["counts"] = full_plan(rng, f, 21)
        c["hopeful"] = rng.choice([0, 60_000])
    plans = plan(shapes)
    assert not any(p["bad"] for p in plans)
    for c, p in zip(shapes, plans):  # every non-empty (class, bucket) is drained once
        for (cls, j), v in c["counts"].items():
            runs = [L for L in p["launches"] if not L["near_hw"]
                    and (L["cls"] == cls or L["cls2"] == cls) and L["j_lo"] <= j <= L["j_hi"]]
            assert sorted(L["lanes_left"] for L in runs) in ([0], [0, 1]), (c["sc"], cls, j, runs)


def test_what_a_narrow_band_leaves_gets_the_engines_narrow_pairs_take(plan):
    sc = ScoringParams(w=512, zdrop=400)
    few, many, tight = plan([
        {"sc": sc, "counts": {(BAND, 12): 3000}},
        {"sc": sc, "counts": {(BAND, 12): 60_000}},
        {"sc": sc, "counts": {(BAND, 12): 60_000}, "budget": 64 << 20}])
    # a CTA of the group launch for every four pairs, up to the GPU's own number
    narrow, group = few["launches"]
    assert narrow["near_hw"] > 0 and group["engine"] == "group" and group["after_prev"]
    assert group["P"] == 32 and group["grid"] >= 456 and narrow["lanes_from"] == 0
    # where lanes would take all of them, lanes or groups by the number left
    narrow, group, lane = many["launches"]
    assert (group["engine"], lane["engine"]) == ("group", "lane")
    assert lane["lanes_left"] and 60_000 / 4 <= narrow["lanes_from"] <= 60_000 / 2
    # no rings beyond the budget
    assert [L["engine"] for L in tight["launches"]] == ["band", "group"]
    assert tight["launches"][0]["lanes_from"] == 0 and tight["pool"] <= 64 << 20


def test_without_a_buffer_for_what_near_passes_leave(plan):
    plans = plan([
        {"counts": {(NEAR, 8): 50_000, (NEAR, 7): 60_000}, "hopeful": 62_000, "n": 400_000, "near_ok": False},
        {"sc": ScoringParams(w=600), "counts": {(BAND, 11): 3000, (BAND, 14): 200}, "near_ok": False},
        {"sc": ScoringParams(w=9000), "counts": {(BAND, 14): 300}, "near_ok": False}])
    for p in plans:
        assert not p["bad"] and p["near_pairs"] == 0
        assert not any(L["near_hw"] or L["after_prev"] or L["lanes_left"] for L in p["launches"])
    assert plans[1]["launches"][0]["j_hi"] == 14 and plans[1]["launches"][-1]["j_lo"] == 11
    assert plans[2]["launches"][0]["global_ring"]


@pytest.mark.parametrize("name,mean,sc", [
    ("mixed reads", {(NEAR, 8): 3200, (NEAR, 7): 8200, (PACKED, 7): 1300, (PACKED, 6): 2900, (PACKED, 5): 1200},
     ScoringParams()),
    ("mixed reads", {(NEAR, 8): 64_000, (NEAR, 7): 148_000, (PACKED, 7): 21_000, (PACKED, 6): 50_000,
                     (PACKED, 5): 22_000}, ScoringParams()),
    ("small calls", {(NEAR, 8): 70, (NEAR, 7): 190, (PACKED, 6): 70, (PACKED, 5): 31}, ScoringParams()),
    ("stream", {(BAND, 11): 1100, (BAND, 10): 3600, (PACKED, 9): 1500, (NEAR, 9): 6900, (NEAR, 8): 10_100,
                (NEAR, 7): 5300, (PACKED, 7): 600, (PACKED, 6): 1300, (PACKED, 5): 1150}, ScoringParams()),
    ("wide bands", {(BAND, 11): 1100, (BAND, 10): 3600, (NEAR, 8): 10_100, (PACKED, 6): 1300},
     ScoringParams(w=600)),
])
def test_calls_of_like_size_share_a_plan(plan, name, mean, sc):
    # batches of up to 7% fewer pairs than one, as a stream of reads forms them
    import random
    rng = random.Random(11)
    cases = []
    for _ in range(200):
        size = rng.uniform(0.93, 1.0)
        counts = {k: max(1, round(rng.gauss(v * size, (v * size) ** 0.5))) for k, v in mean.items()}
        near = sum(v for (cls, _), v in counts.items() if cls == NEAR)
        cases.append({"sc": sc, "counts": counts, "n": 1 << 16, "hopeful": round(near * 0.56)})
    signatures = {p["signature"] for p in plan(cases)}
    assert len(signatures) <= 8, len(signatures)


def test_band_shapes_by_band_and_count(plan):
    from tests.band_shapes import KEY_EDGES, SHAPES
    plans = plan([{"sc": ScoringParams(w=w), "counts": {(BAND, 10): n}} for w, n, _, _ in SHAPES])
    for (w, n, P, K), p in zip(SHAPES, plans):
        (L,) = p["launches"]
        assert (L["engine"], L["P"], L["R"]) == ("band", P, K), (w, n)
    # where they do not fit: no band pairs, or a narrower band first
    for (sc, n, fits), p in zip(KEY_EDGES, plan([{"sc": sc, "counts": {(BAND, 10): n}}
                                                 for sc, n, _ in KEY_EDGES])):
        whole = p["flags"][10] & 16 and p["launches"][0]["near_hw"] == 0
        assert bool(whole) == fits, sc


@pytest.mark.parametrize("w,j,n,lanes", [(255, 8, 60_000, False), (256, 8, 60_000, True), (256, 9, 60_000, True),
                                         (256, 10, 60_000, False), (400, 8, 30_000, False),
                                         (191, 7, 60_000, False), (192, 7, 60_000, True)])
def test_short_queries_under_wide_bands_go_to_lanes(plan, w, j, n, lanes):
    # scores beyond the packed lanes': one bucket of the band engine's pairs
    (p,) = plan([{"sc": ScoringParams(5, -4, 8, 2, w, 100, -1), "counts": {(BAND, j): n}, "n": 100_000}])
    (L,) = p["launches"]
    assert L["engine"] == ("lane" if lanes else "band")
