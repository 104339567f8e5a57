"""bench.py gives a fraction of a peak only for cells the kernels evaluate."""
import bench

RATES = {"sms": 152, "alu_pipe": 64.0, "issue": 100.0, "cell_update_cells": 30.0}


def test_no_fraction_for_proven_cells():
    r = bench.int_roofline(1e12, 100.0, RATES, 1900.0, evaluated=False)
    assert r["frac"] is None and r["achieved"] is None
    assert r["definition_rate"]["updates_per_s"] == 1e13
    r = bench.int_roofline(1e12, 1000.0, RATES, 1900.0)
    assert 0 < r["frac"] < 1 and r["achieved"] > 0
