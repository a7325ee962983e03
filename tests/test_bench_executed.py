"""CPU test of the bench's account of what the tile kernels execute: a fraction
of a pipe stays a utilisation (at most 1) where the ALU roofline of the
sum-factorised work no longer is one."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

PEAKS = {"p64": 1.255, "p32": 79.7, "pdf": 6.70, "clocks": {"sm_mhz": 2070.0}}


@pytest.mark.parametrize("form,ms", [("fp64", 48.0), ("mixed", 16.7)])
def test_executed_work_is_a_utilisation(form, ms):
    r = bench.roofline_form(form, 10_100_000, 5, {"newton": ms}, 2 * ms, PEAKS, 6794.8, 1.02e7, 4.0e8, 6.7e8)
    assert "no utilisation" in r["frac_note"]
    x = r["executed"]
    if form == "mixed":
        assert x["frac"] is None
        return
    assert r["frac"] > 1.0 and 0.5 < x["frac"] <= 1.0
    assert x["ms"] == pytest.approx(1e3 * 10_100_000 * x["ops_per_point"] / (1.255e12 / 2))
    assert x["ops_per_point"] == 2 * (83 * 8 + 60) + 2 * (30 * 8 + 40)
