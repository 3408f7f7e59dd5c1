"""The roofline that bench.py reports: never more instructions than the kernel
executes, and one floor beside it."""
import pytest

import bench


@pytest.mark.parametrize("measured", [bench.ANNEAL_MEASURED, bench.ANNEAL_D31_MEASURED])
def test_roofline_counts_what_is_executed(measured):
    rate, live, clocks, n_sm = 1.5e12, 0.7, {"sm_mhz": 2000.0}, 152
    rec = bench.roofline_record(rate, live, clocks, n_sm, measured=measured)
    peak = n_sm * 128 * 2000e6 / 1e12
    assert rec["peak"] == pytest.approx(peak) and rec["frac"] == pytest.approx(rec["achieved"] / peak)
    assert rec["achieved"] * 1e12 <= rate * measured["inst_per_attempt"] * (1 + 1e-12)
    assert rec["floor_frac"] == pytest.approx(rate * live * bench.FLOOR_INST / 1e12 / peak) and rec["floor_frac"] < rec["frac"]


def test_roofline_without_counters_or_clocks():
    rec = bench.roofline_record(1.5e12, 0.7, {"sm_mhz": 2000.0}, 152)
    assert rec["frac"] == rec["floor_frac"]
    rec = bench.roofline_record(1.5e12, 0.7, {"sm_mhz": None}, 152)
    assert rec["frac"] is None and rec["floor_frac"] is None
