"""The bench line's second fraction: the work model with the surface tests that the cell masks leave."""

import pytest

import bench


def test_fraction_with_the_tests_made():
    st = {"particles": 40, "flights": 1000, "collisions": 960, "attempts": 1200}
    e = bench.roofline_entry([st], [2.0], 16, {"ffma": 1e9}, tests=1.31)
    work = 1000 * (116 + 25 * 1.31) + 1200 * 135 + 960 * 78 + 40 * 280
    assert e["tests_per_flight"] == 1.31
    assert e["frac_with_tests_made"] == pytest.approx(work / 2e-3 / 1e9, rel=1e-12)
    assert e["frac_with_tests_made"] < e["frac"]
    assert "frac_with_tests_made" not in bench.roofline_entry([st], [2.0], 7, {"ffma": 1e9})
    assert set(bench.TESTS_PER_FLIGHT) <= set(bench.WORKLOADS)
