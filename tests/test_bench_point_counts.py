"""The benchmark's operation counts of the Kerr-Schild point form, which the FP64 kernels run, and the fraction
of peak formed from them: every step of both push phases over the time of both."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

ST = {"n_steps": 3_000_000, "n_steps_grid": 1_000_000, "n_iters": 3_100_000, "n_iters_grid": 1_050_000, "n_events": 500,
      "grid_ms": 2.0, "free_ms": 1.0, "init_ms": 0.5, "transport_ms": 3.5, "n_emit": 10_000, "n_child": 500}


def test_point_form_counts():
    # step size 8, position 25, point 36 (29), blend 150 or 80, plasma 78 (72), coefficients 62, depths 11
    assert bench.ops_grid_step("kerr", 3, True) == 370
    assert bench.ops_grid_step("kerr", 2, True) == 300
    assert bench.ops_grid_step("schw", 2, True) == 287
    assert bench.ops_geodesic_step("kerr", True) == 69 and bench.ops_geodesic_step("schw", True) == 62
    assert bench.ops_pass("kerr", True) == 82 and bench.ops_pass("schw", True) == 58


def test_fp64_fraction_counts_what_both_phases_run():
    r = bench.fp64_roofline(ST, "kerr", 3, 1.0e12, "k", point=True)
    ops = 370 * 1_000_000 + 69 * 2_000_000 + 82 * 3_100_000 + 30 * 500
    assert r["frac"] == pytest.approx(ops / 3.0e-3 / 1.0e12)
    # a small generation's free steps move from one phase's time to the other's: the fraction stays
    moved = dict(ST, grid_ms=3.0, free_ms=0.0)
    assert bench.fp64_roofline(moved, "kerr", 3, 1.0e12, "k", point=True)["frac"] == pytest.approx(r["frac"])


def test_split_fraction_takes_the_form_of_the_spin():
    k = bench.split_roofline(ST, "kerr", 1.0e12, "k")
    assert k["frac"] == pytest.approx((69 * 3_000_000 + 14 * 1_000_000 + 82 * 3_100_000) / 3.0e-3 / 1.0e12)
    s = bench.split_roofline(ST, "schw", 1.0e12, "k")
    assert s["frac"] == pytest.approx((102 * 3_000_000 + 63 * 3_100_000) / 3.0e-3 / 1.0e12)
