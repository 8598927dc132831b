"""The benchmark's printed line stays within a few kilobytes, so that a reader who keeps only the end of its output can
parse it: contract keys unchanged, the forms reduced to rate, ratio, spectrum error and fraction of peak."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

ST = {"n_steps": 3363874310, "n_steps_grid": 1363874310, "n_iters": 3374161858, "n_iters_grid": 1374161858,
      "n_events": 8663677, "grid_ms": 3599.5871276855467, "free_ms": 1035.2435245513916, "init_ms": 306.8607990145683,
      "transport_ms": 4941.69, "n_emit": 22560991, "n_child": 8663677}


def test_line_is_short_and_keeps_the_contract():
    def entry(ref=None):
        e = dict(bench.form_entry(ST, 5000.123456, ref), roofline=bench.fp64_roofline(ST, "kerr", 3, 1.0573e12, "k", point=True))
        if ref:
            e["spectrum_error"] = {"total_luminosity_rel_max": 1.0123e-7, "total_luminosity_rel_median": 1.0e-7,
                                   "bins_within_max_1pct_3sigma": 1.0, "bins_compared": 1024, "within_1pct": True}
        return e

    conf = {f: entry(None if f == "plain_fp64" else 6.1e6)
            for f in ("plain_fp64", "mixed", "mixed_surrogate", "split", "split_surrogate")}
    for f in conf.values():
        f["per_tau"] = {str(t): dict(f) for t in (1e-4, 1e-3, 1e-2, 1e-1)}
    line = {"metric": bench.METRIC, "value": 6181523.123456, "unit": bench.UNIT, "config": {"workload": bench.WORKLOAD_C4},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "e2e": {"value": 6.1e6, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
            "roofline": conf["plain_fp64"]["roofline"], "cpu_baseline": None, "gpu_launches": 380,
            "forms": dict({"peaks": {"fp64_tflops": 1.057}},
                          **{"c%d" % i: dict(conf, workload=bench.WORKLOAD_C4) for i in range(5)}),
            "detail": {"step_ms": [622.123456789] * 20, "generate_ms": [4.87] * 20, "wall_s": 12.7}}
    full, short = json.dumps(line), bench.compact(line)
    text = json.dumps(short)
    assert len(full) > 40000 and len(text) < 8000
    for k in line:
        assert k in short
        if k not in ("forms", "detail"):
            assert short[k] == line[k]
    f = short["forms"]["c0"]["mixed"]
    assert f["x_fp64"] > 0 and f["within_1pct"] is True and 0 < f["frac"] < 1
    assert short["detail"]["step_ms"] == [622.123] * 20
    assert json.loads(full)["forms"]["c0"]["mixed"]["roofline"]   # the argument itself is not cut
