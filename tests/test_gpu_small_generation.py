"""Small generations take both push phases in one launch (one to a few superphotons per warp): the same histories,
superphoton by superphoton, as the phase kernels that carry a large list.  FP64 and split geodesics agree
within the 1e-9 of the oracle parity and double-float ones within its 1e-8; FP32 weights within 1e-5
(some ten roundings a step over a few hundred steps, if two kernels round apart at all)."""
import numpy as np
import pytest

from helpers import compare_logs, gpu_model, requires_gpu
from paper_2602_13198_gb300 import synth

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("precision,geo,wtol", [("fp64", 1e-9, 1e-7), ("mixed", 1e-8, 1e-5), ("split", 1e-9, 1e-5)])
@pytest.mark.parametrize("kind", ["sphere", "torus"])
def test_small_lists_match_a_large_one(kind, precision, geo, wtol):
    if kind == "sphere":
        p, g = synth.scattering_sphere(0.1, n1=64, n2=32)
    else:
        p, g = synth.torus(a=0.9375, n1=64, n2=32, n3=8, R_high=10.0, dtype=np.float32, seed=5)
    n_s, seed = 3e4, 9
    m = gpu_model(p, g, precision=precision)
    st = m.run(n_s, seed)
    uids = np.linspace(0, st["n_total"] - 1, 12000).astype(np.int64)   # above the rule's largest list (4 per warp); may repeat
    big = m.trace(n_s, seed, uids, cap=1 << 18)
    for part in (uids[:1], uids[40:73], uids[6000:8500]):
        lg = m.trace(n_s, seed, part, cap=1 << 18)
        primaries = {int(u) for u in part}
        assert primaries <= {int(i) for i in lg["id"]}
        lo = big[np.isin(big["id"], lg["id"])]
        r = compare_logs(lg, lo)
        assert r["n"] == len(np.unique(lg["id"])) and r["unmatched"] == 0
        assert len(r["flips"]) <= 0.002 * len(lg) + 0.5
        assert r["worst"]["X"] <= geo and r["worst"]["K"] <= geo and r["worst"]["w"] <= wtol
