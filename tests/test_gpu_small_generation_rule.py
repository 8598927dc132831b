"""The rule that sends a generation through both push phases in one launch: which path a list takes (the free-streaming
phase has a time of its own only in the phase kernels), and generations of scattered superphotons on either
side of it, whose histories are the same."""
import numpy as np
import pytest

from helpers import compare_logs, gpu_model, requires_gpu
from paper_2602_13198_gb300 import synth

pytestmark = [pytest.mark.gpu, requires_gpu]


def hot_torus():
    # as many scattered superphotons as primaries, so that its second generation is large or small with the first
    return synth.torus(a=0.9375, n1=64, n2=32, R_high=1.0, seed=5)


@pytest.mark.parametrize("precision", ["fp64", "mixed", "split"])
def test_path_taken(precision):
    import torch
    p, g = hot_torus()
    p = dict(p, scatter=0)   # the first generation alone
    m = gpu_model(p, g, precision=precision)
    n_s, seed = 6e4, 3
    total = m.run(n_s, seed, shard=0, n_shards=1)["n_total"]
    limit = 4 * (2 if precision == "mixed" else 8) * torch.cuda.get_device_properties(0).multi_processor_count
    assert total > 2 * limit
    for k, small in ((1, False), (total // limit + 2, True)):
        st = m.run(n_s, seed, shard=0, n_shards=k)
        assert (st["n_emit"] <= limit) == small
        assert (st["free_ms"] == 0.0) == small and st["grid_ms"] > 0.0


@pytest.mark.parametrize("precision,geo,wtol", [("fp64", 1e-9, 1e-7), ("mixed", 1e-8, 1e-5), ("split", 1e-9, 1e-5)])
def test_scattered_generations_on_both_sides(precision, geo, wtol):
    p, g = hot_torus()
    n_s, seed = 3e4, 7
    m = gpu_model(p, g, precision=precision)
    total = m.run(n_s, seed)["n_total"]
    uids = np.linspace(0, total - 1, 12000).astype(np.int64)
    big = m.trace(n_s, seed, uids, cap=1 << 18)
    assert (big["gen"] == 1).sum() > 6000   # above the rule's largest list
    part = uids[3000:3900]
    lg = m.trace(n_s, seed, part, cap=1 << 18)
    assert 300 < (lg["gen"] == 1).sum() < 1200
    r = compare_logs(lg, big[np.isin(big["id"], lg["id"])])
    assert r["unmatched"] == 0 and len(r["flips"]) <= 0.002 * len(lg) + 0.5
    assert r["worst"]["X"] <= geo and r["worst"]["K"] <= geo and r["worst"]["w"] <= wtol
