"""Zone counts of the generation kernels at the edges of their launch rules (one or eight weight-table nodes per
CTA, one thread per zone or one warp per column, node counts that are not multiples of eight, a last chunk
and a last column that are not full): the same integers as the CPU oracle's, zone by zone."""
import numpy as np
import pytest

from helpers import gpu_model, oracle_model, requires_gpu
from paper_2602_13198_gb300 import synth

pytestmark = [pytest.mark.gpu, requires_gpu]

CASES = [
    # n1, n2, n3, n_nu, extra parameters
    (40, 16, 1, 200, {}),            # below one chunk
    (67, 31, 1, 2, {}),              # two nodes: both are trapezoid end points
    (96, 45, 1, 7, {}),              # fewer nodes than lanes of a zone
    (64, 33, 1, 201, dict(brems=1)), # general emissivity path, one node per CTA
    (48, 24, 37, 203, {}),           # columns longer than a warp, eight nodes per CTA, 203 = 25 x 8 + 3
    (30, 17, 32, 400, {}),           # shortest column that takes a warp
    (51, 22, 31, 333, {}),           # one below it: one thread per zone
]


@pytest.mark.parametrize("n1,n2,n3,n_nu,extra", CASES)
def test_zone_counts_equal_oracle(n1, n2, n3, n_nu, extra):
    dtype = np.float32 if n3 > 1 else np.float64
    p, g = synth.torus(a=0.5, n1=n1, n2=n2, n3=n3, R_high=10.0, n_nu=n_nu, dtype=dtype, seed=n1, **extra)
    n_s, seed = 2e5, 17
    m = gpu_model(p, g)
    st = m.run(n_s, seed, shard=0, n_shards=64)
    om = oracle_model(p, g)
    total = om.prepare(n_s, seed)
    assert st["n_total"] == total
    assert np.array_equal(m.zone_counts(), om.zones()["counts"])
