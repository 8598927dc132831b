"""FP64 coefficients where the plasma leaves the ordinary range, on a spinning torus: bands of zones without a
field, with a field so weak that plasma beta is some 1e140, and with a density and energy for which the
temperature's numerator and denominator leave the range of their product.  Histories through them equal the
oracle's.  (A field whose beta^2 overflows is refused as a non-finite zone state.)"""
import numpy as np
import pytest

from helpers import compare_logs, gpu_model, oracle_model, requires_gpu
from paper_2602_13198_gb300 import synth

pytestmark = [pytest.mark.gpu, requires_gpu]


def banded(band, **over):
    p, g = synth.torus(a=0.9375, n1=64, n2=48, R_high=10.0, seed=31, M_unit=1e18, **over)
    prim = np.array(g["prim"], dtype=np.float64).reshape(8, 64, 48)
    rows = np.arange(48) // 4 % 3 == 1     # four rows of every twelve: the inner ones are free of the blend
    if band == "no_field":
        prim[2:5][:, :, rows] = 0.0
    elif band == "tiny_field":
        prim[2:5][:, :, rows] *= 1e-70
    elif band == "refused_field":
        prim[2:5][:, :, rows] *= 1e-150
    else:
        prim[:2][:, :, rows] *= 1e-165
        prim[2:5][:, :, rows] = 0.0
    return p, dict(g, prim=prim.reshape(8, -1))


@pytest.mark.parametrize("band", ["no_field", "tiny_field", "tiny_plasma"])
@pytest.mark.parametrize("brems", [0, 1])
def test_histories_equal_the_oracles(band, brems):
    p, g = banded(band, brems=brems)
    gm, om = gpu_model(p, g), oracle_model(p, g)
    n_s, seed = 2e4, 8
    total = om.prepare(n_s, seed)
    assert gm.run(n_s, seed)["n_total"] == total
    assert np.array_equal(gm.zone_counts(), om.zones()["counts"])
    uids = np.unique(np.linspace(0, total - 1, 500).astype(np.int64))
    lg, lo = gm.trace(n_s, seed, uids), om.run(uids=uids, log=True)["log"]
    r = compare_logs(lg, lo)
    assert len(lg) > len(uids)             # scattered superphotons too
    assert len(r["flips"]) <= 0.01 * r["n"] and r["unmatched"] <= 0.01 * r["n"]
    assert np.isfinite(lg["w"]).all()
    assert r["worst"]["X"] < 1e-9 and r["worst"]["K"] < 1e-9 and r["worst"]["w"] < 1e-6


def test_field_beyond_the_range_is_refused():
    from paper_2602_13198_gb300 import mc
    p, g = banded("refused_field")
    with pytest.raises(mc.MCError):
        gpu_model(p, g).run(2e4, 8)
