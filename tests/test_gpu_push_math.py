"""The FP64 push kernels' elementary functions and one-step reciprocals against CUDA's on the device, over the
arguments the kernels pass and at the joints of their tables.  Bounds: a rounding or two more than the
library functions they replace (3 ulp, as for the smaller-table forms)."""
import numpy as np
import pytest

from helpers import requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]
ULP = 2.2e-16
RNG = np.random.default_rng(21)


def both(which, x):
    from paper_2602_13198_gb300 import build, mc
    build.build()
    return mc.selftest_math(which, x)


def rel(y, ref):
    ok = np.isfinite(ref) & (ref != 0.0)
    return np.abs(y[ok] / ref[ok] - 1.0).max()


def test_exp():
    j = np.arange(-700, 701) * (np.log(2.0) / 512.0)   # the joints between table nodes
    x = np.concatenate([RNG.uniform(-707.9, 707.9, 200000), RNG.uniform(-8, 8, 200000), j, np.nextafter(j, 1e9),
                        [0.0, 708.0, -708.0, 709.5, -745.0]])
    y, ref = both(11, x)
    assert rel(y, ref) <= 3 * ULP and y[-5] == 1.0


def test_log():
    x = np.concatenate([10.0 ** RNG.uniform(-300, 300, 200000), RNG.uniform(0.5, 2.0, 100000),
                        1.0 + np.arange(1024) / 1024.0, np.nextafter(1.0 + np.arange(1, 1024) / 1024.0, 0.0),
                        [1.0, 1e-310, 0.0, 1e308]])
    y, ref = both(12, x)
    ok = np.isfinite(ref)
    # one rounding of the exponent's part and one of the table's, each within half an ulp of |ref| + ln 2
    assert np.all(np.abs(y[ok] - ref[ok]) <= 2 * ULP * (np.abs(ref[ok]) + 0.7))
    assert y[-2] == ref[-2] and y[-3] == ref[-3]


@pytest.mark.parametrize("which", [13, 14])
def test_sincospi(which):
    k = np.arange(-2048, 3073) / 2048.0
    x = np.concatenate([RNG.uniform(0.0, 0.5, 200000), RNG.uniform(-2.0, 3.0, 100000), k, np.nextafter(k, 9.0),
                        10.0 ** RNG.uniform(-300, -3, 1000)])
    y, ref = both(which, x)
    assert np.abs(y - ref).max() <= 3 * ULP
    if which == 13:   # relative near the pole
        small = (np.abs(x) < 0.01) & (x != 0.0)
        assert rel(y[small], ref[small]) <= 3 * ULP


def test_expm1():
    j = np.arange(0, 1200) * (np.log(2.0) / 512.0)
    x = np.concatenate([10.0 ** RNG.uniform(-300, 2.8, 300000), RNG.uniform(0.0, 2.0, 200000), j, np.nextafter(j, 9.0),
                        [0.0, 707.9, 708.0, 800.0, -0.25, -3.0]])
    y, ref = both(15, x)
    # above ln 2 the subtraction costs at most one bit (e^x / (e^x - 1) <= 2)
    assert rel(y[:-2], ref[:-2]) <= 6 * ULP
    assert y[-6] == 0.0 and np.isinf(y[-3]) and rel(y[-2:], ref[-2:]) <= 3e-15


def test_sixth_root():
    x = np.concatenate([10.0 ** RNG.uniform(-29.9, 29.9, 300000), [1.0, 64.0, 1e-30, 1e30, 1e-40, 1e40]])
    y, ref = both(16, x)
    assert rel(y, ref) <= 10 * ULP


@pytest.mark.parametrize("which", [17, 18])
def test_reciprocals(which):
    x = np.concatenate([10.0 ** RNG.uniform(-290, 290, 300000), RNG.uniform(0.5, 4.0, 200000), 2.0 ** np.arange(-100, 101)])
    y, ref = both(which, x)
    assert rel(y, ref) <= 2 * ULP


def test_brems_rate():
    x = np.concatenate([10.0 ** RNG.uniform(-6, 3, 200000), [1.0, np.nextafter(1.0, 0.0), 1e-30, 1e-300, 1e6]])
    y, ref = both(19, x)
    # all terms are positive: some ten roundings, and 3 ulp of an exponent of at most 1.34 |ln x| in a term
    # that x^1.34 makes small
    assert rel(y, ref) <= 20 * ULP
