"""Errors of the transport's FP64 functions against extended precision (numpy's long double), over the arguments
that the kernels pass: within the bounds that follow from their roundings, and no further off than the
functions that they took the place of."""
import numpy as np
import pytest

from helpers import requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]
LD = np.longdouble
EPS = 2.0 ** -52
N = 300000


def evaluate(which, x):
    from paper_2602_13198_gb300 import build, mc
    build.build()
    return mc.selftest_math(which, x)[0].astype(LD)


def decades(rng, lo, hi):
    return 10.0 ** rng.uniform(lo, hi, N)


def ulp(ref):
    return np.spacing(np.abs(ref.astype(np.float64)))


def test_rsqrt():
    rng = np.random.default_rng(1)
    x = np.concatenate([decades(rng, -280, 280), rng.uniform(1.0, 4.0, N)])
    ref = 1 / np.sqrt(x.astype(LD))
    # the final rounding; the third-order remainder is below 0.02 ulp
    assert (np.abs(evaluate(18, x) - ref) <= 0.55 * ulp(ref)).all()


def test_exp():
    rng = np.random.default_rng(2)
    x = np.concatenate([-decades(rng, -16, 2.8), rng.uniform(-300, 20, N), rng.uniform(-1, 1, N)])
    ref = np.exp(x.astype(LD))
    # half an ulp each for the table and the result, 0.03 for the remainder of the series and the reduced argument
    assert (np.abs(evaluate(11, x) - ref) <= 1.05 * ulp(ref)).all()


@pytest.mark.parametrize("which,ulps,absolute", [(20, 1.1, 0.0), (21, 0.52, 1e-17)])
def test_log(which, ulps, absolute):
    rng = np.random.default_rng(3)
    near = decades(rng, -15, -1)
    x = np.concatenate([decades(rng, -14, 3), rng.uniform(0, 1, N), rng.uniform(0.9, 1.1, N), 1 - near, 1 + near,
                        decades(rng, -300, 300), 1 + (np.arange(2048) + 0.5) / 2048, [1.0, 2.0, 0.5]])
    ref = np.log(x.astype(LD))
    y = evaluate(which, x)
    # half an ulp of the result; within 1 % of x = 1 the variates' form has another half of the series' leading term,
    # and the coordinates' form the remainder of its shorter series
    assert (np.abs(y - ref) <= ulps * ulp(ref) + absolute).all()
    assert y[-3] == 0.0 and (y[x < 1.0] <= absolute).all()


def test_bremsstrahlung_rate():
    rng = np.random.default_rng(4)
    th = np.concatenate([decades(rng, -3, 3), [1.0, np.nextafter(1.0, 0.0)]])
    t, pi = th.astype(LD), LD("3.14159265358979323846264338327950288")
    c = LD(7.2973525693e-3) * LD(9.1093837015e-28) * LD(2.99792458e10) ** 3
    ei, ee = LD(1.25) * LD(6.6524587321e-25) * c, LD(2.8179403262e-13) ** 2 * c
    with np.errstate(all="ignore"):
        cold = (4 * np.sqrt(2 * t / pi ** 3) * (1 + LD(1.781) * t ** LD(1.34)) * ei + 20 / (9 * np.sqrt(pi))
                * (44 - 3 * pi ** 2) * t * np.sqrt(t) * (1 + LD(1.1) * t + t * t - LD(1.25) * t * t * np.sqrt(t)) * ee)
        hot = (9 * t / (2 * pi) * (np.log(LD(1.123) * t + LD(0.48)) + LD(1.5)) * ei
               + 24 * t * (np.log(LD(1.1232) * t) + LD(1.28)) * ee)
    ref = np.where(th < 1.0, cold, hot)
    # five roundings of half an ulp on the longest path of the larger term, half of one from its constant
    assert np.abs(evaluate(19, th) / ref - 1).max() <= 3 * EPS
