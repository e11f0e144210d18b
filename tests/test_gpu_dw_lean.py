"""Pins of the lean double-word forms that the edge flux and its VJP run on,
alone and in either lane of the packed FP32 instructions, against exact rational
references of the same split inputs.

u = 2^-24.  The split leaves |l| < 2u |h|; the lean forms leave their low words
unnormalised.  First-order bounds, each rounding counted at the size of what it
rounds (the error-free transformations are exact):
  x + y           the sum of the low words (2u^2) and its addition to the error
                  of the high words (3u^2):                5u^2 (|x| + |y|)
  x y             x_l y_l left out (4u^2), two fused multiply-adds (3u^2, 5u^2):
                                                          12u^2 |x y|
  x y + c         the same, and the low words added to the sums' error:
                                                          23u^2 |x y| + 5u^2 |c|
  (x + c) y + c   an operand with a low word up to 3u (|x| + |c|):
                                          33u^2 (|x| + |c|) |y| + 5u^2 |c|
  1/x, 1/sqrt(x)  correction of up to 2^-22 in FP32, three roundings: 2^-44; the
                  residual of the second has four more terms: 2^-43
  high word       of a normalised sum: half an ulp, 2^-24 |x + y| (1 + 2^-22)
The bounds below carry one u^2 more for the second-order terms.  In the fourth
quarter of the rows c = -x y (1 + d), |d| <= 1e-6, so that the product sum cancels.
"""
from decimal import Decimal, getcontext
from fractions import Fraction

import numpy as np
import pytest

from paper_2102_12933_gb300 import fdu

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

U2 = Fraction(1, 2 ** 48)
N = 2048
FORMS = ["", ".0", ".1"]


def _values(rng, n, positive=False):
    x = 10.0 ** rng.uniform(-6, 4, n) * rng.uniform(0.5, 2.0, n)
    return x if positive else x * rng.choice([-1.0, 1.0], n)


@pytest.fixture(scope="module")
def rows():
    rng = np.random.default_rng(77)
    x, y = _values(rng, N), _values(rng, N)
    y[: N // 4] = -x[: N // 4] * (1.0 + rng.uniform(-1e-6, 1e-6, N // 4))
    k = np.arange(3 * N // 4, N, 2)
    y[k + 1] = -x[k] * y[k] * (1.0 + rng.uniform(-1e-6, 1e-6, k.size))
    x, y = fdu.check_dw("split", x), fdu.check_dw("split", y)
    return x, y, [Fraction(v) for v in x], [Fraction(v) for v in y]


def _check(z, exact, bound):
    worst = max(float(abs(Fraction(a) - b) / c) for a, b, c in zip(z, exact, bound))
    assert worst <= 1.0, worst


@pytest.mark.parametrize("form", FORMS)
def test_sum_product_and_their_chains(rows, form):
    x, y, fx, fy = rows
    c = [fy[i ^ 1] for i in range(N)]
    A = abs
    _check(fdu.check_dw("lean_add" + form, x, y), [a + b for a, b in zip(fx, fy)],
           [6 * U2 * (A(a) + A(b)) for a, b in zip(fx, fy)])
    _check(fdu.check_dw("lean_mul" + form, x, y), [a * b for a, b in zip(fx, fy)],
           [13 * U2 * A(a * b) for a, b in zip(fx, fy)])
    _check(fdu.check_dw("lean_fma" + form, x, y), [a * b + d for a, b, d in zip(fx, fy, c)],
           [U2 * (24 * A(a * b) + 6 * A(d)) for a, b, d in zip(fx, fy, c)])
    _check(fdu.check_dw("lean_chain" + form, x, y), [(a + d) * b + d for a, b, d in zip(fx, fy, c)],
           [U2 * (34 * (A(a) + A(d)) * A(b) + 6 * A(d)) for a, b, d in zip(fx, fy, c)])


@pytest.mark.parametrize("form", FORMS)
def test_high_word_of_a_normalised_sum(rows, form):
    x, y, fx, fy = rows
    v = [Fraction(a) for a in fdu.check_dw("lean_add" + form, x, y)]
    _check(fdu.check_dw("lean_high" + form, x, y), v, [A * (Fraction(1, 2 ** 24) + 4 * U2) or 1 for A in map(abs, v)])


@pytest.mark.parametrize("form", FORMS)
def test_reciprocals(form):
    x = fdu.check_dw("split", _values(np.random.default_rng(9), N, positive=True))
    f = [Fraction(v) for v in x]
    _check(fdu.check_dw("lean_recip" + form, x), [1 / v for v in f], [Fraction(1, 2 ** 44) / v for v in f])
    getcontext().prec = 60
    worst = 0.0
    for s, v in zip(fdu.check_dw("lean_rsqrt" + form, x), x):
        exact = Decimal(1) / Decimal(v).sqrt()
        worst = max(worst, float(abs(Decimal(s) - exact) / exact))
    assert worst <= 2.0 ** -43, worst


@pytest.mark.parametrize("op", ["lean_add", "lean_mul", "lean_fma"])
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e300])
def test_non_finite_operands_stay_non_finite(op, value):
    x = np.array([1.5, value, 2.0, 3.0])
    for form in FORMS:
        z = fdu.check_dw(op + form, x, np.ones(4))
        assert list(np.isfinite(z)) == [True, False, True, True]


def test_bad_arguments():
    with pytest.raises(fdu.FduError):
        fdu.check_dw("lean_add", np.ones(3), np.ones(3))  # rows come in pairs
