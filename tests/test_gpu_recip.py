"""The reciprocal of the stabilisation's pivots against exact arithmetic.

With e the relative error of the approximation it starts from, the series is
cut at e^3 and the result is rounded once; at 20 bits that is 2^-60, 2^-7 of
an ulp at most, and the rounding of the correction adds less than as much:
|y - 1/x| <= (0.5 + 2^-6) ulp(y).  Outside the approximation's range it is the
division: half an ulp, infinities and NaN included."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2303_13403_gb300 import pqmc

pytestmark = pytest.mark.gpu


def recip(x):
    import torch
    torch.cuda.set_device(0)
    d_x = torch.tensor(x, dtype=torch.float64, device="cuda")
    d_y = torch.zeros_like(d_x)
    torch.cuda.synchronize()
    pqmc.test_recip(len(x), d_x.data_ptr(), d_y.data_ptr())
    return d_y.cpu().numpy()


def test_against_exact_reciprocals():
    rng = np.random.default_rng(1)
    m = np.concatenate([1 + rng.random(3000), 1 + 2.0 ** -rng.uniform(1, 52, 500), 2 - 2.0 ** -rng.uniform(0, 52, 500)])
    m = np.clip(m, 1.0, np.nextafter(2.0, 1.0)) * rng.choice([-1.0, 1.0], m.size)
    # exponent fields on both sides of the range's ends, and all between
    e = rng.integers(1, 2045, m.size)
    e[:600] = np.repeat([59, 60, 61, 1979, 1980, 1981], 100)
    x = np.ldexp(m, e - 1023)
    y = recip(x)
    for xi, yi in zip(x, y):
        ulp = Fraction(float(np.spacing(abs(yi))))
        assert abs(Fraction(float(yi)) - 1 / Fraction(float(xi))) <= (Fraction(1, 2) + Fraction(1, 64)) * ulp, (xi, yi)


def test_special_values():
    x = np.array([np.inf, -np.inf, np.nan, 0.0, -0.0, 5e-324, 2.0 ** -1022, 1.0, -2.0, 2.0 ** 1023])
    with np.errstate(divide="ignore", over="ignore"):
        assert np.array_equal(recip(x), 1.0 / x, equal_nan=True)
