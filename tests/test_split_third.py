"""The double-precision RK4 combination x/3 + k f with the third in two parts,
fma(T, x, fma(k, f, TL x)), T + TL = 1/3 to 2^-108: replayed in exact rational
arithmetic with the constants as the kernel's source has them.  x/3 alone is the
correctly rounded quotient (no number of 53 bits has a third within 2^-106 of the
middle between two others), and with k f the sum is off by its last rounding
and by that of k f + TL x."""
import os
import re
from fractions import Fraction

import numpy as np

from test_div3 import round_to, samples

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_05447_gb300", "csrc",
                      "stencil.cuh")


def third():
    m = re.search(r"constexpr double T = 1\.0 / 3\.0, TL = ([0-9.e-]+);", open(SOURCE).read())
    return Fraction(1.0 / 3.0), Fraction(float(m.group(1)))


def rn(v):
    return round_to(v, 53)


def combined(x, k, f):
    T, TL = third()
    return rn(T * x + rn(k * f + rn(TL * x)))


def test_the_two_parts_are_a_third():
    T, TL = third()
    assert TL == rn(Fraction(1, 3) - T)
    assert abs(T + TL - Fraction(1, 3)) <= Fraction(2) ** -108


def test_a_third_alone_is_correctly_rounded():
    for x in samples(np.float64, 4000, 5):
        x = rn(x)
        assert combined(x, Fraction(0), Fraction(0)) == rn(x / 3), float(x)


def test_a_third_and_an_increment():
    rng = np.random.default_rng(9)
    for x in samples(np.float64, 2000, 7):
        x = rn(x)
        k, f = Fraction(float(rng.uniform(1e-4, 0.1))), rn(x * Fraction(float(rng.normal())))
        exact = x / 3 + k * f
        ulp = Fraction(2) ** -53
        assert abs(combined(x, k, f) - exact) <= ulp * abs(exact) + 2 * ulp * abs(k * f) + Fraction(2) ** -104 * abs(x)
