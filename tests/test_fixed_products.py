"""The digit products of the complex128 substitutions, restated in Python integers: a
factor row as 64-bit fixed point in radix 256, a vector chain as balanced digits, orders
0..7 kept.  Pins that every order sum stays an integer FP32 holds, what the dropped orders
and the fixed-point rounding cost, and that planted mistakes are seen."""
import math
import random
from fractions import Fraction

import pytest

COLS = 32


def _exponent(values):
    return max(math.frexp(v)[1] for v in values)


def _matrix_digits(x, e):
    y = int(Fraction(x) * Fraction(2) ** (63 - e)) + (1 << 63)
    b = [(y >> (8 * (7 - i))) & 255 for i in range(8)]
    b[0] -= 128
    return b


def _vector_digits(x, e):
    y = int(Fraction(x) * Fraction(2) ** (62 - e)) + 0x8080808080808080
    assert 0 <= y < 1 << 64
    return [((y >> (8 * (7 - i))) & 255) - 128 for i in range(8)]


def _chain(row, vec, orders=8):
    """Sum of row[c] vec[c] through digits: (value, largest partial order sum in modulus)."""
    e, f = _exponent(row), _exponent(vec)
    D, worst = [0] * orders, 0
    for a, x in zip(row, vec):
        da, dx = _matrix_digits(a, e), _vector_digits(x, f)
        for g in range(orders):
            for i in range(g + 1):
                D[g] += da[i] * dx[g - i]
                worst = max(worst, abs(D[g]))
    total = sum(d << (8 * (7 - g)) for g, d in enumerate(D))
    return Fraction(total) * Fraction(2) ** (e + f - 69), worst


@pytest.mark.parametrize("spread", [0, 20])
def test_chain_is_closer_than_fp64(spread):
    rng = random.Random(spread)
    for _ in range(40):
        row = [rng.uniform(-1, 1) * 2.0 ** -rng.uniform(0, spread) for _ in range(2 * COLS)]
        vec = [rng.uniform(-1, 1) * 2.0 ** rng.uniform(-spread, 0) for _ in range(2 * COLS)]
        got, worst = _chain(row, vec)
        exact = sum(Fraction(a) * Fraction(x) for a, x in zip(row, vec))
        scale = Fraction(2) ** (_exponent(row) + _exponent(vec))
        # 2 COLS products: 2^-63 and 2^-62 fixed-point rounding, seven digit pairs of 255 x 128 in each
        # dropped order from 256^-8 on
        assert abs(got - exact) <= scale * 2 * COLS * Fraction(1, 2 ** 58)
        assert worst < 1 << 24


def test_order_sums_fit_fp32_at_the_digits_extremes():
    # every digit pair at 255 x -128, real and imaginary part of 32 columns, eight pairs in order 7
    assert 2 * COLS * 8 * 255 * 128 < 1 << 24


def test_a_dropped_order_and_a_wrong_offset_are_seen():
    rng = random.Random(1)
    row = [rng.uniform(-1, 1) for _ in range(2 * COLS)]
    vec = [rng.uniform(-1, 1) for _ in range(2 * COLS)]
    exact = sum(Fraction(a) * Fraction(x) for a, x in zip(row, vec))
    tight = Fraction(2 * COLS, 2 ** 58)
    assert abs(_chain(row, vec)[0] - exact) <= tight
    seven = _chain(row, vec, orders=7)[0] * Fraction(2) ** 8
    assert abs(seven - exact) > tight
    digits = _vector_digits(0.3, 0)
    value = sum(Fraction(d, 1) * Fraction(256) ** (7 - i) for i, d in enumerate(digits))
    assert value == int(Fraction(0.3) * Fraction(2) ** 62)
    shifted = sum(Fraction(d + 1, 1) * Fraction(256) ** (7 - i) for i, d in enumerate(digits))
    assert shifted != value
