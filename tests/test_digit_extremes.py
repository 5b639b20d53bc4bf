"""Digit products at their largest sums: operands whose seven digits are all
127, so that every product of every weight adds up, against the exact integer
result."""

from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

X = float(sum(127 * 256 ** (6 - i) for i in range(7)) >> 2) / 2.0 ** 53   # 53 of the 55 bits: digits 127, ..., 127, 124


@pytest.mark.parametrize("m", [640, 4096, 20000])
@pytest.mark.parametrize("flip", [0, 1])
def test_all_digits_largest(gb, m, flip):
    """B - V e_0 (V^T B)_0 for constant V and B (flip: half of B negative, so
    that the sum cancels to its low digits' errors): the sum over the rows is
    exact but for FP32 roundings of the weights 6 and 7 beyond 2^24, at most
    2^-48.5 of the sum of magnitudes, and one rounding of the result."""
    n = nrhs = 128
    v = np.full((m, n), X)
    b = np.full((m, nrhs), X)
    if flip:
        b[m // 2:] = -X
    T = np.zeros((n, n))
    T[0, 0] = 1.0
    out = gb.to_colmajor(b)
    with gb.Context(0) as ctx:
        ctx.apply_qt(gb.to_colmajor(v), gb.to_colmajor(T), out, gb.GBQR_T_PANEL, n)
        assert ctx.sync()[0] == gb.GBQR_OK
    got = gb.to_numpy(out)
    x = Fraction(X)
    plus = m // 2 if flip else m
    w = x + x * x * (plus - 1) - x * x * (m - plus)          # V's unit diagonal at row 0
    size = x * x * m
    for i in (0, 1, m // 2, m - 1):
        vi = Fraction(1) if i == 0 else x
        want = Fraction(float(b[i, 0])) - vi * w
        err = abs(Fraction(float(got[i, 0])) - want)
        assert err <= vi * size * Fraction(2) ** -48 * Fraction(707, 1000) + 4 * Fraction(2) ** -53 * (abs(want) + vi * abs(w) + 1), (i, float(err / size))
