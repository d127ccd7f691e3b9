"""The FP64 reference step divides by cs2 = RN(1/3) and two_cs4 =
RN(2 cs2 cs2) in two operations, fma(x, c, x * (c * 2^-54)) with c = 3 and
4.5 (lbm_ref.cuh).  Host check that this is the IEEE division: exact rational
arithmetic, rounded once, against Python's correctly rounded division, on
random mantissas and on those next to the ties of the proof, at exponents
down to the threshold below which the kernel divides literally."""
import random
from fractions import Fraction as F

import pytest

CS2 = 1.0 / 3.0
TWO_CS4 = 2.0 * CS2 * CS2


def _two_ops(x, c):
    t = x * (c * 2.0 ** -54)  # one rounding
    return float(F(x) * F(c) + F(t))  # one rounding


@pytest.mark.parametrize("y, c", [(CS2, 3.0), (TWO_CS4, 4.5)])
def test_two_operation_division_is_the_ieee_division(y, c):
    r = random.Random(11)
    m = [r.getrandbits(52) | 1 << 52 for _ in range(20000)]
    for base in (1 << 52, (1 << 53) - 1, (1 << 54) // 3, (3 << 54) // 9, (1 << 56) // 9):
        m += [v for v in range(base - 300, base + 300) if 1 << 52 <= v < 1 << 53]
    for e in (0, -52, -400, -757 - 52, -963 - 52, 900):
        for v in m[:: 1 if e == 0 else 17]:
            x = v * 2.0 ** e
            assert _two_ops(x, c) == x / y, (x.hex(), y)
            assert _two_ops(-x, c) == -x / y


def test_high_word_zero_is_exact():
    """Below 2^-1042 (high word zero) the kernel also takes the product form."""
    for v in (1, 2, 3, 5, 12345, (1 << 32) - 1):
        x = v * 2.0 ** -1074
        assert _two_ops(x, 3.0) == x / CS2
