"""The integer combination of the Cholesky products' levels (no GPU): from the exact level
sums acc_2 .. acc_9 (integers below 2^21) the epilogue forms pairs h1 = 2^7 acc_2 + acc_3
.. l2 = 2^7 acc_8 + acc_9 in 32 bits, T = 2^33 h1 + 2^19 h2 + 2^5 l1 + round(2^-9 l2) in
64 bits, and rounds 2^e0 T to 53 bits (half away from zero).  Against the exact sum
2^(e0 + 54 - 35) sum_L acc_L 2^(7 (5 - L)): half a unit of T's last place plus the
rounding to a double."""
from fractions import Fraction
import random

import pytest


def level_sum(h1, h2, l1, l2, e0):
    for v in (h1, h2, l1, l2):
        assert -2 ** 31 <= v < 2 ** 31
    t = h1 * 2 ** 33 + h2 * 2 ** 19 + l1 * 32 + ((l2 + 256) >> 9)
    assert abs(t) < 2 ** 63
    if t == 0:
        return Fraction(0)
    m0, lz = abs(t), 64 - abs(t).bit_length()
    m = m0 << lz
    r = (m >> 11) + ((m >> 10) & 1)
    assert 2 ** 52 <= r <= 2 ** 53  # the carry moves into the exponent field
    v = Fraction(r) * Fraction(2) ** (e0 + 11 - lz)
    return v if t > 0 else -v


@pytest.mark.parametrize("seed", range(4))
def test_level_sum_is_the_exact_sum_rounded(seed):
    rng = random.Random(seed)
    for k in range(2000):
        size = 2 ** rng.choice([0, 3, 10, 20, 21])
        acc = {L: rng.randint(-size, size) for L in range(2, 10)}
        if k == 0:
            acc = {L: -2 ** 21 for L in acc}  # the largest magnitudes
        if k == 1:
            acc = {L: 2 ** 21 for L in acc}
        e0 = rng.randint(-900, 900)
        exact = sum(Fraction(a) * Fraction(2) ** (7 * (5 - L)) for L, a in acc.items()) * Fraction(2) ** (e0 + 19)
        got = level_sum(128 * acc[2] + acc[3], 128 * acc[4] + acc[5], 128 * acc[6] + acc[7], 128 * acc[8] + acc[9], e0)
        unit = Fraction(2) ** e0  # T's last place
        assert abs(got - exact) <= unit / 2 + abs(exact) * Fraction(1, 2 ** 53) + unit * Fraction(1, 2 ** 53)
