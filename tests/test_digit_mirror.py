"""CPU mirror of the digits of the digit-sliced FP64 product (k_matvec_ds.cu):
v = 2^(E+1) sum d_i 256^-i, |d_i| <= 128, |v| < 2^E, seven digits; products of
digits with i + j <= 8 kept.  In exact integers: the digits are in range and
give v back to half a unit of the last one; a product of two values is off by
at most 2^-51.4 (dropped) + 2^-53 (cut off) of the product of their groups'
maxima, a bound that values just above half a power of two with every lower
digit -128 nearly reach."""
import random
from fractions import Fraction

import pytest

ND = 7
DROPPED = Fraction(6 * 2 ** 14 * 4, 2 ** 72) * (1 + Fraction(1, 100))  # of 2^(Eg + Ex); i + j = 9, the rest below 1 %
CUT = Fraction(2, 2 ** 56) * (1 + Fraction(1, 2 ** 50))               # two values, half a unit 2^(E - 55) each


def digits(v, E):
    """v a Fraction below 2^E in size: the integer nearest to v 2^(55 - E) in balanced digits."""
    t = v * Fraction(2) ** (55 - E)
    n = abs(t)
    I = int(n + Fraction(1, 2))
    I = -I if t < 0 else I
    I += 0x808080808080
    d = [0] * ND
    for b in range(ND):
        d[ND - 1 - b] = ((I >> (8 * b)) & 0xff) - 128 if b < ND - 1 else I >> (8 * b)
    return d


def value(d, E):
    return Fraction(2) ** (E + 1) * sum(Fraction(x, 256 ** (i + 1)) for i, x in enumerate(d))


def kept(a, b):
    return sum(Fraction(a[i] * b[j] * 4, 256 ** (i + j + 2)) for i in range(ND) for j in range(ND) if i + j + 2 <= ND + 1)


def _values(rnd, n):
    for _ in range(n):
        yield Fraction(rnd.choice([-1, 1]) * rnd.randrange(2 ** 52, 2 ** 53), 2 ** 53)  # as large as the group's largest
        yield Fraction(rnd.choice([-1, 1]) * rnd.randrange(2 ** 53), 2 ** (53 + rnd.randrange(0, 60)))


WORST = value([65] + [-128] * 6, 0)


def test_digits_in_range_and_exact_to_half_a_unit():
    rnd = random.Random(1)
    for v in [WORST, -WORST, Fraction(0), Fraction(2 ** 53 - 1, 2 ** 53), Fraction(1, 2)] + list(_values(rnd, 400)):
        d = digits(v, 0)
        assert all(-128 <= x <= 128 for x in d), d
        assert abs(value(d, 0) - v) <= Fraction(1, 2 ** 56)


@pytest.mark.parametrize("seed", [1, 2])
def test_product_error_bound(seed):
    rnd = random.Random(seed)
    vs = list(_values(rnd, 60)) + [WORST, -WORST]
    worst = 0
    for g in vs:
        for x in vs:
            err = abs(kept(digits(g, 0), digits(x, 0)) - g * x)
            assert err <= DROPPED + CUT
            worst = max(worst, err)
    assert worst > 0


def test_bound_of_the_product_of_the_maxima_is_nearly_reached():
    err = abs(kept(digits(WORST, 0), digits(WORST, 0)) - WORST * WORST) / (WORST * WORST)
    assert Fraction(1, 2 ** 52) < err <= 4 * (DROPPED + CUT)  # maxima of at least half their power of two


def test_folded_sums_stay_exact_in_fp32_accumulators():
    # nine K-steps of 16 products of the largest digits, seven diagonals i + j = 8
    assert 9 * 16 * 7 * 128 * 128 < 2 ** 24
