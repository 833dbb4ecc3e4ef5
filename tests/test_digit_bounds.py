"""The exactness bound of the tcgen05 digit products (csrc/pm_fxu.cuh): 128 real terms between two read-backs, accumulators that
start at zero, diagonals 0..2 read from the bits of a float below 2^22, the others converted below 2^24."""

import random
import struct

import pytest

from test_digit_products import F, NA, ND, split

TERMS = 128


def f32(x):
    return struct.unpack("f", struct.pack("f", float(x)))[0]


def test_diagonal_sums_fit_for_128_terms():
    """Rows and columns of 2-norm 1.5 (Taylor polynomials; propagators have 1): the top digits by Cauchy-Schwarz, the others at
    their extremes."""
    top = 1.5 * 2 ** 8 + 1
    for t in range(NA):
        bound = 0.0
        for i in range(ND):
            j = t - i
            if not 0 <= j < ND:
                continue
            if i == 0 and j == 0:
                bound += top * top
            elif i == 0 or j == 0:
                bound += top * 128 * TERMS ** 0.5
            else:
                bound += TERMS * 128 * 128
        assert bound < (2 ** 22 if t <= 2 else 2 ** 24), t


@pytest.mark.parametrize("kind", ["random", "low digits 127", "low digits -128", "alternating"])
def test_collected_sum_of_128_terms(kind):
    """The sum that the read-back forms (units of 2^-60) against the exact product: the dropped diagonals (t >= 8), the rounding
    of diagonals 6 and 7 in float and one rounding at the end."""
    rng = random.Random(3)
    ones = sum(1 << (8 * k) for k in range(6))

    def entry(k):
        if kind == "random":
            return rng.randint(-(1 << 53), 1 << 53)
        digit = {"low digits 127": 127, "low digits -128": -128}.get(kind, 127 if k % 2 else -128)
        return (rng.randint(-1, 1) << 48) + digit * ones

    for _ in range(20):
        a, b = ([entry(k) for k in range(TERMS)] for _ in range(2))
        da, db = [split(x) for x in a], [split(x) for x in b]
        assert all(sum(x << (48 - 8 * i) for i, x in enumerate(d)) == q for q, d in zip(a, da))
        v = [sum(x[i] * y[t - i] for x, y in zip(da, db) for i in range(ND) if 0 <= t - i < ND) for t in range(NA)]
        assert all(f32(x) == x for x in v) and all(abs(x) < 2 ** 22 for x in v[:3])
        w6 = round(f32(f32(v[6] + v[7] * 0.00390625) * 0.0625))
        q = v[5] * 16 + w6 + (v[4] << 12) + (v[3] << 20) + (v[2] << 28) + ((v[1] + v[0] * 256) << 36)
        exact = sum(x * y for x, y in zip(a, b))  # units of 2^(-2 F)
        unit = 1 << (2 * F - 60)
        assert abs(q * unit - exact) <= 0.6 * unit + 5 * TERMS * 128 * 128 * 2 ** 32
