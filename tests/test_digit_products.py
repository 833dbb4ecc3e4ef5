"""The digit arithmetic of the FP64 products (csrc/pm_digits.cuh), restated in Python integers.

x = q 2^-56 is split into one 10-bit and six 8-bit balanced digits; a product sums the digit pairs i + j <= 7 of
32 real terms in f32 accumulators that start at 1.5 * 2^23 (diagonals 0..5) or 0 (6, 7).
"""

import random
import struct

import pytest

ND, NA, F = 7, 8, 56
BIAS = 0x0200808080808080


def split(q):
    """Digits 0 (top) .. 6 of a fixed-point number, as the kernel extracts them."""
    x = (q + BIAS) & 0xFFFFFFFFFFFFFFFF
    return [((x >> 48) & 0x3FF) - 512] + [((x >> (8 * k)) & 0xFF) - 128 for k in (5, 4, 3, 2, 1, 0)]


def f32(x):
    return struct.unpack("f", struct.pack("f", float(x)))[0]


def values(kind, rng):
    top = (1 << (F + 1)) - 1
    return {
        "unitary": lambda: rng.randint(-(1 << 56), 1 << 56),
        "edge": lambda: rng.choice([-top - 1 + (1 << 48), top - (1 << 48), 1 << 56, -(1 << 56), 0, 1, -1]),
        "half": lambda: rng.choice([-1, 1]) * ((1 << 54) + rng.choice([-1, 0, 1]) * 0x80808080808),
    }[kind]


@pytest.mark.parametrize("kind", ["unitary", "edge", "half"])
def test_split_is_exact_and_digits_are_f16_integers(kind):
    rng = random.Random(1)
    draw = values(kind, rng)
    for _ in range(2000):
        q = draw()
        d = split(q)
        assert -512 <= d[0] <= 511 and all(-128 <= x <= 127 for x in d[1:])
        assert sum(x << (48 - 8 * i) for i, x in enumerate(d)) == q


def test_accumulators_stay_exact_in_the_worst_case():
    """32 real terms of rows and columns of 2-norm 1.5: every diagonal sum fits the 2^22 window in which the biased
    f32 accumulator counts in ones (top digits by Cauchy-Schwarz, the others at their extremes)."""
    top = 1.5 * 2 ** 8 + 1  # a row's top digits have 2-norm 1.5 * 2^8, plus rounding
    for t in range(NA):
        bound = 0.0
        for i in range(ND):
            j = t - i
            if not 0 <= j < ND:
                continue
            if i == 0 and j == 0:
                bound += top * top
            elif i == 0 or j == 0:
                bound += top * 128 * 32 ** 0.5
            else:
                bound += 32 * 128 * 128
        assert bound < (2 ** 22 if t < 6 else 2 ** 24), t


@pytest.mark.parametrize("kind", ["unitary", "half"])
@pytest.mark.parametrize("fine", [False, True])
def test_collected_sum_is_close_to_the_exact_product(kind, fine):
    """The collected 32-term sum is within the dropped diagonals (t >= 8) and one rounding of the exact one."""
    rng = random.Random(2)
    draw = values(kind, rng)
    for _ in range(200):
        a = [draw() // 4 for _ in range(32)]
        b = [draw() // 4 for _ in range(32)]
        da, db = [split(x) for x in a], [split(x) for x in b]
        v = [sum(x[i] * y[t - i] for x, y in zip(da, db) for i in range(ND) if 0 <= t - i < ND) for t in range(NA)]
        exact = sum(x * y for x, y in zip(a, b))  # units 2^-112
        if fine:  # rounded to 2^-60
            w6 = round(f32(v[6] + v[7] / 256.0))
            low = v[5] * 256 + w6
            o = ((low + 7 + ((low >> 4) & 1)) >> 4) + (v[3] * 256 + v[4]) * 4096 + (v[1] * 256 + v[2]) * (1 << 28) + (v[0] << 44)
            assert abs(low) < 2 ** 31 and abs(v[3] * 256 + v[4]) < 2 ** 31 and abs(v[1] * 256 + v[2]) < 2 ** 31
            err = o * 2 ** 52 - exact
            assert abs(err) <= 0.6 * 2 ** 52 + 5 * 32 * 128 * 128 * 2 ** 32 + 2 ** 48
        else:  # rounded to 2^-56
            w5 = v[5] + round((v[6] + v[7] / 256.0) / 256.0)
            lo, mid, hi = v[4] * 256 + w5, v[2] * 256 + v[3], v[0] * 256 + v[1]
            assert abs(lo) < 2 ** 31 and abs(mid) < 2 ** 31
            o = mid * 65536 + lo + (hi << 32)
            err = o * 2 ** 56 - exact
            assert abs(err) <= 0.6 * 2 ** 56 + 5 * 32 * 128 * 128 * 2 ** 32


def test_halving_is_unbiased():
    """Ties to even: over consecutive numbers the rounding errors of x / 2 cancel."""
    err = [((x + ((x >> 1) & 1)) >> 1) * 2 - x for x in range(-64, 64)]
    assert sum(err) == 0 and max(abs(e) for e in err) == 1
