"""FP64 products whose digits are at their extremes: exponents with all low digits 127 and, on the diagonal of X^2, equal signs in
every term."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def generator(d):
    """Hermitian G with |Re| = |Im| = a in every entry (the diagonal real), a a multiple of 2^-56 whose six low base-256 digits
    are 127 and whose top digit brings the 1-norm near 0.3."""
    top = max(0, int(0.3 / (d * 2 ** 0.5) * 256 - 0.5))
    a = ((top << 48) + 127 * sum(1 << (8 * k) for k in range(6))) * 2.0 ** -56
    up = np.triu(np.ones((d, d)), 1)
    return a * np.ones((d, d)) + 1j * a * (up - up.T)


@pytest.mark.parametrize("scale", [1.0, 2.0])
@pytest.mark.parametrize("d", [5, 8, 12, 16, 17, 32, 33, 64, 128, 144])
def test_slice_with_extreme_digits(d, scale):
    """One slice against a Taylor series in extended precision (some columns).  The products, coefficients and the conversion to
    double each round by 2^-57 to 2^-54 of one, squarings double what went before them: 2^-52 each.  (An inexact sum on the
    diagonals 0..4 would be off by 2^-48 or more.)"""
    import torch

    from paper_2108_07126_gb300.binding import Propagator

    G = generator(d) * scale
    prop = Propagator(0)
    try:
        prop.set_hamiltonians(torch.as_tensor(G), torch.zeros(1, d, d, dtype=torch.complex128), "midpoint")
        prop.set_controls(torch.zeros(1, 1, dtype=torch.float64), 1.0, 1)
        U = prop.propagate("fp64").cpu().numpy()
        s = prop.stats()["max_squarings"]
    finally:
        prop.close()
    cols = sorted({0, 1, d // 2, d - 1})
    re, im = G.real.astype(np.longdouble), G.imag.astype(np.longdouble)
    x, y = np.zeros((d, len(cols)), np.longdouble), np.zeros((d, len(cols)), np.longdouble)  # the k-th term
    x[cols, np.arange(len(cols))] = 1
    sx, sy = x.copy(), y.copy()
    for k in range(1, 30):  # -i (re + i im) (x + i y) / k
        x, y = (re @ y + im @ x) / k, (im @ y - re @ x) / k
        sx, sy = sx + x, sy + y
    err = max(np.max(np.abs(U.real[:, cols] - sx)), np.max(np.abs(U.imag[:, cols] - sy)))
    assert err <= 2.0 ** (s - 52)
