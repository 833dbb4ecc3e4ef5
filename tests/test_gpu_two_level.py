"""Two-level systems (d <= 2) on unit quaternions: the FP32 norm correction, and the options of the matrix scheme."""

import numpy as np
import pytest

import oracle
from paper_2108_07126_gb300 import workloads as wl
from tolerances import TOL64, tol32

pytestmark = pytest.mark.gpu


@pytest.fixture()
def prop():
    import torch

    from paper_2108_07126_gb300.binding import Propagator

    assert torch.cuda.is_available()
    p = Propagator(0)
    yield p
    p.close()


@pytest.mark.parametrize("n,grid,warps", [(2048, 0, 0), (16384, 0, 0), (16384, 1, 1), (3001, 3, 2), (100, 0, 0)])
def test_fp32_norm_does_not_drift(prop, n, grid, warps):
    """The Rabi qubit in leaves of one slice and of many.  Unitarity: a product of 128 slices has a norm off by at most
    128 x 2^-22, which the step squares away; what is left is the rounding of U to complex64 (2^-24 an entry, 2^-22 with
    room).  Error: below the 1.2e-5 of the 2 x 2 matrix products with a step on every leaf, measured at N = 2^14 (N = 100:
    exponents of 31 radians, whose own rounding is larger)."""
    import torch

    from paper_2108_07126_gb300 import binding as b

    prob = wl.rabi_qubit(n)
    H0, Hk, c = prob.H0.astype(np.complex64), prob.Hk.astype(np.complex64), prob.c.astype(np.float32)
    prop.set_option(b.PARAMENT_OPT_GRID_BLOCKS, grid)
    prop.set_option(b.PARAMENT_OPT_BLOCK_WARPS, warps)
    prop.set_hamiltonians(torch.as_tensor(H0), torch.as_tensor(Hk), prob.integrator)
    prop.set_controls(torch.as_tensor(c), prob.dt, n)
    U = prop.propagate("fp32").cpu().numpy().astype(np.complex128)
    assert np.max(np.abs(U.conj().T @ U - np.eye(2))) <= 2.0 ** -22
    if n < 2048:
        return
    R = oracle.propagate(H0.astype(np.complex128), Hk.astype(np.complex128), c.astype(np.float64), prob.dt, prob.integrator)
    assert np.max(np.abs(U - R)) <= 1.2e-5


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("degree,extra", [(0, 0), (4, 0), (12, 0), (0, 3), (9, 2)])
def test_forced_degree_and_extra_squarings(prop, d, prec, degree, extra):
    """Forced degrees and extra squarings run (the matrix scheme has them), and the statistics name what ran."""
    import torch

    from paper_2108_07126_gb300 import binding as b

    n = 300
    prob = wl.random_problem(d, 2, n, "magnus4_gl2", seed=6200 + d, g_norm=0.3)
    hd, cd = (torch.complex128, torch.float64) if prec == "fp64" else (torch.complex64, torch.float32)
    H0, Hk, c = torch.as_tensor(prob.H0).to(hd), torch.as_tensor(prob.Hk).to(hd), torch.as_tensor(prob.c).to(cd)
    R = oracle.propagate(H0.numpy().astype(complex), Hk.numpy().astype(complex), c.numpy().astype(float), prob.dt,
                         prob.integrator)
    prop.set_option(b.PARAMENT_OPT_TAYLOR_DEGREE, degree)
    prop.set_option(b.PARAMENT_OPT_EXTRA_SQUARINGS, extra)
    prop.set_hamiltonians(H0, Hk, prob.integrator)
    prop.set_controls(c, prob.dt, n)
    U = prop.propagate(prec).cpu().numpy()
    # every squaring doubles the rounding of the polynomial (a few 2^-53 a slice), and a low degree needs many
    squarings = prop.stats()["max_squarings"]
    tol = max(TOL64, 4 * n * 2.0 ** (squarings - 53)) if prec == "fp64" else tol32(d, n) * 2.0 ** squarings
    assert np.max(np.abs(U - R)) <= tol
    st = prop.stats()
    assert st["tree_products"] == n and st["device_status"] == 0
    if degree or extra:
        assert st["max_degree"] == degree or degree == 0
        assert squarings >= extra and st["exp_products"] >= n * extra
    else:
        assert st["exp_products"] == 0 and st["max_degree"] == (15 if prec == "fp64" else 11)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("w", [0.6875, -3.0, 77.0])
@pytest.mark.parametrize("n,grid,warps", [(100, 0, 0), (16384, 0, 0), (16384, 1, 1), (300001, 0, 0)])
def test_phases_add_up_exactly(prop, n, grid, warps, w, prec):
    """H = (w + c_j) I with exponents that are exact in the precision, but not their sums: U = e^{-i sum} I.  The phases are summed
    as integers, so what is left is the reduction of a slice's phase above 4 rad (2^-60 a slice), the angle's (2^-52) and the
    cosine's and sine's rounding, and with complex64 that of U."""
    from fractions import Fraction

    import torch

    from paper_2108_07126_gb300 import binding as b

    bits = 46 if prec == "fp64" else 8  # c: multiples of 2^-bits up to 1 / 4
    k = np.random.default_rng(n).integers(-(1 << (bits - 2)), (1 << (bits - 2)) + 1, (1, n))
    hd, cd = (torch.complex128, torch.float64) if prec == "fp64" else (torch.complex64, torch.float32)
    prop.set_option(b.PARAMENT_OPT_GRID_BLOCKS, grid)
    prop.set_option(b.PARAMENT_OPT_BLOCK_WARPS, warps)
    prop.set_hamiltonians(torch.eye(2, dtype=hd) * w, torch.eye(2, dtype=hd)[None], "midpoint")
    prop.set_controls(torch.as_tensor(k * 2.0 ** -bits).to(cd), 0.25, n)
    U = prop.propagate(prec).cpu().numpy()
    phi = (n * Fraction(w) + Fraction(int(k.sum()), 1 << bits)) / 4
    two_pi = 2 * Fraction("3.14159265358979323846264338327950288419716939937510")
    phi = float(phi - round(phi / two_pi) * two_pi)
    tol = n * 2.0 ** -60 + 2.0 ** -50 + (0 if prec == "fp64" else 2.0 ** -23)
    assert np.max(np.abs(U - np.exp(-1j * phi) * np.eye(2))) <= tol
