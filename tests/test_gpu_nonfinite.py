"""Non-finite control samples: every result that depends on the sample is NaN, and nothing else is."""

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


N, BAD, EVERY = 1203, 619, 7  # BAD: slice of the sample, inside a tile and a leaf for every geometry below


def trajectory_with_nan(prop, d, prec, grid, with_psi, bad=BAD, value=float("nan")):
    """(rounded inputs, dt, psi_0 or None, output) of a run whose slice `bad` has a non-finite sample."""
    import torch

    from paper_2108_07126_gb300 import binding as b

    prob = wl.random_problem(d, 2, N, "midpoint", seed=6000 + d, g_norm=0.3)
    hd, cd = (torch.complex128, torch.float64) if prec == "fp64" else (torch.complex64, torch.float32)
    H0, Hk, c = torch.as_tensor(prob.H0).to(hd), torch.as_tensor(prob.Hk).to(hd), torch.as_tensor(prob.c).to(cd)
    psi = torch.as_tensor(wl.haar_unitary(np.random.default_rng(6001 + d), d)[:, 0].copy()).to(hd) if with_psi else None
    c[1, bad] = value
    prop.set_option(b.PARAMENT_OPT_GRID_BLOCKS, grid)
    prop.set_hamiltonians(H0, Hk, prob.integrator)
    prop.set_controls(c, prob.dt, N)
    out = prop.propagate_trajectory(prec, EVERY, psi).cpu().numpy()
    assert prop.stats()["device_status"] & b.PARAMENT_DEV_NONFINITE_NORM
    wide = [np.asarray(x).astype(np.complex128 if x.dtype.is_complex else np.float64) for x in (H0, Hk, c)]
    return wide, prob.dt, psi, out


@pytest.mark.parametrize("grid", [0, 2])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("d", [2, 8, 12, 16, 24, 40])
@pytest.mark.parametrize("with_psi", [False, True])
def test_trajectory_is_nan_from_the_sample_on(prop, d, prec, grid, with_psi):
    _, _, _, out = trajectory_with_nan(prop, d, prec, grid, with_psi)
    after = out[BAD // EVERY:]  # outputs at slices EVERY (o + 1) > BAD, and the last
    assert np.isnan(after.real).all() and np.isnan(after.imag).all()


@pytest.mark.parametrize("grid", [0, 2])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("d", [8, 12, 16, 24, 40])
@pytest.mark.parametrize("with_psi", [False, True])
def test_trajectory_before_the_sample_is_valid(prop, d, prec, grid, with_psi):
    """The outputs before the sample equal the oracle's of the run that ends there."""
    (H0, Hk, c), dt, psi, out = trajectory_with_nan(prop, d, prec, grid, with_psi)
    n = BAD // EVERY
    R = oracle.trajectory(H0, Hk, c[:, :n * EVERY], dt, "midpoint", EVERY)
    if psi is not None:
        R = R @ psi.numpy().astype(np.complex128)
    err = np.max(np.abs(out[:n].astype(np.complex128) - R))
    assert err <= (TOL64 if prec == "fp64" else tol32(d, n * EVERY))


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("bad", [50, 619, 1000])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_other_leaves_of_the_warp_keep_their_class(prop, d, prec, bad, value):
    """d <= 8: several leaves per warp, whose slices share the degree and the squarings of the highest norm."""
    (H0, Hk, c), dt, _, out = trajectory_with_nan(prop, d, prec, 0, False, bad, value)
    n = bad // EVERY
    R = oracle.trajectory(H0, Hk, c[:, :n * EVERY], dt, "midpoint", EVERY)
    assert np.max(np.abs(out[:n].astype(np.complex128) - R)) <= (TOL64 if prec == "fp64" else tol32(d, n * EVERY))
    assert np.isnan(out[n:].real).all() and np.isnan(out[n:].imag).all()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("d", [8, 16, 24, 40])
def test_gradient_is_nan_everywhere(prop, d, prec):
    """Every component of the gradient depends on U(T), and so on every sample."""
    import torch

    prob = wl.random_problem(d, 2, 400, "midpoint", seed=6100 + d, g_norm=0.3)
    prob.c[0, 133] = np.nan
    hd, cd = (torch.complex128, torch.float64) if prec == "fp64" else (torch.complex64, torch.float32)
    prop.set_hamiltonians(torch.as_tensor(prob.H0).to(hd), torch.as_tensor(prob.Hk).to(hd), prob.integrator)
    prop.set_controls(torch.as_tensor(prob.c).to(cd), prob.dt, prob.n_steps)
    loss, g = prop.propagate_grad(torch.eye(d, dtype=hd), prec)
    assert np.isnan(loss) and torch.isnan(g).all()
