"""FP64 paths on exact digit products (d >= 5) and on unit quaternions (d <= 2) at the sizes where they can go
wrong: partial tiles of 16 slices, empty leaves, matrices that fill or just exceed 8, 16, 32, 48, 64, 128 rows,
squarings, NaN, and targets far from unitary.  Against the FP64 oracle at the FP64 bound of the other tests (1e-11
max-entry, gradients 1e-9 relative)."""

import numpy as np
import pytest

import oracle
from paper_2108_07126_gb300 import workloads as wl
from tolerances import TOL64, check, tol32

pytestmark = pytest.mark.gpu


@pytest.fixture()
def prop():
    import torch

    from paper_2108_07126_gb300.binding import Propagator

    assert torch.cuda.is_available()
    p = Propagator(0)
    yield p
    p.close()


def load(prop, prob, prec="fp64"):
    import torch

    hd = torch.complex128 if prec == "fp64" else torch.complex64
    cd = torch.float64 if prec == "fp64" else torch.float32
    prop.set_hamiltonians(torch.as_tensor(prob.H0).to(hd), torch.as_tensor(prob.Hk).to(hd), prob.integrator)
    prop.set_controls(torch.as_tensor(prob.c).to(cd), prob.dt, prob.n_steps)


def ref(prob):
    return oracle.propagate(prob.H0, prob.Hk, prob.c, prob.dt, prob.integrator)


@pytest.mark.parametrize("d", [5, 8, 9, 16])
@pytest.mark.parametrize("n", [2, 15, 16, 17, 33, 2500])
def test_small_d_slice_tiles(prop, d, n):
    """Tiles of 16 slices: one short of, at and beyond the edge, and leaves without slices."""
    prob = wl.random_problem(d, 3, n, "magnus4_gl2", seed=4000 + d + n, g_norm=0.4)
    load(prop, prob)
    assert np.max(np.abs(prop.propagate("fp64").cpu().numpy() - ref(prob))) <= TOL64


@pytest.mark.parametrize("d,K", [(8, 8), (16, 8), (16, 10)])
def test_small_d_many_basis_matrices(prop, d, K):
    """45 and 66 dense basis matrices: the assembly's GEMM in steps of 32."""
    prob = wl.random_problem(d, K, 40, "magnus4_gl2", seed=4100 + K, g_norm=0.3)
    load(prop, prob)
    assert np.max(np.abs(prop.propagate("fp64").cpu().numpy() - ref(prob))) <= TOL64


@pytest.mark.parametrize("d", [17, 32, 33, 48, 49, 64, 65, 80, 112, 113, 128, 144])
def test_large_d_extents(prop, d):
    """Products restricted to the leading multiple of 16 of the padded frame."""
    prob = wl.random_problem(d, 2, 5, "midpoint", seed=4200 + d, g_norm=1.5)
    load(prop, prob)
    assert np.max(np.abs(prop.propagate("fp64").cpu().numpy() - ref(prob))) <= TOL64


@pytest.mark.parametrize("d", [40, 72])
def test_large_d_trajectory_extents(prop, d):
    for prec in ("fp64", "fp32"):
        prob = wl.random_problem(d, 2, 7, "magnus4_simpson", seed=4300 + d, g_norm=0.4)
        load(prop, prob, prec)
        T = prop.propagate_trajectory(prec, 2).cpu().numpy().astype(np.complex128)
        R = oracle.trajectory(prob.H0, prob.Hk, prob.c, prob.dt, prob.integrator, 2)
        # FP32: the inputs are rounded too (2^-24 of exponents below one per slice)
        assert np.max(np.abs(T - R)) <= (TOL64 if prec == "fp64" else 2 * tol32(d, 7) + 7 * 2.0 ** -23)


@pytest.mark.parametrize("integrator", ["midpoint", "magnus4_gl2", "magnus4_simpson"])
@pytest.mark.parametrize("d,n", [(5, 1), (8, 16), (8, 500), (11, 17), (16, 40)])
def test_adjoint_tiles(prop, integrator, d, n):
    prob = wl.random_problem(d, 3, n, integrator, seed=4400 + d + n, g_norm=0.5)
    V = wl.haar_unitary(np.random.default_rng(d + n), d)
    load(prop, prob)
    loss, g = prop.propagate_grad(V, "fp64")
    l_ref, g_ref, _ = oracle.loss_and_gradient(prob.H0, prob.Hk, prob.c, prob.dt, V, integrator)
    assert abs(loss - l_ref) <= 1e-11
    assert np.max(np.abs(g.cpu().numpy() - g_ref)) <= 1e-9 * np.max(np.abs(g_ref))


@pytest.mark.parametrize("scale", [1e-3, 1.0, 40.0])
@pytest.mark.parametrize("d", [8, 12, 24])
def test_adjoint_with_a_target_that_is_not_unitary(prop, d, scale):
    """V enters scaled to the range of the fixed-point numbers and the gradient is scaled back."""
    prob = wl.random_problem(d, 2, 30, "midpoint", seed=4500 + d, g_norm=2.5)
    V = scale * np.random.default_rng(d).standard_normal((d, d)).astype(np.complex128)
    load(prop, prob)
    loss, g = prop.propagate_grad(V, "fp64")
    l_ref, g_ref, _ = oracle.loss_and_gradient(prob.H0, prob.Hk, prob.c, prob.dt, V)
    assert abs(loss - l_ref) <= 1e-11 * max(1.0, abs(l_ref))
    assert np.max(np.abs(g.cpu().numpy() - g_ref)) <= 1e-9 * np.max(np.abs(g_ref))


@pytest.mark.parametrize("d", [2, 8, 16, 40])
def test_nan_control_gives_nan(prop, d):
    import torch

    prob = wl.random_problem(d, 2, 100, "midpoint", seed=4600 + d, g_norm=0.3)
    prob.c[1, 50] = np.nan
    load(prop, prob)
    U = prop.propagate("fp64")
    assert torch.isnan(torch.view_as_real(U)).all()
    assert prop.stats()["device_status"] & 1


@pytest.mark.parametrize("integrator", ["midpoint", "magnus4_gl2", "magnus4_simpson"])
@pytest.mark.parametrize("n,g_norm", [(1, 0.3), (31, 0.3), (256, 0.3), (257, 0.3), (19457, 0.05), (60, 9.0), (60, 40.0)])
@pytest.mark.parametrize("d", [1, 2])
def test_two_level_systems(prop, integrator, d, n, g_norm):
    """One and several blocks, more threads than slices, halvings of the exponent; FP64 and FP32."""
    prob = wl.random_problem(d, 2, n, integrator, seed=4700 + n, g_norm=g_norm)
    load(prop, prob)
    assert np.max(np.abs(prop.propagate("fp64").cpu().numpy() - ref(prob))) <= TOL64 * max(1.0, g_norm)
    load(prop, prob, "fp32")
    r32 = oracle.propagate(prob.H0.astype(np.complex64).astype(complex), prob.Hk.astype(np.complex64).astype(complex),
                           prob.c.astype(np.float32).astype(float), prob.dt, integrator)
    U = prop.propagate("fp32").cpu().numpy().astype(np.complex128)
    check(np.max(np.abs(U - r32)), tol32(d, n) * max(1.0, g_norm))


@pytest.mark.parametrize("grid,warps", [(1, 1), (3, 2), (7, 8), (304, 3)])
def test_two_level_geometry(prop, grid, warps):
    from paper_2108_07126_gb300 import binding as b

    prob = wl.random_problem(2, 2, 3001, "magnus4_gl2", seed=4800, g_norm=0.3)
    prop.set_option(b.PARAMENT_OPT_GRID_BLOCKS, grid)
    prop.set_option(b.PARAMENT_OPT_BLOCK_WARPS, warps)
    load(prop, prob)
    for _ in range(2):  # the arrival counter is ready for the next call
        assert np.max(np.abs(prop.propagate("fp64").cpu().numpy() - ref(prob))) <= TOL64
    st = prop.stats()
    assert st["grid_blocks"] == grid and st["tree_products"] == 3001
