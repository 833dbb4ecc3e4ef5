"""Gradient routes on both sides of their limits: FP32 at d = 5..8 (up to 2048 slices through FP64, then the float sweeps), and the
checkpointed block-level sweeps, which FP32 takes at d >= 17."""

import numpy as np
import pytest

import oracle
from paper_2108_07126_gb300 import workloads as wl
from test_gpu_grad import GRAD32_REL, gpu_grad, prop  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("integrator", ["midpoint", "magnus4_gl2", "magnus4_simpson"])
@pytest.mark.parametrize("n", [2047, 2048, 2049, 3000])
@pytest.mark.parametrize("d", [5, 8])
@pytest.mark.parametrize("host", [False, True])
def test_fp32_gradient_around_the_fp64_route(prop, d, n, integrator, host):  # noqa: F811
    """Device and host gradients in float against the oracle; the loss and U(T) too."""
    from paper_2108_07126_gb300 import binding as b

    prob = wl.random_problem(d, 2, n, integrator, seed=6800 + d, g_norm=0.3)
    V = wl.haar_unitary(np.random.default_rng(6801 + d), d)
    l_ref, g_ref, _ = oracle.loss_and_gradient(prob.H0, prob.Hk, prob.c, prob.dt, V, integrator)
    if host:
        c, g, V32 = prob.c.astype(np.float32), np.full(prob.c.shape, np.nan, np.float32), V.astype(np.complex64)
        H0, Hk = prob.H0.astype(np.complex64), prob.Hk.astype(np.complex64)
        kind = {"midpoint": b.PARAMENT_MIDPOINT, "magnus4_gl2": b.PARAMENT_MAGNUS4_GL2,
                "magnus4_simpson": b.PARAMENT_MAGNUS4_SIMPSON}[integrator]
        b.parament_set_hamiltonians(prop.ctx, d, 2, H0.ctypes.data, Hk.ctypes.data, b.PARAMENT_C64, kind)
        b.parament_set_controls(prop.ctx, c.ctypes.data, b.PARAMENT_F32, n, prob.dt)
        loss = b.parament_propagate_grad(prop.ctx, V32.ctypes.data, g.ctypes.data, None, b.PARAMENT_PREC_FP32)
    else:
        loss, g, _ = gpu_grad(prop, prob, V, "fp32", integrator=integrator)
    assert np.max(np.abs(g - g_ref)) <= GRAD32_REL * np.max(np.abs(g_ref))
    assert abs(loss - l_ref) <= 2e-4


@pytest.mark.parametrize("d,n", [(20, 400), (40, 700), (70, 320)])
def test_fp32_block_level_checkpoints_agree(prop, d, n):  # noqa: F811
    """Leaves longer than the sub-chunk buffer re-compute their prefixes: the same operations, the same float results (1e-6)."""
    prob = wl.random_problem(d, 2, n, "magnus4_gl2", seed=6900 + d, g_norm=0.3)
    V = wl.haar_unitary(np.random.default_rng(6901), d)
    _, g_full, _ = gpu_grad(prop, prob, V, "fp32", integrator="magnus4_gl2")
    leaf = -(-n // prop.stats()["leaves"])
    assert leaf > 1
    _, g_ck, _ = gpu_grad(prop, prob, V, "fp32", subchunk=1, integrator="magnus4_gl2")
    assert prop.stats()["grad_subchunk"] == 1
    assert np.max(np.abs(g_full - g_ck)) <= 1e-6 * np.max(np.abs(g_full))
    _, g_ref, _ = gpu_grad(prop, prob, V, integrator="magnus4_gl2")  # FP64, one sweep
    assert np.max(np.abs(g_ck - g_ref)) <= GRAD32_REL * np.max(np.abs(g_ref))
