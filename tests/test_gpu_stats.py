"""Statistics of a call whose path does not follow every option."""

import numpy as np
import pytest

from paper_2108_07126_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [40, 100])
def test_gradient_threads_with_the_chebyshev_option(d):
    """The gradient always takes the Taylor exponential: the same geometry with either setting of the option."""
    import torch

    from paper_2108_07126_gb300 import binding as b

    prob = wl.random_problem(d, 1, 6, "midpoint", seed=6700 + d, g_norm=0.3)
    prop = b.Propagator(0)
    try:
        prop.set_hamiltonians(torch.as_tensor(prob.H0), torch.as_tensor(prob.Hk), "midpoint")
        prop.set_controls(torch.as_tensor(prob.c), prob.dt, prob.n_steps)
        threads, grads = [], []
        for method in (0, 1):
            prop.set_option(b.PARAMENT_OPT_EXP_METHOD, method)
            grads.append(prop.propagate_grad(np.eye(d), "fp64")[1].cpu())
            threads.append(prop.stats()["block_threads"])
        assert threads[0] == threads[1] and torch.equal(grads[0], grads[1])
    finally:
        prop.close()


@pytest.mark.parametrize("d", [3, 4])
@pytest.mark.parametrize("n", [1, 511, 513, 12800, 12801, 51201, 102400, 330000])
def test_fp32_leaves_of_small_systems(d, n):
    """d = 3, 4, FP32: two slices a leaf up to a sixth of the SMs, then up to eight, then more blocks; U(T) against FP64."""
    import torch

    from paper_2108_07126_gb300 import binding as b
    from tolerances import tol32

    prob = wl.random_problem(d, 2, n, "midpoint", seed=7000 + d, g_norm=0.3)
    H0, Hk, c = prob.H0.astype(np.complex64), prob.Hk.astype(np.complex64), prob.c.astype(np.float32)
    prop = b.Propagator(0)
    try:
        U = {}
        for prec, hd, cd in (("fp32", torch.complex64, torch.float32), ("fp64", torch.complex128, torch.float64)):
            prop.set_hamiltonians(torch.as_tensor(H0).to(hd), torch.as_tensor(Hk).to(hd), "midpoint")
            prop.set_controls(torch.as_tensor(c).to(cd), prob.dt, n)
            U[prec] = prop.propagate(prec).cpu().numpy()
            if prec == "fp32":
                st = prop.stats()
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        leaf = n / st["leaves"]
        assert st["grid_blocks"] <= max(sms // 6, -(-n // (8 * 256))) and (leaf <= 8 or st["grid_blocks"] >= sms)
        assert np.max(np.abs(U["fp32"] - U["fp64"])) <= tol32(d, n)
    finally:
        prop.close()
