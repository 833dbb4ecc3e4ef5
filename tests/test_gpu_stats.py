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
