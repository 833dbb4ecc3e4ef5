"""The FP64 tree levels of the batched FP32 kernel at d = 17..64 (digit products of 32 x 32 blocks)."""

import numpy as np
import pytest

import oracle
from paper_2108_07126_gb300 import workloads as wl
from tolerances import check, tol32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 17, 150])
@pytest.mark.parametrize("d", [17, 31, 32, 33, 48, 49, 64])
def test_short_leaves_of_one_dimension(d, n):
    """Leaves of one slice: trees of up to eight levels, the top three in FP64."""
    import torch

    from paper_2108_07126_gb300 import binding as b

    probs = [wl.random_problem(d, 2, n, "midpoint", seed=7100 + d + i, g_norm=0.3) for i in range(3)]
    prop = b.Propagator(0)
    try:
        prop.set_option(b.PARAMENT_OPT_BATCH_LEAF_STEPS, 1)
        prop.set_option(b.PARAMENT_OPT_BATCH_ITEMS_PER_SM, 64)
        inst, keep, outs = prop.batch([(p.H0, p.Hk, p.c, p.dt, n) for p in probs], "fp32")
        prop.propagate_batched(inst, "fp32")
        torch.cuda.synchronize()
    finally:
        prop.close()
    for p, U in zip(probs, outs):
        R = oracle.propagate(p.H0.astype(np.complex64).astype(complex), p.Hk.astype(np.complex64).astype(complex),
                             p.c.astype(np.float32).astype(float), p.dt, "midpoint")
        check(np.max(np.abs(U.cpu().numpy() - R)), tol32(d, n))
