"""The workspace cap of the gradient."""

import numpy as np
import pytest

from paper_2108_07126_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("integrator", ["midpoint", "magnus4_simpson"])
@pytest.mark.parametrize("d,n,prec", [(8, 3001, "fp64"), (16, 2500, "fp64"), (8, 1000, "fp32")])
def test_few_workspace_slots_give_the_same_gradient(d, n, prec, integrator):
    """1 MiB holds 42 leaves (d = 8) or 8 (d = 16): each warp sweeps many leaves in turn.  Every leaf's arithmetic is the same;
    Simpson end points are sums of two slices in either order."""
    import torch

    from paper_2108_07126_gb300 import binding as b

    hd, cd = (torch.complex128, torch.float64) if prec == "fp64" else (torch.complex64, torch.float32)
    prob = wl.random_problem(d, 2, n, integrator, seed=6600 + d, g_norm=0.3)
    V = wl.haar_unitary(np.random.default_rng(6601), d)
    out, used = [], []
    for mb in (4096, 1):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        prop = b.Propagator(0)
        try:
            prop.set_option(b.PARAMENT_OPT_WORKSPACE_MB, mb)
            prop.set_hamiltonians(torch.as_tensor(prob.H0).to(hd), torch.as_tensor(prob.Hk).to(hd), integrator)
            prop.set_controls(torch.as_tensor(prob.c).to(cd), prob.dt, n)
            out.append(prop.propagate_grad(V, prec)[1].cpu())
            used.append(free - torch.cuda.mem_get_info()[0])
        finally:
            prop.close()
    assert torch.equal(out[0], out[1])
    leaves = 600  # at least, in one wave of blocks of eight or sixteen warps
    if prec == "fp64":
        assert used[0] - used[1] > (leaves - 42) * (120 if d == 16 else 24) * 1024 // 2
