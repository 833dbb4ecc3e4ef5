"""Gradients in captured CUDA graphs: a context whose buffers are in place, new Hamiltonians, and calls outside the graph."""

import numpy as np
import pytest

import oracle
from paper_2108_07126_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["eager first", "replay after new Hamiltonians"])
@pytest.mark.parametrize("d", [4, 8, 12, 24])
def test_captured_gradient_and_new_hamiltonians(d, order):
    import torch

    from paper_2108_07126_gb300 import binding as b

    n = 60
    old, new = (wl.random_problem(d, 2, n, "midpoint", seed=s + d, g_norm=0.4) for s in (6300, 6400))
    V = wl.haar_unitary(np.random.default_rng(6500 + d), d)
    ref = {p.H0.tobytes(): oracle.loss_and_gradient(p.H0, p.Hk, old.c, p.dt, V)[1] for p in (old, new)}
    prop = b.Propagator(0)
    try:
        c, Vd = torch.as_tensor(old.c).cuda(), torch.as_tensor(V).cuda()
        out = torch.zeros(2, n, dtype=torch.float64, device="cuda")

        def load(p):
            prop.set_hamiltonians(torch.as_tensor(p.H0), torch.as_tensor(p.Hk), "midpoint")
            prop.set_controls(c, p.dt, n)

        def gradient():
            b.parament_propagate_grad(prop.ctx, Vd.data_ptr(), out.data_ptr(), None, b.PARAMENT_PREC_FP64, want_loss=False)

        def close(p):
            torch.cuda.synchronize()
            g = ref[p.H0.tobytes()]
            assert np.max(np.abs(out.cpu().numpy() - g)) <= 1e-9 * np.max(np.abs(g))

        stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.stream(stream):
            load(old)
            prop._sync_stream()
            gradient()  # every buffer is in place
            close(old)
            if order == "eager first":
                load(new)
                prop._sync_stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            prop._sync_stream()
            gradient()
        with torch.cuda.stream(stream):
            if order == "eager first":  # a call outside the graph, which has not run yet
                gradient()
            else:  # the graph reads the context's basis, which is another one now
                load(new)
                graph.replay()
            close(new)
    finally:
        prop.close()
