"""Backward passes on a grid whose permeability was replaced after their forward
pass by something else than this module's calls: the C interface, or a CUDA
graph of another forward pass that is replayed.  The gradients are those of the
forward's own log-permeability, bit for bit."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("by", ["c call", "graph", "graph of both passes", "nothing"])
def test_backward_after_a_replacement(precision, by):
    from paper_2304_11274_gb300 import _capi
    from paper_2304_11274_gb300.api import Grid, residual
    prob = synth.round_to_f32(synth.make_problem(12, 9, 5, seed=3, connectivity=10))
    dt = torch.float64 if precision == "fp64" else torch.float32
    v = torch.as_tensor(np.random.default_rng(1).standard_normal(prob.n), device="cuda")
    with Grid(prob.nx, prob.ny, prob.nz, prob.phys, precision, prob.perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        p = torch.as_tensor(prob.p, device="cuda", dtype=dt).requires_grad_(True)
        k1 = torch.log(torch.as_tensor(prob.perm, device="cuda")).requires_grad_(True)
        k2 = (k1.detach() + 0.7).requires_grad_(True)
        want = torch.autograd.grad(residual(g, p, k1), (p, k1), v)
        want2 = torch.autograd.grad(residual(g, p, k2), (p, k2), v)
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        if by == "graph":
            with torch.no_grad(), torch.cuda.graph(graph):
                residual(g, p, k2)
        elif by == "graph of both passes":
            with torch.cuda.graph(graph):
                got2 = torch.autograd.grad(residual(g, p, k2), (p, k2), v)
        R1 = residual(g, p, k1)
        if by == "c call":
            _capi.check(g.lib.tpfa_set_log_permeability(g.handle, ctypes.c_void_p(k2.data_ptr()),
                                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
        elif by != "nothing":
            graph.replay()
        for _ in range(2):
            got = torch.autograd.grad(R1, (p, k1), v, retain_graph=True)
            assert all(torch.equal(a, b) for a, b in zip(got, want))
        if by == "graph of both passes":
            graph.replay()
            assert all(torch.equal(a, b) for a, b in zip(got2, want2))
        g.sync_status()
