"""Backward passes on a grid whose permeability was replaced after their
forward pass: the gradients are those of the forward's own log-permeability."""
import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_backward_after_another_forward(precision):
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
        R1 = residual(g, p, k1)
        residual(g, p, k2)
        got = torch.autograd.grad(R1, (p, k1), v, retain_graph=True)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        g.set_permeability(prob.perm * 3.0)
        got = torch.autograd.grad(R1, (p, k1), v)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
