"""The linear solve is indifferent to the scale of b and J.

On the mixed path the products take the vector as FP32 pairs.  A trailing half
that is lost (small right-hand sides, large matrix entries) leaves single
precision products, with which BiCGStab stalls at a relative residual of about
1e-7.  The iterations of one system scatter by about a fifth from scale to
scale; twice the unscaled number is allowed.
"""
import numpy as np
import pytest

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("matrix, rhs", [(1.0, 1e-27), (1.0, 1e-29), (1.0, 1e-31), (1.0, 1e-33), (1e6, 1e-28),
                                         (1e12, 1e-22), (1e12, 1e-24), (1e12, 1e-26)])
@pytest.mark.parametrize("precond", ["zline", "jacobi"])
def test_scaled_systems_converge_alike(matrix, rhs, precond):
    from paper_2304_11274_gb300.api import Grid
    shape = (40, 30, 20)
    iterations = []
    for m, r in ((1.0, 1.0), (matrix, rhs)):
        prob = synth.make_problem(*shape, seed=5, connectivity=10, c_r=1e-8, dt=3600.0 / m)
        b = np.random.default_rng(2).standard_normal(prob.n) * r
        with Grid(*shape, prob.phys, "mixed", prob.perm * m, prob.poro, prob.depth) as g:
            g.set_state(prob.p, prob.pn)
            _, st = g.linear_solve(b, rtol=1e-10, max_iters=2000, precond=precond)
            iterations.append(st["iterations"])
    assert iterations[1] <= 2 * iterations[0], iterations
