"""The Krylov kernels at the edges of their shapes.

Columns are solved from both ends (nz = 1: the middle row alone; 2, 3: one
half empty or both of one row; lengths around the chunks of four steps), 32
columns per block, the product's runs of planes and 256-column tiles.  The
solution is checked against the assembled matrix the solver uses: the
recursively updated residual is below rtol ||b||, and the true one differs
from it by the rounding of the iterations, 1e-12 of |J| |x| allowed.
"""
import numpy as np
import pytest

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 2, 1), (5, 7, 2), (40, 3, 3), (31, 1, 4), (8, 8, 9), (17, 16, 37),
                                   (3, 2, 131)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("conn", [6, 10])
@pytest.mark.parametrize("precond", ["zline", "jacobi"])
def test_linear_solve_on_edge_shapes(shape, precision, conn, precond):
    from scipy.sparse import csr_matrix

    from paper_2304_11274_gb300.api import Grid
    prob = synth.make_problem(*shape, seed=sum(shape), connectivity=conn, c_r=1e-8, dt=3600.0)
    b = np.random.default_rng(2).standard_normal(prob.n)
    rtol = 1e-10
    with Grid(*shape, prob.phys, precision, prob.perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        x, st = g.linear_solve(b, rtol=rtol, max_iters=3000, precond=precond)
        _, vals, diag = g.assemble_jacobian()
        rp, ci = (t.cpu().numpy() for t in g.pattern())
        x, vals = x.cpu().numpy(), vals.double().cpu().numpy()
        if diag is not None:
            vals[ci == np.repeat(np.arange(prob.n), np.diff(rp))] = diag.cpu().numpy()
    assert st["converged"] == 1 and st["rel_residual"] <= rtol
    J = csr_matrix((vals, ci, rp), shape=(prob.n, prob.n))
    bound = 2 * rtol * np.linalg.norm(b) + 1e-12 * np.linalg.norm(abs(J) @ np.abs(x))
    assert np.linalg.norm(J @ x - b) <= bound
    if shape == (1, 1, 1) or (precond == "zline" and shape[0] * shape[1] == 1):
        assert st["iterations"] <= 2  # the preconditioner is the inverse
