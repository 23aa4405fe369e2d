"""The FP64 tile kernel against the naive kernel and the assembled matrix.

R and J of the tile kernel are the naive kernel's bits on every tile shape
(one row or column of cells, partial tiles, several runs of planes), with
level layers (its links without gravity terms), tilted ones (every link with
them) and a mix of both in one warp, and with exact ties on the vertical and
in-plane links.  J w and J^T v come from the same links summed in another
order, so they agree with the products of the assembled matrix to the
rounding of such sums: at most 30 operations per row, each within 2^-53 of
sum |J| |w|; 64 of those are allowed.
"""
import numpy as np
import pytest

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 300, 3), (300, 1, 2), (129, 7, 5), (33, 9, 40), (9, 28, 70), (2, 2, 130)]


def _problem(shape, conn, c_r, depth):
    prob = synth.make_problem(*shape, seed=sum(shape), connectivity=conn, c_r=c_r)
    rng = np.random.default_rng(3)
    nx, ny, nz = shape
    if depth == "tilted":
        prob.depth = prob.depth + 0.03 * np.tile(np.arange(nx), ny * nz)
    elif depth == "mixed":  # half of the rows level, steps in the others
        prob.depth = prob.depth + np.where(rng.random(prob.n) < 0.02, 0.5, 0.0)
    elif depth == "ties":  # equal pressures in level layers; equal potentials need g = 0
        prob.phys["g"] = 0.0
        p = prob.p.reshape(nz, ny, nx)
        p[:, :, : (nx + 1) // 2] = 1.0e7
        prob.p = p.reshape(-1)
    return prob


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("conn", [6, 10])
@pytest.mark.parametrize("c_r", [0.0, 1e-9])
@pytest.mark.parametrize("depth", ["level", "tilted", "mixed", "ties"])
def test_fp64_tile_kernel_matches_naive_and_matrix(shape, conn, c_r, depth):
    from scipy.sparse import csr_matrix

    from paper_2304_11274_gb300.api import Grid
    prob = _problem(shape, conn, c_r, depth)
    w = np.random.default_rng(5).standard_normal(prob.n)
    with Grid(*shape, prob.phys, "fp64", prob.perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        a = [x.cpu().numpy() for x in g.assemble_jacobian(kernel="auto")[:2]]
        b = [x.cpu().numpy() for x in g.assemble_jacobian(kernel="naive")[:2]]
        R = g.assemble_residual().cpu().numpy()
        Jw, R2 = (x.cpu().numpy() for x in g.jvp(w, want_residual=True))
        g_p, g_lnk = (x.cpu().numpy() for x in g.vjp(w))
        rp, ci = (x.cpu().numpy() for x in g.pattern())
        g.sync_status()
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert np.array_equal(R, a[0]) and np.array_equal(R2, a[0])
    J = csr_matrix((a[1], ci, rp), shape=(prob.n, prob.n))
    assert (np.abs(Jw - J @ w) <= 64 * 2.0 ** -53 * (abs(J) @ np.abs(w))).all()
    assert (np.abs(g_p - J.T @ w) <= 64 * 2.0 ** -53 * (abs(J).T @ np.abs(w))).all()
    assert np.isfinite(g_lnk).all()
