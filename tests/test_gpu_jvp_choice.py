"""The library's choice of J w march: not slower than the one-cell march on small
grids, and, from the sizes on where the two-cell march runs, the naive kernel's
values at the edges of its shapes (one row, one plane, a ragged last segment, one
of a single cell pair) with exact ties, impermeable cells and a direction with
zeros, FP32 subnormals and entries below them.

Times are the best of ten of 20 calls in a row; 1.15 times the one-cell march's is
allowed (the two-cell march took up to 2.6 times as long).
"""
import numpy as np
import pytest
import torch

import _compare as C
from paper_2304_11274_gb300 import synth
from test_gpu_autotune_choice import _best_us

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(512, 2, 128), (128, 8, 128), (192, 16, 64), (300, 4, 300), (100000, 1, 1)])
@pytest.mark.parametrize("conn", [6, 10])
def test_small_grids_take_the_faster_march(shape, conn):
    from paper_2304_11274_gb300.api import Grid
    prob = synth.round_to_f32(synth.make_problem(*shape, seed=1, connectivity=conn))
    w = torch.as_tensor(np.random.default_rng(1).standard_normal(prob.n), device="cuda")
    with Grid(*shape, prob.phys, "mixed", prob.perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        Jw = torch.empty_like(w)
        one, auto = _best_us(lambda: g.jvp(w, out=Jw, kernel="tiled")), _best_us(lambda: g.jvp(w, out=Jw))
    assert auto <= 1.15 * one, (one, auto)


@pytest.mark.parametrize("shape", [(128, 1, 16400), (256, 8200, 1), (258, 70, 120), (190, 111, 101), (2048, 32, 33)])
@pytest.mark.parametrize("conn", [6, 10])
@pytest.mark.parametrize("c_r", [0.0, 1e-9])
def test_values_where_the_two_cell_march_runs(shape, conn, c_r):
    from paper_2304_11274_gb300.api import Grid
    prob = C.tie_pairs_problem("mixed", conn, shape=shape, frac=0.01)
    prob.phys["c_r"] = c_r
    rng = np.random.default_rng(2)
    perm = np.where(rng.random(prob.n) < 0.02, 0.0, prob.perm)
    w = rng.standard_normal(prob.n)
    odd = rng.random(prob.n) < 0.001
    w = np.where(odd, w * 10.0 ** rng.uniform(-330.0, -30.0, prob.n), np.where(rng.random(prob.n) < 0.1, 0.0, w))
    w = torch.as_tensor(w, device="cuda")
    with Grid(*shape, prob.phys, "mixed", perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        Jn, Rn = g.jvp(w, want_residual=True, kernel="naive")
        Jt, Rt = g.jvp(w, want_residual=True)
        assert torch.equal(Jt, Jn) and torch.equal(Rt, Rn) and torch.equal(g.jvp(w)[0], Jn)
        g.sync_status()
