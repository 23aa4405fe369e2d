"""Cells of permeability zero on a wide grid: the two-cell march's links of
such cells have T = 0, no flux and no derivative, from either end.

The outputs are the naive kernel's values (a zero derivative may carry either
sign, so values are compared), and the calls cost what they cost without such
cells: a twentieth of the cells leaves hardly a 64-cell row without one, and a
march that computed those rows again one thread per cell took four to eight
times as long.  1.5 times is allowed.
"""
import numpy as np
import pytest
import torch

import _compare as C
from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


def median_us(call, reps=15):
    times = []
    for _ in range(3):
        call()
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 1e3)
    return sorted(times)[reps // 2]


@pytest.mark.parametrize("shape", [(128, 9, 4), (182, 37, 5), (256, 6, 3)])
@pytest.mark.parametrize("conn", [6, 10])
def test_values_with_impermeable_cells_and_ties(shape, conn):
    from paper_2304_11274_gb300.api import Grid
    prob = C.tie_pairs_problem("mixed", conn, shape=shape)  # exact ties beside them: those rows are recomputed
    perm = np.where(np.random.default_rng(4).random(prob.n) < 0.2, 0.0, prob.perm)
    w = torch.as_tensor(np.random.default_rng(1).standard_normal(prob.n), device="cuda")
    with Grid(*shape, prob.phys, "mixed", perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        ref = [t.clone() for t in g.assemble_jacobian(kernel="naive")]
        assert all(torch.equal(a, b) for a, b in zip(g.assemble_jacobian(kernel="tiled2"), ref))
        assert torch.equal(g.assemble_residual(), ref[0])
        for a, b in zip(g.jvp(w, want_residual=True), g.jvp(w, want_residual=True, kernel="naive")):
            assert torch.equal(a, b)
        g.sync_status()


@pytest.mark.parametrize("conn", [6, 10])
def test_time_with_impermeable_cells(conn):
    from paper_2304_11274_gb300.api import Grid
    shape = (512, 512, 32)
    prob = synth.round_to_f32(synth.make_problem(*shape, seed=3, connectivity=conn))
    off = np.random.default_rng(4).random(prob.n) < 0.05
    w = torch.as_tensor(np.random.default_rng(1).standard_normal(prob.n), device="cuda")
    times = []
    for perm in (prob.perm, np.where(off, 0.0, prob.perm)):
        with Grid(*shape, prob.phys, "mixed", perm, prob.poro, prob.depth) as g:
            g.set_state(prob.p, prob.pn)
            outs, Jw = g.empty_outputs(), torch.empty_like(w)
            times.append([median_us(lambda: g.jvp(w, out=Jw)), median_us(lambda: g.assemble_jacobian(*outs))])
            g.sync_status()
    assert all(b <= 1.5 * a for a, b in zip(*times)), times
