"""R alone and J w on the two-cell marches: the naive kernels' bits.

Widths of one and several 64-cell segments, a ragged last one, one row, one
plane; marches of every length class; exact ties on in-plane links; J w with
and without R, and with a direction whose storage is not 16-byte aligned
(the one-cell march then runs).
"""
import numpy as np
import pytest
import torch

import _compare as C
from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


def _bits(t):
    return t.view(torch.int64)


@pytest.mark.parametrize("shape", [(64, 5, 3), (66, 9, 5), (128, 66, 9), (230, 41, 11), (256, 1, 6), (258, 7, 1)])
@pytest.mark.parametrize("conn", [6, 10])
@pytest.mark.parametrize("c_r", [0.0, 1e-9])
@pytest.mark.parametrize("ties", [False, True])
def test_residual_and_jvp_bits(shape, conn, c_r, ties):
    from paper_2304_11274_gb300.api import Grid
    if ties:
        prob = C.tie_pairs_problem("mixed", conn, shape=shape)
        prob.phys["c_r"] = c_r
    else:
        prob = synth.round_to_f32(synth.make_problem(*shape, seed=7, connectivity=conn, c_r=c_r))
    w = torch.as_tensor(np.random.default_rng(1).standard_normal(prob.n + 1), device="cuda")
    with Grid(*shape, prob.phys, "mixed", prob.perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        R = _bits(g.assemble_jacobian(kernel="naive")[0])
        for tiling in (None, (1, 4), (7, 8), (64, 4)):
            if tiling:
                g.set_tiling(*tiling)
            got = _bits(g.assemble_residual())
            # a tie's zero flux may carry either sign: zeros compare by value
            assert torch.equal(got, R) or bool(((got == R) | ((got << 1 == 0) & (R << 1 == 0))).all()), tiling
            for d in (w[:-1], w[1:]):
                Jn, Rn = g.jvp(d, want_residual=True, kernel="naive")
                Jt, Rt = g.jvp(d, want_residual=True)
                assert torch.equal(_bits(Jt), _bits(Jn)) and torch.equal(_bits(Rt), _bits(Rn)), tiling
                assert torch.equal(_bits(g.jvp(d)[0]), _bits(Jn)), tiling
        g.sync_status()
