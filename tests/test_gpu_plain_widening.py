"""Rows whose FP32 sums or FP64 results lie outside the marches' cheap widening.

Permeabilities scaled so far down that fluxes are around and below 2^-126
(FP32 subnormals), cotangents and directions of 1e-30 and of a few ones
among zeros: the marches must still give the naive kernels' bits.
"""
import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(130, 9, 4), (71, 9, 4)])
@pytest.mark.parametrize("scale", [1e-5, 1e-17, 1e-24])
@pytest.mark.parametrize("c_r", [0.0, 1e-9])
def test_marches_keep_naive_bits_for_tiny_sums(shape, scale, c_r):
    from paper_2304_11274_gb300.api import Grid
    prob = synth.round_to_f32(synth.make_problem(*shape, seed=8, connectivity=10, c_r=c_r))
    perm = prob.perm * np.where(np.random.default_rng(4).random(prob.n) < 0.5, scale, 1.0)
    pn = prob.pn.copy()
    pn[: prob.n // 2] = prob.p[: prob.n // 2]  # no accumulation in half of the cells
    rng = np.random.default_rng(6)
    ws = [rng.standard_normal(prob.n), 1e-30 * rng.standard_normal(prob.n), (rng.random(prob.n) < 0.01) * 1.0]
    with Grid(*shape, prob.phys, "mixed", perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, pn)
        bits = lambda ts: [t.view(torch.int64 if t.dtype == torch.float64 else torch.int32).clone() for t in ts]
        ref = bits(g.assemble_jacobian(kernel="naive"))
        for kernel in ("tiled", "tiled2"):
            assert all(torch.equal(a, b) for a, b in zip(bits(g.assemble_jacobian(kernel=kernel)), ref)), kernel
        assert torch.equal(g.assemble_residual().view(torch.int64), ref[0])
        for w in ws:
            a, b = g.jvp(w, want_residual=True), g.jvp(w, want_residual=True, kernel="naive")
            assert torch.equal(a[0], b[0]) and torch.equal(a[1].view(torch.int64), ref[0])
            b = bits(g.vjp(w, kernel="naive"))
            for kernel in ("tiled", "tiled2"):
                assert all(torch.equal(x, y) for x, y in zip(bits(g.vjp(w, kernel=kernel)), b)), kernel
        g.sync_status()


@pytest.mark.parametrize("shape", [(130, 9, 4), (71, 9, 4)])
def test_every_march_reports_nan_sums(shape):
    """Permeabilities below the FP32 range make 1 / (2 k) infinite and the
    adjoint's sums NaN while g_p stays finite; a NaN pressure makes every sum
    of its rows NaN."""
    from paper_2304_11274_gb300 import TPFAError
    from paper_2304_11274_gb300.api import Grid
    prob = synth.round_to_f32(synth.make_problem(*shape, seed=8, connectivity=10))
    perm = prob.perm * np.where(np.random.default_rng(4).random(prob.n) < 0.5, 1e-28, 1.0)
    p = prob.p.copy()
    p[prob.n // 2] = np.nan
    v = np.random.default_rng(6).standard_normal(prob.n)
    with Grid(*shape, prob.phys, "mixed", perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        for kernel in ("naive", "tiled", "tiled2"):
            g.vjp(v, kernel=kernel)
            with pytest.raises(TPFAError, match="NONFINITE"):
                g.sync_status()
        g.set_state(p, prob.pn)
        calls = [lambda k=k: g.assemble_jacobian(kernel=k) for k in ("naive", "tiled", "tiled2")]
        calls += [g.assemble_residual, lambda: g.jvp(v), lambda: g.vjp(v, want_lnk=False)]
        for call in calls:
            call()
            with pytest.raises(TPFAError, match="NONFINITE"):
                g.sync_status()
