"""Small sums, small directions and small masses: the marches' values are the
naive kernels', and cost no second pass over the rows.

Cells switched off by a permeability of 1e-35 m^2 have flux sums of about
1e-22; a direction that decays as a bell does has entries below every FP32
number.  Neither needs more than the marches' own conversions.  A march that
computed such rows again one thread per cell took two to six times as long;
1.5 times is allowed.
"""
import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth
from test_gpu_impermeable_cells import median_us

pytestmark = pytest.mark.gpu


def _problem(shape, what, c_r):
    prob = synth.round_to_f32(synth.make_problem(*shape, seed=8, connectivity=10, c_r=c_r))
    rng = np.random.default_rng(4)
    half = rng.random(prob.n) < 0.5
    perm, poro, p, pn = prob.perm.copy(), prob.poro.copy(), prob.p.copy(), prob.pn.copy()
    pn[: prob.n // 2] = p[: prob.n // 2]
    if what == "off":
        perm = np.where(half, 10.0 ** rng.uniform(-48.0, -28.0, prob.n), perm)
    elif what == "large":  # results of 2^60 and more
        perm = perm * np.where(half, 1e22, 1e13)
    elif what == "mass":  # previous masses that are FP32 subnormals, or zero
        poro = np.where(half, 10.0 ** rng.uniform(-46.0, -36.0, prob.n), np.where(rng.random(prob.n) < 0.5, 0.0, poro))
        perm = np.where(half, 1e-40, perm)
    elif what == "step":  # pressure changes whose accumulation factor is an FP32 subnormal
        p = np.where(half, 10.0 ** rng.uniform(-38.0, -26.0, prob.n), 0.0)
        pn = np.where(rng.random(prob.n) < 0.5, 10.0 ** rng.uniform(-38.0, -26.0, prob.n), 0.0)
        perm = np.where(half, 0.0, 1e-38)
    return prob, perm, poro, p, pn


@pytest.mark.parametrize("shape", [(130, 9, 4), (71, 9, 4), (256, 5, 3)])
@pytest.mark.parametrize("what", ["off", "large", "mass", "step"])
@pytest.mark.parametrize("c_r", [0.0, 1e-9])
def test_values_are_the_naive_kernels(shape, what, c_r):
    from paper_2304_11274_gb300.api import Grid
    prob, perm, poro, p, pn = _problem(shape, what, c_r)
    rng = np.random.default_rng(6)
    ws = [rng.standard_normal(prob.n) * 10.0 ** rng.uniform(-50.0, -30.0, prob.n),
          np.where(rng.random(prob.n) < 0.5, rng.standard_normal(prob.n) * 10.0 ** rng.uniform(-330.0, 10.0, prob.n), 0.0)]
    with Grid(*shape, prob.phys, "mixed", perm, poro, prob.depth) as g:
        g.set_state(p, pn)
        ref = [t.clone() for t in g.assemble_jacobian(kernel="naive")]
        for kernel in ("tiled", "tiled2"):
            assert all(torch.equal(a, b) for a, b in zip(g.assemble_jacobian(kernel=kernel), ref)), kernel
        assert torch.equal(g.assemble_residual(), ref[0])
        for w in ws:
            a, b = g.jvp(w, want_residual=True), g.jvp(w, want_residual=True, kernel="naive")
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], ref[0]) and torch.equal(b[1], ref[0])
            assert torch.equal(g.jvp(w)[0], b[0])
        g.sync_status()


@pytest.mark.parametrize("shape", [(130, 9, 4), (71, 9, 4), (256, 5, 3)])
def test_overflow_is_reported(shape):
    """Sums beyond the FP32 range, and directions beyond it."""
    from paper_2304_11274_gb300 import TPFAError
    from paper_2304_11274_gb300.api import Grid
    prob = synth.round_to_f32(synth.make_problem(*shape, seed=8, connectivity=10))
    w = np.random.default_rng(6).standard_normal(prob.n)
    with Grid(*shape, prob.phys, "mixed", prob.perm * 1e44, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        for call in [lambda k=k: g.assemble_jacobian(kernel=k) for k in ("naive", "tiled", "tiled2")] + [
                g.assemble_residual]:
            call()
            with pytest.raises(TPFAError, match="NONFINITE"):
                g.sync_status()
        g.set_permeability(prob.perm)
        for kernel in ("naive", "auto"):
            g.jvp(w * 1e60, kernel=kernel)
            with pytest.raises(TPFAError, match="NONFINITE"):
                g.sync_status()
        g.jvp(w * 1e30)
        g.sync_status()


@pytest.mark.parametrize("shape", [(512, 512, 32), (201, 200, 100)])
def test_time_with_cells_switched_off_and_a_decaying_direction(shape):
    from paper_2304_11274_gb300.api import Grid
    prob = synth.round_to_f32(synth.make_problem(*shape, seed=3, connectivity=10))
    off = np.random.default_rng(4).random(prob.n) < 0.05
    w = torch.as_tensor(np.random.default_rng(1).standard_normal(prob.n), device="cuda")
    c = torch.arange(prob.n, device="cuda")
    x, y = c % shape[0] - shape[0] // 2, c // shape[0] % shape[1] - shape[1] // 2
    bell = torch.exp(-(x * x + y * y).double() / (shape[0] / 20.0) ** 2)
    times = []
    for perm, d, pn in ((prob.perm, w, prob.pn), (np.where(off, 1e-35, prob.perm), bell, prob.p)):
        with Grid(*shape, prob.phys, "mixed", perm, prob.poro, prob.depth) as g:
            g.set_state(prob.p, pn)
            outs, Jw = g.empty_outputs(), torch.empty_like(w)
            times.append([median_us(lambda: g.assemble_jacobian(*outs)), median_us(lambda: g.assemble_residual(outs[0])),
                          median_us(lambda: g.jvp(d, out=Jw))])
            g.sync_status()
    assert all(b <= 1.5 * a for a, b in zip(*times)), times
