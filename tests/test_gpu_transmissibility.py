"""Owned transmissibilities of the mixed path against the FP64 formula.

The kernel evaluates 2 (area/d) / (1/k_K + 1/k_L) in FP32 pairs and keeps the
FP32 result only where every number within 2^-40 of the pair rounds to it, so
the stored values must be the rounded values of the FP64 formula exactly:
the pair's error and the FP64 formula's are both far below 2^-40.  (The FP64
formula here is torch's, whose roundings can differ from the library's by a
few 2^-53; that moves a rounded FP32 value only if it lies within that of a
rounding boundary, about one link in 10^7.)
"""
import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu


def _formula(k, axes, geo):
    a, b = axes
    T = 2.0 * k[a] * k[b] / (k[a] + k[b]) * geo
    return torch.where((k[a] > 0) & (k[b] > 0), T, 0.0)


# tile edges (32 x 8 cells, runs of 4 planes), single rows and columns
@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 9, 5), (64, 8, 4), (31, 7, 9), (1, 300, 3), (97, 1, 2)])
@pytest.mark.parametrize("log_k", [False, True])
@pytest.mark.parametrize("spread", ["usual", "wide"])
def test_mixed_transmissibilities_are_the_rounded_fp64_values(shape, log_k, spread):
    from paper_2304_11274_gb300.api import Grid
    nx, ny, nz = shape
    phys = synth.physics(connectivity=10)
    rng = np.random.default_rng(nx * ny + nz)
    n = nx * ny * nz
    lk = rng.normal(-13.0, 0.5, n) if spread == "usual" else rng.uniform(-45.0, 12.0, n)
    k = np.power(10.0, lk)
    if spread == "wide":
        k[rng.random(n) < 0.05] = 0.0
    ones = np.full(n, 0.2)
    kt = torch.as_tensor(k, device="cuda")
    with Grid(nx, ny, nz, phys, "mixed", np.full(n, 1e-13) if log_k else k, ones, ones) as g:
        if log_k:
            lnk = torch.log(kt)  # -inf where k = 0
            g.set_log_permeability(lnk)
            kt = torch.exp(lnk)
        got = [g.transmissibility(w).view(nz, ny, nx) for w in range(5)]
        g.sync_status()
    kt = kt.view(nz, ny, nx)
    dx, dy, dz = phys["dx"], phys["dy"], phys["dz"]
    al, lo, hi = slice(None), slice(None, -1), slice(1, None)
    links = [((al, al, lo), (al, al, hi), dy * dz / dx), ((al, lo, al), (al, hi, al), dx * dz / dy),
             ((lo, al, al), (hi, al, al), dx * dy / dz),
             ((al, lo, lo), (al, hi, hi), dz * dx * dy / (dx * dx + dy * dy)),
             ((al, lo, hi), (al, hi, lo), dz * dx * dy / (dx * dx + dy * dy))]
    for T, (a, b, geo) in zip(got, links):
        want = torch.zeros_like(T)
        want[a] = _formula(kt, (a, b), geo).float()
        assert torch.equal(T, want)
