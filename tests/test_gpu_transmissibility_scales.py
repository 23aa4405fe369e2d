"""Mixed transmissibilities of cells whose face area over distance is far from 1 m.

As in test_gpu_transmissibility.py the stored values must be the FP64 formula's,
rounded.  Below 2^-90 the geometry has no FP32 pair of 45 bits (its trailing
half, or a remainder, is subnormal), so the pair's value cannot decide the
rounding; the sizes here reach from there to beyond the FP32 range.
"""
import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth
from test_gpu_transmissibility import _formula

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [1e-45, 1e-39, 1e-36, 1e-34, 1e-32, 1e-28, 1e26, 1e30, 1e38, 1e40])
def test_values_are_the_rounded_fp64_formula(length):
    from paper_2304_11274_gb300.api import Grid
    nx, ny, nz = 61, 40, 9
    n = nx * ny * nz
    phys = synth.physics(connectivity=10, dx=length, dy=length, dz=length)
    # transmissibilities around 1e-13 and above whatever the length
    k = np.power(10.0, np.random.default_rng(2).uniform(-13.0, -5.0, n)) / length
    ones = np.full(n, 0.2)
    with Grid(nx, ny, nz, phys, "mixed", k, ones, ones) as g:
        got = [g.transmissibility(w).view(nz, ny, nx) for w in range(5)]
        g.sync_status()
    kt = torch.as_tensor(k, device="cuda").view(nz, ny, nx)
    al, lo, hi = slice(None), slice(None, -1), slice(1, None)
    a, d = length * length / length, length * length * length / (length * length + length * length)
    links = [((al, al, lo), (al, al, hi), a), ((al, lo, al), (al, hi, al), a), ((lo, al, al), (hi, al, al), a),
             ((al, lo, lo), (al, hi, hi), d), ((al, lo, hi), (al, hi, lo), d)]
    for T, (x, y, geo) in zip(got, links):
        want = torch.zeros_like(T)
        want[x] = _formula(kt, (x, y), geo).float()
        assert torch.equal(T, want), int((T != want).sum())
