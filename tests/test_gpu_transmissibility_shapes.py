"""Transmissibilities and the stored k on shapes whose tiles are small or few: from
one cell per plane to planes of a few tiles, from k and from ln k.  FP64 values
are the formula's bits, mixed ones the formula's, rounded; and a call costs no
more than 1.5 times one on a grid of as many cells in 8 x 8 planes (it cost up to
6.5 times as much with one warp per cell of 1 x 1 planes)."""
import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth
from test_gpu_autotune_choice import _best_us
from test_gpu_transmissibility import _formula

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 70), (2, 1, 9), (1, 3, 40), (2, 2, 33), (4, 4, 17), (5, 3, 4), (17, 1, 5), (7, 9, 11)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("conn", [6, 10])
@pytest.mark.parametrize("log_k", [False, True])
def test_values(shape, precision, conn, log_k):
    from paper_2304_11274_gb300.api import Grid
    nx, ny, nz = shape
    phys = synth.physics(connectivity=conn)
    rng = np.random.default_rng(nx * ny + nz)
    n = nx * ny * nz
    k = np.power(10.0, rng.normal(-13.0, 1.0, n))
    k[rng.random(n) < 0.05] = 0.0
    ones = np.full(n, 0.2)
    kt = torch.as_tensor(k, device="cuda")
    with Grid(nx, ny, nz, phys, precision, np.full(n, 1e-13) if log_k else k, ones, ones) as g:
        if log_k:
            lnk = torch.log(kt)
            g.set_log_permeability(lnk)
            kt = torch.exp(lnk)
        got = [g.transmissibility(w).view(nz, ny, nx) for w in range(5 if conn == 10 else 3)]
        g.sync_status()
    kt = kt.view(nz, ny, nx)
    dx, dy, dz = phys["dx"], phys["dy"], phys["dz"]
    al, lo, hi = slice(None), slice(None, -1), slice(1, None)
    d = dz * dx * dy / (dx * dx + dy * dy)
    links = [((al, al, lo), (al, al, hi), dy * dz / dx), ((al, lo, al), (al, hi, al), dx * dz / dy),
             ((lo, al, al), (hi, al, al), dx * dy / dz), ((al, lo, lo), (al, hi, hi), d), ((al, lo, hi), (al, hi, lo), d)]
    for T, (a, b, geo) in zip(got, links):
        want = torch.zeros(nz, ny, nx, dtype=torch.float64, device="cuda")
        want[a] = _formula(kt, (a, b), geo)
        assert torch.equal(T, want.to(T.dtype))


@pytest.mark.parametrize("shape", [(1, 1, 102400), (2, 2, 25600), (4, 4, 6400)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_time_on_thin_columns(shape, precision):
    from paper_2304_11274_gb300.api import Grid
    n = 102400
    k = torch.as_tensor(np.power(10.0, np.random.default_rng(1).normal(-13.0, 0.5, n)), device="cuda")
    lnk, ones = torch.log(k), torch.full((n,), 0.2, dtype=torch.float64, device="cuda")
    times = []
    for s in ((8, 8, 1600), shape):
        with Grid(*s, synth.physics(connectivity=10), precision, k, ones, ones) as g:
            times.append([_best_us(lambda: g.set_permeability(k)), _best_us(lambda: g.set_log_permeability(lnk))])
    assert all(b <= 1.5 * a + 20.0 for a, b in zip(*times)), times
