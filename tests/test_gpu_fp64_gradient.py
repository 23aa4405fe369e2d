"""The FP64 gradient with respect to ln k against extended precision, and the
FP64 transmissibilities against the plain formula.

Elementwise: a term F (v_K - v_L) k_L / (k_K + k_L) takes fewer than 32
roundings, each within 2^-53 of the magnitudes that enter it (the pressure
and gravity parts of the potential difference, |v_K| + |v_L|); 64 are allowed.
In the 2-norm: no further from the exact value than the formula itself
evaluated in plain FP64 with the ratio as a quotient (5 % for the scatter of
the other roundings; the ratio taken from T alone is 15 % further).
"""
import numpy as np
import pytest
import torch

from paper_2304_11274_gb300 import synth

pytestmark = pytest.mark.gpu

AL, LO, HI = slice(None), slice(None, -1), slice(1, None)


def _links(phys, conn):
    dx, dy, dz = phys["dx"], phys["dy"], phys["dz"]
    out = [((AL, AL, LO), (AL, AL, HI), dy * dz / dx), ((AL, LO, AL), (AL, HI, AL), dx * dz / dy),
           ((LO, AL, AL), (HI, AL, AL), dx * dy / dz)]
    if conn == 10:
        d = dz * dx * dy / (dx * dx + dy * dy)
        out += [((AL, LO, LO), (AL, HI, HI), d), ((AL, LO, HI), (AL, HI, LO), d)]
    return out


def _gradient(prob, v, dtype):
    """g_lnk and the sum of its terms' magnitudes, in dtype."""
    ph = {k: dtype(x) for k, x in prob.phys.items()}
    shape = (prob.nz, prob.ny, prob.nx)
    k, p, z, v = (np.asarray(x, dtype=np.float64).reshape(shape).astype(dtype) for x in
                  (prob.perm, prob.p, prob.depth, v))
    rho = ph["rho_ref"] * np.exp(ph["c_f"] * (p - ph["p_ref"]))
    g, size = np.zeros(shape, dtype), np.zeros(shape, dtype)
    for a, b, geo in _links(ph, int(prob.phys["connectivity"])):
        s = k[a] + k[b]
        s = np.where(s > 0, s, dtype(1))
        T = 2 * k[a] * k[b] / s * geo / ph["mu"]
        hg = ph["g"] / 2 * (z[a] - z[b])
        dphi = (p[a] - p[b]) - (rho[a] + rho[b]) * hg
        F = T * np.where(dphi > 0, rho[a], rho[b]) * dphi
        m = T * rho[a] * (abs(p[a] - p[b]) + (rho[a] + rho[b]) * abs(hg)) * (abs(v[a]) + abs(v[b]))
        g[a] += (v[a] - v[b]) * (F * (k[b] / s))
        g[b] += (v[a] - v[b]) * (F * (k[a] / s))
        size[a] += m * (k[b] / s)
        size[b] += m * (k[a] / s)
    return g.reshape(-1), size.reshape(-1)


def _run(prob, v):
    from paper_2304_11274_gb300.api import Grid
    with Grid(prob.nx, prob.ny, prob.nz, prob.phys, "fp64", prob.perm, prob.poro, prob.depth) as g:
        g.set_state(prob.p, prob.pn)
        g_p, g_lnk = g.vjp(v)
        assert torch.equal(g.vjp(v, want_lnk=False)[0], g_p)
        g.sync_status()
    return g_lnk.cpu().numpy()


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 300, 3), (300, 1, 2), (129, 7, 5), (33, 9, 40), (9, 28, 70), (2, 2, 130)])
@pytest.mark.parametrize("conn", [6, 10])
@pytest.mark.parametrize("perm", ["usual", "impermeable", "wide", "large"])
def test_gradient_elementwise(shape, conn, perm):
    prob = synth.make_problem(*shape, seed=sum(shape), connectivity=conn)
    rng = np.random.default_rng(3)
    if perm == "impermeable":
        prob.perm = np.where(rng.random(prob.n) < 0.1, 0.0, prob.perm)
    elif perm == "wide":
        prob.perm = 10.0 ** rng.uniform(-60.0, -5.0, prob.n)
    elif perm == "large":
        prob.perm = prob.perm * 10.0 ** rng.uniform(25.0, 40.0, prob.n)
    v = rng.standard_normal(prob.n)
    want, size = _gradient(prob, v, np.longdouble)
    assert (abs(_run(prob, v) - want) <= 64 * 2.0 ** -53 * size).all()


@pytest.mark.parametrize("conn", [6, 10])
def test_gradient_error_is_the_formulas(conn):
    prob = synth.make_problem(60, 50, 40, seed=2, connectivity=conn)
    v = np.random.default_rng(3).standard_normal(prob.n)
    want, _ = _gradient(prob, v, np.longdouble)
    err = [np.linalg.norm((x - want).astype(np.float64)) for x in (_run(prob, v), _gradient(prob, v, np.float64)[0])]
    assert err[0] <= 1.05 * err[1], err


# one cell, ragged tiles, single rows and columns, several runs of four planes
@pytest.mark.parametrize("shape", [(1, 1, 1), (129, 7, 5), (97, 83, 4), (31, 7, 9), (1, 300, 3), (300, 1, 2)])
@pytest.mark.parametrize("spread", ["usual", "wide"])
def test_transmissibilities_have_the_formulas_bits(shape, spread):
    from paper_2304_11274_gb300.api import Grid
    nx, ny, nz = shape
    phys = synth.physics(connectivity=10)
    rng = np.random.default_rng(nx * ny + nz)
    n = nx * ny * nz
    k = np.power(10.0, rng.normal(-13.0, 0.5, n) if spread == "usual" else rng.uniform(-45.0, 12.0, n))
    if spread == "wide":
        k[rng.random(n) < 0.05] = 0.0
    ones = np.full(n, 0.2)
    with Grid(nx, ny, nz, phys, "fp64", k, ones, ones) as g:
        got = [g.transmissibility(w).view(nz, ny, nx).cpu().numpy() for w in range(5)]
        g.sync_status()
    k = k.reshape(nz, ny, nx)
    for T, (a, b, geo) in zip(got, _links(phys, 10)):
        want = np.zeros_like(T)
        s = k[a] + k[b]
        want[a] = np.where((k[a] > 0) & (k[b] > 0), 2.0 * k[a] * k[b] / np.where(s > 0, s, 1.0) * geo, 0.0)
        assert np.array_equal(T, want)
