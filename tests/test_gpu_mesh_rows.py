"""Meshes at the edges of the assembly's shared-memory stretch of CSR entries.

A block of 128 rows stages 2048 entries (16 per row) and reads longer
stretches directly: blocks of exactly 2048, of two more, a row longer than the
buffer, and last blocks of one and of few rows.  Bars as for every mesh (each
link is within a few units of the last place and no row's sum cancels: the hub
has the lowest pressure).
"""
import dataclasses

import numpy as np
import pytest

import _compare as C
from test_gpu_mesh import EPS, TOL, _prepare, _reference, _run

pytestmark = pytest.mark.gpu


def _rings(n, reach, antipodal):
    """Every cell linked to its `reach` next cells on a ring (and the opposite one)."""
    i = np.arange(n)
    pairs = [(i, (i + d) % n) for d in range(1, reach + 1)]
    if antipodal:
        pairs.append((i[: n // 2], i[: n // 2] + n // 2))
    return np.concatenate([a for a, _ in pairs]), np.concatenate([b for _, b in pairs])


def _connections(name):
    if name == "16 per row":
        return 256, *_rings(256, 7, True)
    if name == "2050 in a block":
        a, b = _rings(256, 7, True)
        return 256, np.append(a, 3), np.append(b, 33)
    if name == "last block of one row":
        return 257, *_rings(257, 3, False)
    i = np.arange(2500)  # a hub row of 2500 entries, the others three or four
    a, b = _rings(2500, 1, False)
    far = (i != 1200) & (np.abs(i - 1200) > 1)
    return 2500, np.append(a, i[far]), np.append(b, np.full(far.sum(), 1200))


@pytest.mark.parametrize("name", ["16 per row", "2050 in a block", "last block of one row", "hub"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("c_r", [0.0, 1e-9])
def test_mesh_rows_around_the_staging_buffer(name, precision, c_r):
    n, ci, cj = _connections(name)
    m = _prepare((n + n // 4, 1, 1), "fp64", 6, c_r)  # (some of its cells are pinched out)
    T = m.T[0] * np.random.default_rng(5).uniform(0.5, 2.0, ci.size)
    p = m.p[:n].copy()
    if name == "hub":
        p[1200] = p.min() - 1e6
    m = dataclasses.replace(m, n=n, V=m.V[:n], poro=m.poro[:n], depth=m.depth[:n], pn=m.pn[:n], p=p,
                            ci=ci.astype(m.ci.dtype), cj=cj.astype(m.cj.dtype), T=T)
    if precision == "mixed":
        from paper_2304_11274_gb300 import synth
        m = synth.round_mesh_to_f32(m)
    got, ref = _run(m, precision), _reference(m, EPS[precision])
    assert np.array_equal(got["rp"], ref["row_ptr"]) and np.array_equal(got["ci"], ref["col_idx"])
    assert np.array_equal(got["R"], got["R_only"])
    J = got["vals"].copy()
    if got["diag"] is not None:
        rows = np.repeat(np.arange(m.n), np.diff(got["rp"]))
        J[got["ci"] == rows] = got["diag"]
    assert C.residual_error(got["R"], ref) <= TOL[precision]
    assert C.jacobian_row_error(J, ref) <= TOL[precision]
