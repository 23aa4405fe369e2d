"""Ensembles of one or two models: not slower than 32 rows per march everywhere
(they took up to 1.13 times as long, with 64-row marches or a second wave of short
ones that nothing evened out), 1.05 times allowed; and the single launches' bits.
"""
import pytest
import torch

from test_gpu_autotune_choice import _best_us
from test_gpu_ensemble import _models, _same, _single

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(223, 129, 126)], [(189, 82, 70), (97, 187, 33)], [(189, 163, 35), (91, 115, 74)],
                                    [(300, 300, 60)]])
@pytest.mark.parametrize("conn", [6, 10])
def test_few_models(shapes, conn, tmp_path):
    from paper_2304_11274_gb300.api import Ensemble
    _, grids = _models(shapes, conn=conn)
    singles = [_single(g) for g in grids]
    cells = sum(g.n for g in grids)
    cache = tmp_path / "t.txt"
    cache.write_text("ensemble/sm103/M%d/c%d/r0/n%d 32 4\n" % (len(grids), conn, cells.bit_length() - 1))
    times = []
    with Ensemble(grids) as ens:
        outs = ens.allocate_outputs()
        for tune in (False, True):
            if tune:  # a cached choice of at most 32 rows
                assert ens.autotune(str(cache))["rows_per_march"] == 32
            times.append(_best_us(ens.assemble))
            for m, g in enumerate(grids):
                assert _same(outs[m], singles[m]), m
                g.sync_status()
    for g in grids:
        g.close()
    assert times[0] <= 1.05 * times[1], times
