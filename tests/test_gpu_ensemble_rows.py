"""Rows per march chosen model by model in an ensemble: long marches for the
early models, short ones for the last, equal runs, shorter ones still in an
ensemble of few tiles.  Every model's outputs must have the single launch's
bits (the tiling changes no sum), so no tolerance is involved.
"""
import pytest
import torch

from test_gpu_ensemble import _models, _same, _single

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [
    [(256, 200, 96), (100, 65, 40), (70, 25, 9), (31, 129, 3)],  # 64-row marches, then the short tail
    [(64, 64, 32), (33, 7, 5), (1, 1, 1)],                       # a fraction of a tile per block
    [(40, 24, 8)],                                               # exactly one short march
    [(96, 150, 60), (96, 49, 60)],                               # all in the tail, uneven runs
])
@pytest.mark.parametrize("conn", [6, 10])
def test_rows_by_model_keep_the_bits(shapes, conn):
    from paper_2304_11274_gb300.api import Ensemble
    _, grids = _models(shapes, conn=conn)
    singles = [_single(g) for g in grids]
    with Ensemble(grids) as ens:
        outs = ens.allocate_outputs()
        ens.assemble()
        torch.cuda.synchronize()
        for m, g in enumerate(grids):
            assert _same(outs[m], singles[m]), m
            g.sync_status()
    for g in grids:
        g.close()
