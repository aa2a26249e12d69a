"""The row-copy adjoint at x-spacings above 8 (units of tile-planes: batches, and one
volume with fewer than 16 rows per cell) against the FP64 oracle: tile widths of every
remainder of four voxels, cut tiles, one and several rows per plane, few units (stages of
two rows) and enough to fill the GPU (stages of one)."""
import pytest
import torch

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import synth
from gpu_util import adj_err, dev, gpu_adjoint

pytestmark = pytest.mark.gpu

FEW = [((7, 9, 9 * k + c), (3, 4, k)) for k, c in ((9, 0), (10, 3), (11, 10), (12, 1), (13, 5), (14, 13), (15, 2), (16, 0))] + [
    ((5, 6, 130), (2, 1, 13)), ((9, 1, 200), (4, 5, 64)), ((20, 33, 63), (16, 16, 64)), ((6, 40, 64), (3, 20, 32))]
MANY = [((24, 24, 150), (3, 3, 9 + i % 9)) for i in range(24)] + [((24, 25, 151), (3, 1, 20 + i)) for i in range(8)]


@pytest.mark.parametrize("volumes", [FEW, MANY], ids=["few_units", "many_units"])
def test_batch(volumes):
    gs = [synth.normal_field(s, seed=sum(s) + i) for i, (s, _) in enumerate(volumes)]
    got = P.bsi_field_adjoint_batched([torch.from_numpy(g).to(dev()) for g in gs], [d for _, d in volumes])
    for g, t, (_, sp) in zip(gs, got, volumes):
        err, tol = adj_err(t, g, sp)
        assert err <= tol, (g.shape, sp, err, tol)
    assert P.bsi_check_device_status() == 0


@pytest.mark.parametrize("shape,spacing", [((10, 11, 77), (3, 4, 13)), ((50, 60, 140), (1, 4, 22)), ((9, 10, 65), (15, 1, 64)),
                                           ((120, 130, 127), (3, 3, 17))])
def test_one_volume_of_few_rows_per_cell(shape, spacing):
    g = synth.normal_field(shape, seed=sum(shape))
    err, tol = adj_err(gpu_adjoint(g, spacing), g, spacing)
    assert err <= tol, (err, tol)
    assert P.bsi_check_device_status() == 0
