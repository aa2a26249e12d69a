"""The resampling's units where whole tile-planes make units for half to three quarters of
the warps: whole, in parts that divide the planes and in parts that do not."""
import numpy as np
import pytest
import torch

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import build as Bd
from paper_2004_05962_gb300 import synth

VOLUMES = [((97, 290, 64), (4, 3, 6)), ((354, 167, 96), (5, 5, 8)), ((160, 192, 192), (5, 5, 5)), ((128, 128, 140), (7, 2, 3)), ((131, 253, 165), (8, 4, 4))]


@pytest.mark.parametrize("shape,spacing", VOLUMES, ids=[f"{s}-{d}" for s, d in VOLUMES])
def test_selfcheck(shape, spacing):
    Bd.build()
    for op in ("resample", "resample_grad"):
        n, msg = P.bsi_selfcheck_ranges([shape], [spacing], op, cover=True)
        assert n == 0, msg


@pytest.mark.gpu
@pytest.mark.parametrize("shape,spacing", VOLUMES, ids=[f"{s}-{d}" for s, d in VOLUMES])
def test_parts_do_not_change_a_voxel(shape, spacing):
    """The same bits as a sub-volume of the first tile-planes, whose few units take other parts."""
    dev = torch.device("cuda", 0)
    phi = torch.from_numpy(synth.uniform_phi(shape, spacing, -2, 2, seed=sum(shape))).to(dev)
    F = torch.from_numpy(synth.blob_image(shape, seed=5).astype(np.float32)).to(dev)
    got = P.bsi_resample_forward(phi, shape, spacing, F)
    part = (2 * spacing[0], shape[1], shape[2])
    few = P.bsi_resample_forward(phi[:5].contiguous(), part, spacing, F)
    assert torch.equal(got[:part[0]], few)
    assert P.bsi_check_device_status() == 0
