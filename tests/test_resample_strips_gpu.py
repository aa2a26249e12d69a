"""The resampling's strips and parts of tile-planes: the same bits whatever the
strips' width."""
import pytest
import torch

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu

# (volume, spacing): one strip, strips evened out, more than half as many again (kept
# wide), rows of 1, 32 and 129 voxels, tile-planes cut by the volume's end
CASES = [
    ((64, 64, 64), (5, 5, 5)),
    ((9, 20, 300), (4, 3, 8)),
    ((11, 13, 230), (8, 2, 7)),
    ((10, 12, 175), (5, 4, 7)),
    ((7, 9, 129), (3, 3, 6)),
    ((20, 33, 32), (16, 5, 8)),
    ((13, 8, 1), (2, 2, 5)),
    ((17, 30, 400), (6, 5, 3)),
]


@pytest.mark.parametrize("shape,spacing", CASES, ids=[f"{c[0]}-{c[1]}" for c in CASES])
def test_strips_do_not_change_a_bit(shape, spacing):
    phi = torch.from_numpy(synth.uniform_phi(shape, spacing, -2.0, 2.0, seed=21)).to(dev())
    F = torch.from_numpy(synth.blob_image(shape, seed=22)).float().to(dev())
    w = torch.from_numpy(synth.normal_field(shape, seed=23)[..., 0].copy()).to(dev())

    def both():
        return P.bsi_resample_forward(phi, shape, spacing, F), P.bsi_resample_backward(phi, shape, spacing, F, w)

    got = both()
    try:
        P.bsi_set_tile_configs([dict(fwd_strip_tiles=7)])
        want = both()
    finally:
        P.bsi_set_tile_configs([])
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert P.bsi_check_device_status() == 0
