"""Small volumes: tile-planes split over the idle warps (forward), units of cells
(adjoint)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import synth
from gpu_util import ADJ_TOL, dev

pytestmark = pytest.mark.gpu

# (volume, spacing): planes that do not divide into the parts, tile-planes cut by the
# volume's end, one voxel, one plane, every store path, more units than warps
CASES = [
    ((64, 64, 64), (5, 5, 5)),
    ((17, 23, 41), (7, 3, 8)),
    ((9, 12, 200), (64, 2, 6)),
    ((1, 40, 30), (8, 8, 3)),
    ((1, 1, 1), (5, 5, 5)),
    ((30, 64, 64), (6, 4, 4)),
    ((20, 33, 71), (16, 16, 12)),
    ((120, 120, 128), (3, 4, 5)),
    ((200, 200, 64), (3, 3, 3)),
]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("shape,spacing", CASES, ids=[f"{c[0]}-{c[1]}" for c in CASES])
def test_forward_parts_equal_whole_planes(shape, spacing, dtype):
    """The same bits as the whole tile-planes of a batch."""
    phi = torch.from_numpy(synth.uniform_phi(shape, spacing, -3.0, 3.0, seed=11)).to(dev())
    got = P.bsi_field_forward(phi, shape, spacing, out_dtype=dtype)
    want = P.bsi_field_forward_batched([phi, phi], [shape, shape], [spacing, spacing], out_dtype=dtype)
    assert torch.equal(got, want[0]) and torch.equal(got, want[1])
    scalar = P.bsi_scalar_forward(phi[..., 0].contiguous(), shape, spacing, out_dtype=dtype)
    assert torch.equal(scalar, want[0][..., 0])


@pytest.mark.parametrize("shape,spacing", CASES, ids=[f"{c[0]}-{c[1]}" for c in CASES])
def test_adjoint_on_cells_matches_oracle(shape, spacing):
    """One small volume (units of cells) and the same volume in a batch (units of
    tile-planes), each against the oracle."""
    G = synth.normal_field(shape, seed=13)
    want = oracle.adjoint(G, spacing)
    g = torch.from_numpy(G).to(dev())
    off = torch.zeros(G.size + 1, device=dev())[1:].view(G.shape)   # rows off 16-byte boundaries
    off.copy_(g)
    got = [P.bsi_field_adjoint(g, spacing), P.bsi_field_adjoint(off, spacing),
           P.bsi_field_adjoint_batched([g, off], [spacing, spacing])[1]]
    for d in got:
        err = float(np.max(np.abs(d.double().cpu().numpy() - want)))
        assert err <= ADJ_TOL * max(float(np.max(np.abs(want))), 1e-30), err
    assert P.bsi_check_device_status() == 0
