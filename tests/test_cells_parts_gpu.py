"""Forward of small volumes of wide cells against the FP64 oracle: units of parts of
y-cells (kernels on cells of any width) and, at non-integer spacing, the windowed kernel,
which takes small volumes and strips that fill few lanes."""
import numpy as np
import pytest
import torch

import oracle
import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import synth
from gpu_util import FWD_TOL, dev, fwd_err, gpu_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,spacing", [((12, 61, 30), (57, 62, 43)), ((1, 64, 64), (64, 64, 64)), ((64, 64, 64), (12, 12, 12)),
                                           ((65, 33, 40), (24, 13, 24)), ((2, 90, 31), (20, 31, 10)), ((30, 30, 61), (16, 16, 8))])
def test_integer_spacing(shape, spacing):
    phi = synth.uniform_phi(shape, spacing, -2, 2, seed=sum(shape))
    err, tol = fwd_err(gpu_forward(phi, shape, spacing), phi, shape, spacing)
    assert err <= tol, (err, tol)
    assert P.bsi_check_device_status() == 0


# (shape, num, den, off): both sides of 10000 rows of 32 voxels, of 32 columns, of 24 columns
# and 60% of the lanes, 512 voxels per row; tall y-cells
RATIONAL = [((39, 256, 30), (47, 47, 47), (10, 10, 10), (3, 0, 9)), ((40, 256, 30), (47, 47, 47), (10, 10, 10), (3, 0, 9)),
            ((9, 20, 130), (5, 25, 9), (2, 2, 2), (1, 0, 7)), ((9, 20, 126), (5, 25, 9), (2, 2, 2), (1, 0, 7)),
            ((61, 70, 100), (121, 250, 401), (10, 10, 20), (0, 3, 4)), ((65, 70, 180), (130, 14, 153), (8, 1, 8), (117, 2, 135)),
            ((65, 70, 180), (130, 11, 153), (8, 1, 8), (117, 2, 135)), ((3, 9, 520), (9, 127, 127), (2, 2, 2), (1, 1, 126)),
            ((12, 61, 30), (57, 437, 298), (1, 7, 7), (0, 1, 2))]


@pytest.mark.parametrize("shape,num,den,off", RATIONAL, ids=[f"{c[0]}-{c[1]}/{c[2]}" for c in RATIONAL])
def test_non_integer_spacing(shape, num, den, off):
    rng = np.random.default_rng(sum(shape))
    phi = rng.uniform(-2, 2, P.rational_grid_shape(shape, num, den, off) + (3,)).astype(np.float32)
    want = oracle.forward_rational(phi, shape, num, den, off)
    flat = torch.zeros(want.size + 1, device=dev())
    for out in (flat[:-1].view(want.shape), flat[1:].view(want.shape)):   # on and off a 16-byte boundary
        P.bsi_field_forward_rational(torch.from_numpy(phi).to(dev()), shape, num, den, off, out=out)
        assert float(np.max(np.abs(out.double().cpu().numpy() - want))) <= FWD_TOL * 2.0
    assert P.bsi_check_device_status() == 0
