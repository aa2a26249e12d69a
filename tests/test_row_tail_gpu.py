"""The row-copy adjoint at widths whose cut last x-tile ends a strip of 32 tiles (just
under 58 and 87 tiles): every staged row's zeros end where the next row's values begin.
Against the FP64 oracle, single volumes in units of tile-planes and all in one batch."""
import numpy as np
import pytest
import torch

import oracle
import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import synth
from gpu_util import ADJ_TOL, adj_err, dev
from test_resample_gpu import _kink_free

pytestmark = pytest.mark.gpu

# units enough that a call of one volume takes units of tile-planes too
SINGLE = [((45, 111, 347), (3, 3, 6)), ((45, 111, 405), (3, 3, 7)), ((45, 111, 463), (3, 3, 8)), ((45, 111, 289), (3, 3, 5))]
BATCH = [((9, 17, 347), (3, 6, 6)), ((7, 9, 346), (3, 4, 6)), ((9, 17, 405), (3, 8, 7)), ((9, 17, 463), (3, 8, 8)),
         ((5, 11, 461), (2, 5, 8)), ((6, 9, 231), (3, 5, 4)), ((6, 9, 289), (3, 5, 5)), ((4, 9, 690), (2, 5, 8)),
         ((6, 9, 231), (3, 5, 64)), ((4, 7, 460), (2, 5, 8))]


def _shifted(t):
    """t's values in an array that starts 4 bytes off a 16-byte boundary."""
    v = torch.empty(t.numel() + 4, device=t.device)[1:1 + t.numel()].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("shape,spacing", SINGLE, ids=[f"{s}-{d}" for s, d in SINGLE])
def test_single_volume_adjoint(shape, spacing):
    g = synth.normal_field(shape, seed=sum(shape))
    gt = torch.from_numpy(g).to(dev())
    for t in (gt, _shifted(gt)):
        err, tol = adj_err(P.bsi_field_adjoint(t, spacing), g, spacing)
        assert err <= tol, (err, tol)
    assert P.bsi_check_device_status() == 0


def test_batch_adjoint():
    gs = [synth.normal_field(s, seed=sum(s)) for s, _ in BATCH]
    gts = [_shifted(torch.from_numpy(g).to(dev())) for g in gs]
    for g, got, (_, sp) in zip(gs, P.bsi_field_adjoint_batched(gts, [d for _, d in BATCH]), BATCH):
        err, tol = adj_err(got, g, sp)
        assert err <= tol, (g.shape, sp, err, tol)
    assert P.bsi_check_device_status() == 0


@pytest.mark.parametrize("shape,spacing", SINGLE[:3], ids=[f"{s}-{d}" for s, d in SINGLE[:3]])
def test_resample_backward(shape, spacing):
    phi = synth.uniform_phi(shape, spacing, -2, 2, seed=17)
    F = synth.blob_image(shape, seed=18).astype(np.float32)
    dW = synth.normal_field(shape, seed=19)[..., 0].copy()
    dW[~_kink_free(phi, shape, spacing)] = 0.0
    got = P.bsi_resample_backward(*(torch.from_numpy(phi).to(dev()), shape, spacing),
                                  *(torch.from_numpy(a).to(dev()) for a in (F, dW)))
    want = oracle.resample_backward(phi, shape, spacing, F, dW)
    err = float(np.max(np.abs(got.double().cpu().numpy() - want)))
    assert err <= ADJ_TOL * max(float(np.max(np.abs(want))), 1e-30), err
