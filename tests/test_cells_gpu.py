"""The kernels on x-cells of any width (bsi_cells_forward.cu, bsi_cells_adjoint.cu)
where their split can go wrong, against the FP64 oracle: every run length, cells
shared by several lanes, vector runs and the same geometry off the 16-byte
boundary, cells cut by either end of the volume, z-cells split into several units,
strips of few cells, the widest spacing."""
import numpy as np
import pytest
import torch

import oracle
import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import synth
from gpu_util import ADJ_TOL, FWD_TOL, adj_err, dev, fwd_err, gpu_adjoint, gpu_forward

pytestmark = pytest.mark.gpu

# integer x-spacings above 8 with at least 16 rows per cell (shape, spacing), (z, y, x)
WIDE = [
    ((20, 18, 100), (5, 4, 9)),          # two lanes per cell, cut last cell
    ((26, 30, 128), (12, 12, 12)),       # vector runs of 4, z-cells split, cut last cell
    ((26, 30, 127), (12, 12, 12)),       # the same spacing, rows off 16-byte boundaries
    ((9, 17, 16), (16, 16, 16)),         # one cell per row
    ((17, 33, 197), (16, 8, 64)),        # the widest spacing, ten lanes per cell
    ((17, 20, 256), (16, 4, 64)),        # the same in vector runs: two cells per strip
    ((70, 70, 45), (64, 64, 22)),        # 64 planes and rows per unit
    ((5, 40, 330), (4, 4, 31)),          # several strips
    ((40, 16, 13), (4, 16, 9)),          # fewer voxels than half a warp
]


def _shifted(t, k=1):
    """t's values in an array that starts k elements off a 16-byte boundary."""
    buf = torch.empty(t.numel() + 4, dtype=t.dtype, device=t.device)
    v = buf[k:k + t.numel()].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("shape,spacing", WIDE, ids=[f"{s}-{d}" for s, d in WIDE])
def test_wide_cells_match_oracle(shape, spacing):
    phi = synth.uniform_phi(shape, spacing, -2, 2, seed=sum(shape) + sum(spacing))
    err, tol = fwd_err(gpu_forward(phi, shape, spacing), phi, shape, spacing)
    assert err <= tol, (err, tol)
    out = _shifted(torch.zeros(shape + (3,), device=dev()))
    P.bsi_field_forward(torch.from_numpy(phi).to(dev()), shape, spacing, out=out)
    err, tol = fwd_err(out, phi, shape, spacing)
    assert err <= tol, (err, tol)
    g = synth.normal_field(shape, seed=sum(shape))
    err, tol = adj_err(gpu_adjoint(g, spacing), g, spacing)
    assert err <= tol, (err, tol)
    got = P.bsi_field_adjoint(_shifted(torch.from_numpy(g).to(dev())), spacing)
    err, tol = adj_err(got, g, spacing)
    assert err <= tol, (err, tol)
    assert P.bsi_check_device_status() == 0


# every run length 1..7 (x-spacing num/den just above it), 8-voxel cells in two
# parts, cells cut at the start (shift) and the end, one and several strips
RATIONAL = [((7, 9, 64 + r), (9, 7, 3 * r - 1), (2, 2, 3), (4, 0, r)) for r in range(1, 8)] + [
    ((9, 11, 240), (5, 9, 15), (1, 2, 2), (3, 8, 14)),
    ((30, 9, 31), (61, 5, 37), (2, 2, 5), (60, 1, 36)),
]


@pytest.mark.parametrize("shape,num,den,off", [c for c in RATIONAL if c[1][2] >= c[2][2]],
                         ids=[f"{c[0]}-{c[1]}/{c[2]}+{c[3]}" for c in RATIONAL if c[1][2] >= c[2][2]])
def test_rational_cells_match_oracle(shape, num, den, off):
    off = tuple(min(o, n - 1) for o, n in zip(off, num))
    rng = np.random.default_rng(sum(shape) + sum(num))
    phi = rng.uniform(-2, 2, P.rational_grid_shape(shape, num, den, off) + (3,)).astype(np.float32)
    got = P.bsi_field_forward_rational(torch.from_numpy(phi).to(dev()), shape, num, den, off)
    err = float(np.max(np.abs(got.double().cpu().numpy() - oracle.forward_rational(phi, shape, num, den, off))))
    assert err <= FWD_TOL * 2.0, err
    G = rng.standard_normal(shape + (3,)).astype(np.float32)
    want = oracle.adjoint_rational(G, num, den, off)
    got = P.bsi_field_adjoint_rational(_shifted(torch.from_numpy(G).to(dev()), 2), num, den, off)
    err = float(np.max(np.abs(got.double().cpu().numpy() - want)))
    assert err <= ADJ_TOL * float(np.max(np.abs(want))), err
    assert P.bsi_check_device_status() == 0


@pytest.mark.parametrize("shape,spacing", [((26, 30, 128), (12, 12, 12)), ((20, 18, 101), (5, 4, 9))])
def test_wide_adjoint_keeps_an_infinity_in_its_support(shape, spacing):
    """An infinite voxel gradient reaches the control points of its own cell's
    neighbourhood and no other (lanes without a voxel add exact zeros)."""
    g = synth.normal_field(shape, seed=3)
    z, y, x = shape[0] - 1, shape[1] // 2, shape[2] - 1
    g[z, y, x] = np.inf
    got = gpu_adjoint(g, spacing)
    got = got if isinstance(got, np.ndarray) else got.cpu().numpy()
    c = tuple(v // d for v, d in zip((z, y, x), spacing))
    out = np.ones(got.shape, bool)
    out[c[0]:c[0] + 4, c[1]:c[1] + 4, c[2]:c[2] + 4] = False
    assert np.isfinite(got[out]).all()
    assert not np.isfinite(got[~out]).all()
