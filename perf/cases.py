"""Performance cases of the B-spline interpolation library: the calls a registration program makes.

Volumes are (Z, Y, X) voxels, spacings (dz, dy, dx) voxels, as everywhere in the package.  A case's ``kind`` is the entry
point it goes through:

* ``step``      -- ``bsi_field_forward`` and ``bsi_field_adjoint``: the dense field, and dL/dphi for a voxel gradient (one
  registration iteration with the program's own optimiser)
* ``field``     -- ``bsi_field_forward`` alone (the final transformation, written as FP32 or BF16)
* ``batch``     -- ``bsi_field_forward_batched`` + ``bsi_field_adjoint_batched`` over uneven volumes
* ``resample``  -- ``bsi_resample_forward`` and ``bsi_resample_backward``: a floating image warped by the field, and dL/dphi
* ``rational``  -- ``bsi_field_forward_rational`` and ``bsi_field_adjoint_rational``: a step on a grid of non-integer
  spacing, shifted against the voxels
* ``scalar``    -- ``bsi_scalar_forward``: cubic B-spline zoom of an image
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2004_05962_gb300 as bsi

DEV = "cuda"


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # a 64^3 volume or region of interest: the launches and the host path decide
        {"name": "step_64", "kind": "step", "shape": "64x64x64", "spacing": "5x5x5", "phi": "uniform", "amp": 2.0},
        # the CT-sized volume at the paper's spacing: one iteration of the registration loop
        {"name": "step_ct", "kind": "step", "shape": "300x512x512", "spacing": "5x5x5", "phi": "smooth", "amp": 3.0},
        # the largest volume at the paper's finest spacing
        {"name": "step_512_s3", "kind": "step", "shape": "512x512x512", "spacing": "3x3x3", "phi": "uniform", "amp": 4.0},
        # a cropped MR volume: odd sizes, anisotropic spacing, rows off 16-byte boundaries
        {"name": "step_odd", "kind": "step", "shape": "155x203x317", "spacing": "4x5x7", "phi": "smooth", "amp": 3.0},
        # the coarse level of a multi-resolution registration: wide control cells
        {"name": "step_coarse", "kind": "step", "shape": "256x256x256", "spacing": "12x12x12", "phi": "smooth", "amp": 4.0},
        # the field kept in half the memory for the resampling that follows
        {"name": "field_bf16_ct", "kind": "field", "shape": "300x512x512", "spacing": "5x5x5", "phi": "smooth", "amp": 3.0,
         "dtype": "bf16"},
        # 64 registrations of uneven volumes and spacings advanced together
        {"name": "batch_64", "kind": "batch", "n": 64, "geom_seed": 5, "amp": 3.0},
        # warping the floating image and the gradient of the similarity, field never stored
        {"name": "resample_ct", "kind": "resample", "shape": "300x512x512", "spacing": "5x5x5", "fshape": "300x512x512",
         "amp": 3.0, "image_seed": 6},
        # the same on an MR-sized volume
        {"name": "resample_mr", "kind": "resample", "shape": "160x192x192", "spacing": "5x5x5", "fshape": "160x192x192",
         "amp": 2.0, "image_seed": 4},
        # a grid laid out in millimetres on a CT: 4.7 voxels, shifted
        {"name": "rational_ct", "kind": "rational", "shape": "300x512x512", "num": "47x47x47", "den": "10x10x10",
         "off": "3x0x9", "amp": 3.0},
        # the same on an odd volume with a fine, anisotropic grid
        {"name": "rational_odd", "kind": "rational", "shape": "101x203x317", "num": "5x33x33", "den": "2x10x10",
         "off": "1x0x7", "amp": 3.0},
        # an image zoomed four times per axis to the CT's size
        {"name": "zoom_4x", "kind": "scalar", "shape": "300x512x512", "spacing": "4x4x4"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text(values):
    return "x".join(str(v) for v in values)


def _ints(text):
    """The (z, y, x) integers of a case's size, spacing or shift."""
    return tuple(int(v) for v in text.split("x"))


def _shape(rng, lo, hi, most):
    """A volume of edges lo..hi (in the logarithm), odd ones among them, of at most ``most`` voxels."""
    while True:
        s = [_log_int(rng, lo, hi) for _ in range(3)]
        if rng.random() < 0.5:   # half the volumes have rows of a multiple of four voxels, as scanners give them
            s[2] = max(4, s[2] // 4 * 4)
        if s[0] * s[1] * s[2] <= most:
            return s


def draw(rng):
    kind = rng.choice(["step", "step", "coarse", "field", "batch", "resample", "rational", "scalar"])
    phi = rng.choice(["uniform", "smooth"])
    amp = round(rng.uniform(1.0, 4.0), 3)
    if kind == "step":
        return {"kind": "step", "shape": _text(_shape(rng, 32, 512, 100_000_000)), "spacing": _text(rng.randint(3, 8) for _ in range(3)),
                "phi": phi, "amp": amp}
    if kind == "coarse":
        return {"kind": "step", "shape": _text(_shape(rng, 48, 384, 30_000_000)), "spacing": _text(rng.randint(9, 24) for _ in range(3)),
                "phi": phi, "amp": amp}
    if kind == "field":
        return {"kind": "field", "shape": _text(_shape(rng, 48, 512, 100_000_000)), "spacing": _text(rng.randint(3, 8) for _ in range(3)),
                "phi": phi, "amp": amp, "dtype": rng.choice(["bf16", "bf16", "f32"])}
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(4, 64), "geom_seed": rng.randint(0, 10 ** 6), "amp": amp}
    if kind == "resample":
        shape = _shape(rng, 48, 512, 60_000_000)
        fshape = list(shape) if rng.random() < 0.5 else [max(16, int(s * rng.uniform(0.8, 1.1))) for s in shape]
        return {"kind": "resample", "shape": _text(shape), "spacing": _text(rng.randint(3, 8) for _ in range(3)), "fshape": _text(fshape),
                "amp": round(rng.uniform(0.5, 3.0), 3), "image_seed": rng.randint(0, 10 ** 6)}
    if kind == "rational":
        den = [rng.randint(1, 10) for _ in range(3)]
        num = [max(d, int(round(d * rng.uniform(2.5, 8.0)))) for d in den]
        return {"kind": "rational", "shape": _text(_shape(rng, 48, 512, 60_000_000)), "num": _text(num), "den": _text(den),
                "off": _text(rng.randint(0, n - 1) for n in num), "amp": amp}
    f = rng.randint(2, 8)
    return {"kind": "scalar", "shape": _text(_shape(rng, 64, 512, 100_000_000)), "spacing": _text([f, f, f])}


# ---------------------------------------------------------------- inputs

def _parse(case):
    """The case with its sizes as tuples of integers."""
    return {k: _ints(v) if k in ("shape", "spacing", "fshape", "num", "den", "off") else v for k, v in case.items()}


def _grid(case):
    if case["kind"] == "rational":
        return tuple(((n_vox - 1) * d + o) // n + 4
                     for n_vox, n, d, o in zip(case["shape"], case["num"], case["den"], case["off"]))
    return tuple(-(-n_vox // d) + 3 for n_vox, d in zip(case["shape"], case["spacing"]))


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform_phi(grid, amp, g):
    return (torch.rand(grid + (3,), generator=g, device=DEV, dtype=torch.float64) * 2 - 1).mul_(amp).float()


def _smooth_phi(grid, amp, g, cells=2.0):
    """Smooth random displacements: white noise blurred by a Gaussian of ``cells`` control cells, standard deviation amp."""
    a = torch.randn(grid + (3,), generator=g, device=DEV, dtype=torch.float64)
    for axis in range(3):
        i = torch.arange(grid[axis], device=DEV, dtype=torch.float64)
        k = torch.exp(-((i[:, None] - i[None, :]) ** 2) / (2 * cells * cells))
        a = torch.tensordot(k / k.sum(1, keepdim=True), a, dims=([1], [axis])).movedim(0, axis)
    return (a * (amp / a.std(dim=(0, 1, 2), keepdim=True))).float().contiguous()


def _phi(case, g):
    f = _uniform_phi if case.get("phi") == "uniform" else _smooth_phi
    return f(_grid(case), case["amp"], g)


def _image(shape, seed, nblobs=8):
    """A smooth image: Gaussian blobs 8 to 20 voxels wide."""
    rng = np.random.default_rng(seed)
    img = torch.zeros(tuple(shape), device=DEV, dtype=torch.float32)
    for _ in range(nblobs):
        c, s, a = rng.uniform([0, 0, 0], shape), rng.uniform(8.0, 20.0), rng.uniform(0.5, 1.0)
        e = [torch.exp(-((torch.arange(n, device=DEV, dtype=torch.float64) - float(m)) ** 2) / (2 * float(s) ** 2)).float()
             for n, m in zip(shape, c)]
        img += float(a) * (e[0][:, None, None] * (e[1][:, None] * e[2][None, :]))
    return img


def _batch_geometries(case):
    rng = np.random.default_rng(case["geom_seed"])
    shapes, spacings = [], []
    for _ in range(case["n"]):
        x, y = int(rng.integers(48, 257)), int(rng.integers(48, 257))
        z = int(rng.integers(48, 161))
        d = rng.integers(3, 9, size=3)
        shapes.append((z, y, x))
        spacings.append((int(d[2]), int(d[1]), int(d[0])))
    return shapes, spacings


def _scalar_coeff(case, g):
    """An image of CT numbers, scaled to 0..1, as B-spline coefficients."""
    return torch.rand(_grid(case), generator=g, device=DEV, dtype=torch.float64).float()


def _arena(shapes, dtype=torch.float32):
    """One zeroed buffer and a view of each shape into it, every view on a 256-byte boundary."""
    off = [0]
    for s in shapes:
        off.append(off[-1] + -(-math.prod(s) // 64) * 64)
    flat = torch.zeros(off[-1], device=DEV, dtype=dtype)
    return flat, [flat[o:o + math.prod(s)].view(s) for o, s in zip(off, shapes)]


def prepare(case, seed):
    case = _parse(case)
    g = _gen(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "batch":
        shapes, spacings = _batch_geometries(case)
        grids = [tuple(-(-n // d) + 3 for n, d in zip(s, p)) for s, p in zip(shapes, spacings)]
        st.update(shapes=shapes, spacings=spacings, phis=[_uniform_phi(gr, case["amp"], g) for gr in grids],
                  grads=[torch.randn(s + (3,), generator=g, device=DEV) for s in shapes])
        # the fields, and the gradients, of all volumes in one buffer each
        st["fields"], st["outs"] = _arena([s + (3,) for s in shapes])
        st["dphis"], st["douts"] = _arena([gr + (3,) for gr in grids])
        return st
    shape = case["shape"]
    st["shape"] = shape
    if kind == "scalar":
        st["coeff"] = _scalar_coeff(case, g)
        return st
    st["phi"] = _phi(case, g)
    if kind in ("step", "rational"):
        st["grad"] = torch.randn(shape + (3,), generator=g, device=DEV)
    if kind == "resample":
        st["image"] = _image(case["fshape"], (case["image_seed"], seed))
        st["grad"] = torch.randn(shape, generator=g, device=DEV)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        u = bsi.bsi_field_forward(st["phi"], st["shape"], case["spacing"])
        return u, bsi.bsi_field_adjoint(st["grad"], case["spacing"])
    if kind == "rational":
        u = bsi.bsi_field_forward_rational(st["phi"], st["shape"], case["num"], case["den"], case["off"])
        return u, bsi.bsi_field_adjoint_rational(st["grad"], case["num"], case["den"], case["off"])
    if kind == "resample":
        w = bsi.bsi_resample_forward(st["phi"], st["shape"], case["spacing"], st["image"])
        return w, bsi.bsi_resample_backward(st["phi"], st["shape"], case["spacing"], st["image"], st["grad"])
    if kind == "field":
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        return bsi.bsi_field_forward(st["phi"], st["shape"], case["spacing"], out_dtype=dt)
    if kind == "scalar":
        return bsi.bsi_scalar_forward(st["coeff"], st["shape"], case["spacing"])
    bsi.bsi_field_forward_batched(st["phis"], st["shapes"], st["spacings"], outs=st["outs"])
    bsi.bsi_field_adjoint_batched(st["grads"], st["spacings"], outs=st["douts"])
    return st["fields"], st["dphis"]


# ---------------------------------------------------------------- bytes and operations

def _field_flops(shape, spacing, c=3):
    """The separable contraction: 4 taps per axis, z and y stages shared along a cell's rows."""
    v = math.prod(shape)
    return 2 * 4 * c * v * (1 + 1 / spacing[2] + 1 / (spacing[2] * spacing[1]))


def work(case):
    case = _parse(case)
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        for s, p in zip(*_batch_geometries(case)):
            pts = math.prod(-(-n // d) + 3 for n, d in zip(s, p))
            b += 24 * (math.prod(s) + pts)
            f += 2 * _field_flops(s, p)
        return {"bytes": b, "flops": f}
    v, pts = math.prod(case["shape"]), math.prod(_grid(case))
    if kind == "scalar":
        return {"bytes": 4 * (v + pts), "flops": _field_flops(case["shape"], case["spacing"], 1)}
    spacing = [n / d for n, d in zip(case["num"], case["den"])] if kind == "rational" else case["spacing"]
    f = _field_flops(case["shape"], spacing)
    if kind == "field":
        return {"bytes": v * (6 if case["dtype"] == "bf16" else 12) + 12 * pts, "flops": f}
    if kind == "resample":
        # image, dL/dwarped and grid read once, warped image and dL/dphi written once; the field, 7 lerps, their gradient
        return {"bytes": 4 * math.prod(case["fshape"]) + 8 * v + 24 * pts, "flops": 2 * f + 50 * v}
    return {"bytes": 24 * v + 24 * pts, "flops": 2 * f}


# ---------------------------------------------------------------- 64-bit results

def _axis(n_vox, num, den, off, n_pts):
    """The [n_vox, n_pts] matrix of one axis: the four cubic B-spline weights of every voxel."""
    q = torch.arange(n_vox, device=DEV, dtype=torch.int64) * den + off
    f = torch.div(q, num, rounding_mode="floor")
    u = (q - f * num).double() / num
    w = torch.stack([(1 - u) ** 3, 3 * u ** 3 - 6 * u ** 2 + 4, -3 * u ** 3 + 3 * u ** 2 + 3 * u + 1, u ** 3], 1) / 6
    m = torch.zeros(n_vox, n_pts, device=DEV, dtype=torch.float64)
    return m.scatter_(1, f[:, None] + torch.arange(4, device=DEV)[None, :], w)


def _axes(shape, grid, spacing=None, case=None):
    if case is not None and case["kind"] == "rational":
        return [_axis(s, n, d, o, p) for s, n, d, o, p in zip(shape, case["num"], case["den"], case["off"], grid)]
    return [_axis(s, d, 1, 0, p) for s, d, p in zip(shape, spacing, grid)]


def _contract(t, mats):
    """t[z, y, x, c] with each axis multiplied by its matrix (rows: the new axis)."""
    c = t.shape[3]
    t = torch.matmul(mats[0], t.reshape(t.shape[0], -1)).reshape(mats[0].shape[0], t.shape[1], t.shape[2], c)
    t = torch.matmul(mats[1], t.reshape(t.shape[0], t.shape[1], -1)).reshape(t.shape[0], mats[1].shape[0], t.shape[2], c)
    return _along_x(t, mats[2])


def _along_x(t, m):
    """t[z, y, x, c] with its x axis multiplied by m (rows: the new axis), as one matrix product."""
    r = t.transpose(2, 3).reshape(-1, t.shape[2]) @ m.t()
    return r.reshape(t.shape[0], t.shape[1], t.shape[3], -1).transpose(2, 3).contiguous()


def _field64(phi, mats):
    return _contract(phi.detach().double(), mats)


def _adjoint64(grad, mats):
    # x first: the largest reduction, a slab of planes at a time (no full 64-bit copy of the gradient)
    t = torch.cat([_along_x(grad[z:z + 32].double(), mats[2].t()) for z in range(0, grad.shape[0], 32)])
    t = torch.matmul(mats[1].t(), t.reshape(t.shape[0], t.shape[1], -1)).reshape(t.shape[0], -1, t.shape[2], 3)
    return torch.matmul(mats[0].t(), t.reshape(t.shape[0], -1)).reshape(-1, t.shape[1], t.shape[2], 3)


def _sample64(image, t, z0, grad_warped):
    """The trilinear interpolant (zeros outside) at x + T(x) for a slab of planes from z0, and dL/dwarped times its gradient."""
    nz, ny, nx = t.shape[:3]
    base = [torch.arange(n, device=DEV, dtype=torch.float64) for n in (nz, ny, nx)]
    pos = [t[..., 2] + (base[0] + z0)[:, None, None], t[..., 1] + base[1][None, :, None], t[..., 0] + base[2][None, None, :]]
    cell = [torch.floor(p) for p in pos]
    fr = [p - c for p, c in zip(pos, cell)]
    lim = image.shape
    flat = image.reshape(-1).double()
    val = torch.zeros_like(pos[0])
    grads = [torch.zeros_like(val) for _ in range(3)]
    for k in range(8):
        bit = ((k >> 2) & 1, (k >> 1) & 1, k & 1)
        idx = [c.long() + b for c, b in zip(cell, bit)]
        ok = torch.ones_like(val, dtype=torch.bool)
        for i, n in zip(idx, lim):
            ok &= (i >= 0) & (i < n)
        lin = (idx[0].clamp(0, lim[0] - 1) * lim[1] + idx[1].clamp(0, lim[1] - 1)) * lim[2] + idx[2].clamp(0, lim[2] - 1)
        f = torch.where(ok, flat[lin], torch.zeros((), device=DEV, dtype=torch.float64))
        w = [r if b else 1 - r for r, b in zip(fr, bit)]
        s = [1.0 if b else -1.0 for b in bit]
        val += w[0] * w[1] * w[2] * f
        grads[0] += w[0] * w[1] * s[2] * f   # d/dx
        grads[1] += w[0] * s[1] * w[2] * f   # d/dy
        grads[2] += s[0] * w[1] * w[2] * f   # d/dz
    return val, torch.stack(grads, -1) * grad_warped.double()[..., None]


def exact(case, seed):
    st = prepare(case, seed)
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        fields, us = _arena([u.shape for u in st["outs"]], torch.float64)
        dphis, ds = _arena([d.shape for d in st["douts"]], torch.float64)
        for s, p, phi, g, u, d in zip(st["shapes"], st["spacings"], st["phis"], st["grads"], us, ds):
            m = _axes(s, phi.shape[:3], p)
            u.copy_(_field64(phi, m))
            d.copy_(_adjoint64(g, m))
        return fields, dphis
    shape, grid = st["shape"], _grid(case)
    m = _axes(shape, grid, case.get("spacing"), case)
    if kind == "scalar":
        return _contract(st["coeff"].double()[..., None], m)[..., 0]
    if kind == "field":
        return _field64(st["phi"], m)
    if kind in ("step", "rational"):
        return _field64(st["phi"], m), _adjoint64(st["grad"], m)
    # resample: slabs of z-planes
    phi = st["phi"].detach().double()
    warped, dphi = [], torch.zeros(grid + (3,), device=DEV, dtype=torch.float64)
    step = max(1, 8_000_000 // (shape[1] * shape[2]))
    for z in range(0, shape[0], step):
        mz = [m[0][z:z + step], m[1], m[2]]
        v, g = _sample64(st["image"], _contract(phi, mz), z, st["grad"][z:z + step])
        warped.append(v)
        dphi += _adjoint64(g, mz)
    return torch.cat(warped), dphi
