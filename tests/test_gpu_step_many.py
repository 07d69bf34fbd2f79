"""The variants of the tile kernels that large surveys run, and the free
surface with 16-bit boundaries, against the generic kernels.

- 2D launches of 1200 tiles (32 x 32, all shots) and more take 32-wide reverse
  tiles and another register budget: many shots on small ragged grids, at
  sizes around the edges of a tile.
- With a free surface the largest band magnitudes (16-bit storage) are found
  after the mirror, by another kernel in 3D than without.

Tolerance: both sides compute the same FP32 sums in another order, a few
roundings of 2^-24 a step (4 nt 2^-24 = 1.9e-5 for nt = 80): 5e-5 for the
seismograms, 2e-4 for products of two fields summed over the steps.  16-bit
stores round values that differ in their last bits to other neighbours: 2^-11
(FP16) and 2^-8 (BF16) of a step's largest magnitude on the values of one
band, 3e-3 and 3e-2 of the norm of the sums.
"""
import numpy as np
import pytest
import torch

from paper_2311_02293_gb300 import synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = (x.double().cpu().numpy().ravel() for x in (a, b))
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _compare(w, srcs, recs, order, nb, opt):
    from paper_2311_02293_gb300 import smi
    dev = torch.device("cuda:0")
    vp, rho, stf = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho, w.stf))
    rng = np.random.default_rng(5)
    out = {}
    for kernels in ("auto", "generic"):
        prob = smi.Problem(w.d, w.nt, w.dt, w.fm, order=order, nb=nb, kernels=kernels, **opt)
        u = smi.smi_forward(vp, rho, prob, srcs, recs, stf, flat=True)
        if kernels == "auto":
            d = u * torch.from_numpy(rng.uniform(0.2, 1.8, u.numel()).astype(np.float32)).to(dev)
        J, g = smi.smi_fwi_gradient(vp, rho, prob, srcs, recs, stf, d)
        img = smi.smi_rtm(vp, rho, prob, srcs, recs, stf, d)
        La = smi.smi_forward_adjoint(vp, rho, prob, srcs, recs, stf, d)
        g1 = smi.smi_fwi_gradient_family(vp, rho, prob, srcs, recs, stf, d, family=1)[2]
        norm = smi.Problem(w.d, w.nt, w.dt, w.fm, order=order, nb=nb, kernels=kernels, img_norm=True, **opt)
        out[kernels] = (u, La, g, img, g1, smi.smi_rtm(vp, rho, norm, srcs, recs, stf, d), J)
    a, b = out["auto"], out["generic"]
    tol = {"f16": 3e-3, "bf16": 3e-2}.get(opt.get("shell_prec"), 2e-4)
    assert abs(float(a[6][0]) - float(b[6][0])) <= 1e-4 * float(b[6][0])
    for k in range(6):
        assert rel(a[k], b[k]) <= (5e-5 if k < 2 else tol), k


def _line(nz, nx, nt, order, nb, off, nshot, freesurf):
    w = synth.tiny_2d(nz=nz, nx=nx, nt=nt, order=order, nb=nb, src=(3, nx // 2))
    h, fx = w.d[0], 0.41 if off else 0.0
    sz, rz = (6.37, 5.2) if off and freesurf else (4.37, 3.2) if off else (3.0, 2.0)
    xs = np.round(np.linspace(2, nx - 3, nshot)) + fx
    srcs = np.stack([np.full(nshot, min(sz, nz - 2)), xs, np.zeros(nshot)], 1) * h
    xr = np.arange(0, nx - 1, 5) + fx
    rec = np.stack([np.full(xr.size, min(rz, nz - 2)), xr, np.zeros(xr.size)], 1) * h
    return w, srcs, [rec[k % 4:] for k in range(nshot)]


# nz, nx, order, nb, off-grid, options (extended sizes beside)
MANY = [
    (53, 83, 8, 6, False, {}),                             # 65 x 95
    (52, 84, 8, 6, True, {"shell_prec": "f16"}),           # 64 x 96
    (51, 85, 4, 6, False, {"use_box": False}),             # 63 x 97
    (40, 81, 4, 7, True, {"dr": 3}),
    (45, 100, 8, 9, False, {"dr": 2, "shell_prec": "bf16"}),
    (33, 90, 8, 8, True, {"freesurf": True}),
    (41, 70, 4, 8, False, {"freesurf": True, "shell_prec": "f16"}),
    (9, 300, 8, 4, True, {}),                              # one row of tiles
]


@pytest.mark.parametrize("nz,nx,order,nb,off,opt", MANY)
def test_2d_steps_of_many_tiles_equal_generic(nz, nx, order, nb, off, opt):
    per_shot = -(-(nz + 2 * nb) // 32) * -(-(nx + 2 * nb) // 32)
    nshot = 1200 // per_shot + 1
    w, srcs, recs = _line(nz, nx, 80, order, nb, off, nshot, opt.get("freesurf", False))
    _compare(w, srcs, recs, order, nb, opt)


@pytest.mark.parametrize("order,prec,dr", [(8, "f16", 1), (4, "bf16", 1), (4, "f16", 2), (8, "bf16", 3)])
@pytest.mark.parametrize("ndim", [2, 3])
def test_free_surface_with_16bit_boundaries(ndim, order, prec, dr):
    opt = {"freesurf": True, "shell_prec": prec, "dr": dr}
    if ndim == 2:
        w, srcs, recs = _line(43, 61, 80, order, 8, True, 2, True)
    else:
        w = synth.tiny_3d(nz=36, nx=41, ny=30, nt=60, order=order, nb=8)
        h = w.d[0]
        srcs = np.array([[6.37, 14.4, 12.6], [5.0, 28.0, 17.0]]) * h
        ix, iy = np.meshgrid(np.arange(0, 40, 3) + 0.41, np.arange(0, 29, 4) + 0.41)
        rec = np.stack([np.full(ix.size, 5.2), ix.ravel(), iy.ravel()], 1) * h
        recs = [rec, rec[1:]]
    _compare(w, srcs, recs, order, 8, opt)
