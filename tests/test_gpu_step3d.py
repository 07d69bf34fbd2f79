"""The two-pass 3D tile kernels (CPML terms inline, work list drawn by the
CTAs) against the generic kernels at sizes around the edges of their 32 x 16
tiles and slabs, on thin models where both CPML slabs meet one tile, and with
every option that takes another branch.

Tolerance: both sides compute the same FP32 sums in another order.  A step
adds a few roundings of 2^-24 to every value, so after nt steps the relative
difference stays below about 4 nt 2^-24 (1.7e-5 for nt = 70): 5e-5 for the
seismograms, 2e-4 for products of two fields summed over the steps.
"""
import numpy as np
import pytest
import torch

from paper_2311_02293_gb300 import synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = (x.double().cpu().numpy().ravel() for x in (a, b))
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# nz, nx, ny, order, nb, off-grid, options
CASES = [
    (8, 9, 8, 8, 4, False, {}),                        # smallest grid: a window meets both slabs
    (4, 5, 6, 4, 2, False, {}),
    (20, 20, 21, 8, 6, False, {"use_box": False}),     # 32 x 32 x 33 extended
    (53, 37, 30, 4, 6, True, {"shell_prec": "f16"}),   # 65 x 49 x 42
    (61, 62, 19, 8, 4, False, {"dr": 3}),              # two slabs an axis, one each a tile
    (70, 40, 25, 8, 9, True, {"dr": 2, "shell_prec": "bf16"}),
    (33, 30, 28, 8, 8, False, {"freesurf": True}),
    (28, 40, 20, 8, 6, True, {}),                      # the physical box needs one row of tiles, not two
    (41, 64, 22, 4, 5, True, {"freesurf": True, "use_box": False}),
]


@pytest.mark.parametrize("nz,nx,ny,order,nb,off,opt", CASES)
@pytest.mark.parametrize("nshot", [1, 2])
def test_step3d_equals_generic(nz, nx, ny, order, nb, off, opt, nshot):
    from paper_2311_02293_gb300 import smi
    w = synth.tiny_3d(nz=nz, nx=nx, ny=ny, nt=70, order=order, nb=nb)
    h = w.d[0]
    fx = 0.41 if off else 0.0
    sz, rz = (5.37, 4.6) if off else (min(3.0, nz - 2), min(2.0, nz - 2))
    sx = np.round(np.linspace(1, nx - 3, nshot + 2))[1:-1]
    srcs = np.stack([np.full(nshot, sz), sx + fx, np.full(nshot, ny // 2 + fx)], 1) * h
    ix, iy = np.meshgrid(np.arange(0, nx - 1, 2) + fx, np.arange(0, ny - 1, 3) + fx, indexing="xy")
    rec = np.stack([np.full(ix.size, rz), ix.ravel(), iy.ravel()], 1) * h     # reaches the slabs' edges
    recs = [rec[k:] for k in range(nshot)]
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
        out[kernels] = (u, g, img, La, g1, J)
    a, b = out["auto"], out["generic"]
    tol = {"f16": 3e-3, "bf16": 3e-2}.get(opt.get("shell_prec"), 2e-4)   # 16-bit stores round other values
    assert rel(a[0], b[0]) <= 5e-5
    assert rel(a[3], b[3]) <= 5e-5
    assert abs(float(a[5][0]) - float(b[5][0])) <= 1e-4 * float(b[5][0])
    for k in (1, 2, 4):
        assert rel(a[k], b[k]) <= tol
