"""The single-launch 2D steps against the generic kernels (the same scheme in
two passes, node by node) at sizes around the edges of their 32 x 16 and
32 x 32 tiles, on thin models where both CPML slabs meet one tile, and with
every option that takes another branch.

Tolerance: both sides compute the same FP32 sums in another order.  A step
adds a few roundings of 2^-24 to every value, so after nt steps the relative
difference stays below about 4 nt 2^-24 (3.1e-5 for nt = 130): 5e-5 for the
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


# nz, nx, order, nb, off-grid, options
CASES = [
    (8, 9, 8, 4, False, {}),                       # smallest grid: one tile holds every slab
    (4, 5, 4, 2, False, {}),
    (19, 20, 4, 6, True, {}),                      # 31 x 32 extended
    (20, 21, 8, 6, False, {"use_box": False}),     # 32 x 33
    (53, 51, 8, 6, True, {"shell_prec": "f16"}),   # 65 x 63
    (40, 37, 4, 7, False, {"dr": 3}),
    (45, 70, 8, 9, True, {"dr": 2, "shell_prec": "bf16"}),
    (33, 50, 8, 8, False, {"freesurf": True}),
    (41, 34, 4, 8, True, {"freesurf": True, "use_box": False}),
    (301, 420, 8, 20, False, {}),                  # many tiles, wide tiles with the four shots below
]


@pytest.mark.parametrize("nz,nx,order,nb,off,opt", CASES)
@pytest.mark.parametrize("nshot", [1, 4])
def test_step2d_equals_generic(nz, nx, order, nb, off, opt, nshot):
    from paper_2311_02293_gb300 import smi
    if off and opt.get("freesurf"):
        sz, rz = 6.37, 5.2
    else:
        sz, rz = (4.37, 3.2) if off else (3.0, 2.0)
    w = synth.tiny_2d(nz=nz, nx=nx, nt=130, order=order, nb=nb, src=(3, nx // 2))
    h = w.d[0]
    fx = 0.41 if off else 0.0
    xs = np.round(np.linspace(2, nx - 3, nshot)) if nshot > 1 else np.array([nx // 2])
    srcs = np.stack([np.full(nshot, min(sz, nz - 2)), xs + fx, np.zeros(nshot)], 1) * h
    xr = np.arange(0, nx - 1, 2) + fx                # receivers reach both x slabs' edges
    rec = np.stack([np.full(xr.size, min(rz, nz - 2)), xr, np.zeros(xr.size)], 1) * h
    recs = [rec[k % 2:] for k in range(nshot)]
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
