"""A 2D line of more than 65535 tile rows (1048560 columns of 16-wide tiles):
a step takes more than one launch.  Against the generic kernels, with the
source and the receivers around the rows where the launches meet and at the
far end; tolerances as for the other sizes (4 nt 2^-24 for the seismograms,
four times that for sums of products)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = (x.double().cpu().numpy().ravel() for x in (a, b))
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("use_box", [True, False])
def test_line_of_many_columns(use_box):
    from paper_2311_02293_gb300 import smi
    nz, nx, nb, nt, h, dt = 9, 65535 * 16 + 40, 2, 40, 10.0, 1e-3
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(5)
    vp = 1800.0 + 600.0 * torch.rand((nx, nz), generator=gen, device=dev)
    rho = 1500.0 + 500.0 * torch.rand((nx, nz), generator=gen, device=dev)
    stf = torch.ones(nt, device=dev)
    xs = np.array([65535.0 * 16 - 6, nx - 12.0, 30.0])
    srcs = np.stack([np.full(3, 3.0), xs, np.zeros(3)], 1) * h
    recs = []
    for x in xs:
        r = x + np.arange(-8, 9)
        recs.append(np.stack([np.full(r.size, 4.0), r, np.zeros(r.size)], 1) * h)
    out = {}
    for kernels in ("auto", "generic"):
        prob = smi.Problem((h, h), nt, dt, 0.0, order=4, nb=nb, use_box=use_box, kernels=kernels)
        u = smi.smi_forward(vp, rho, prob, srcs, recs, stf, flat=True)
        if kernels == "auto":
            d = (0.4 * u).contiguous()
        _, g = smi.smi_fwi_gradient(vp, rho, prob, srcs, recs, stf, d)
        out[kernels] = (u, g)
    a, b = out["auto"], out["generic"]
    tol = 4 * nt * 2.0 ** -24
    assert rel(a[0], b[0]) <= tol
    assert rel(a[1], b[1]) <= 4 * tol
    for part in (slice(0, 100), slice(65535 * 16 - 60, 65535 * 16 + 30), slice(nx - 60, nx)):
        assert rel(a[1][part], b[1][part]) <= 4 * tol
