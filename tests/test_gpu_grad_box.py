"""The gradient outside the computing box of the source: the forward steps
update no pressure there, so the discrete gradient is exactly zero, also on
the nodes that share a tile with the box.  The source is strong, so that the
field at the edge of the box does not underflow to zero by itself."""
import numpy as np
import pytest
import torch

from paper_2311_02293_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("dr", [1, 2])
def test_gradient_is_zero_outside_the_box(ndim, order, dr):
    from paper_2311_02293_gb300 import smi
    h, nb = 10.0, 8
    if ndim == 2:
        w = synth.tiny_2d(nz=120, nx=150, nt=24, order=order, nb=nb, src=(60, 70), rec_z=58)
    else:
        w = synth.tiny_3d(nz=80, nx=70, ny=70, nt=24, order=order, nb=nb)
        w.srcs[:] = [400.0, 350.0, 350.0]
        z = np.arange(2, 78)              # a well: the residual's field reaches the box's edges along z at once
        w.recs = [np.stack([z * h, np.full(z.size, 320.0), np.full(z.size, 350.0)], 1)]
    dev = torch.device("cuda:0")
    vp, rho = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho))
    stf = torch.full((w.nt,), 1e12, device=dev)
    prob = smi.Problem(w.d, w.nt, w.dt, w.fm, order=order, nb=nb, dr=dr)
    u = smi.smi_forward(vp, rho, prob, w.srcs, w.recs, stf, flat=True)
    _, g = smi.smi_fwi_gradient(vp, rho, prob, w.srcs, w.recs, stf, (0.3 * u).contiguous())
    lo, hi = smi.smi_box_table(vp, rho, prob, w.srcs, w.recs, stf, 0, "source", w.nt - 1, 1)
    lo, hi = (np.asarray(b).ravel()[:ndim] - nb for b in (lo, hi))
    g = g.cpu().numpy()
    outside = np.ones(g.shape, bool)
    outside[tuple(slice(max(0, int(lo[a])), int(hi[a]) + 1) for a in reversed(range(ndim)))] = False
    assert outside.sum() > g.size // 4 and np.abs(g[~outside]).max() > 0
    assert np.count_nonzero(g[outside]) == 0
