"""Free surface in 2D while the computing box of a deep source grows into the
rows next to the surface: the image rows above the box take part in the next
step.  The field there is far below the source's (1e-17 to 1e-9 of it), so the
seismograms of receivers next to the surface are compared step by step, each
against the largest of its own step.

Tolerance: both kernel families sum the same FP32 terms in another order, a
few roundings of 2^-24 a step of values of the step's own size: 4 nt 2^-24
(2.1e-5 for nt = 90).
"""
import numpy as np
import pytest
import torch

from paper_2311_02293_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [8, 9, 10, 11])      # the surface row at every place in a quad
@pytest.mark.parametrize("order", [4, 8])
def test_image_rows_above_the_box(order, nb):
    from paper_2311_02293_gb300 import smi
    nt, h = 90, 10.0
    rz, rx = np.meshgrid(np.arange(1, 6), np.arange(20, 40, 3))
    recs = [np.stack([rz.ravel() * h, rx.ravel() * h, 0.0 * rx.ravel()], 1)]
    w = synth.tiny_2d(nz=70, nx=60, nt=nt, order=order, nb=nb, src=(34 if order == 8 else 28, 30))
    dev = torch.device("cuda:0")
    vp, rho = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho))
    stf = torch.ones(nt, device=dev)
    out = {}
    for kernels in ("auto", "generic"):
        prob = smi.Problem(w.d, nt, w.dt, w.fm, order=order, nb=nb, kernels=kernels, freesurf=True)
        out[kernels] = smi.smi_forward(vp, rho, prob, w.srcs, recs, stf, flat=True).double().cpu().numpy().reshape(nt, -1)
    lo, _ = smi.smi_box_table(vp, rho, prob, w.srcs, recs, stf, 0, "source", 0, nt)
    lo = np.asarray(lo).reshape(nt, -1)[:, 0]
    N, L = order // 2, nb
    assert ((lo > L - N) & (lo <= L + N)).sum() >= 8         # the case meets the rows in question
    a, b = out["auto"], out["generic"]
    big = np.abs(b).max(1)
    live = big > 1e-30
    assert np.array_equal(a[big == 0], b[big == 0])
    assert (np.abs(a - b).max(1)[live] / big[live]).max() <= 4 * nt * 2.0 ** -24
