"""A survey cut into batches of shots (max_batch) against the same call in one
batch, with decimated boundaries: the forward loop then runs past the last
recorded step (to the last stored sample), so a shot's rows in the box tables
are more than nt + 1.

Tolerance: a shot's steps are the same sums in either cut up to their order
(receivers' and shots' sums, the grouping of CPML terms): a few roundings of
2^-24 a step, 4 nt 2^-24 (1.4e-5 for nt = 60) of the norm.
"""
import numpy as np
import pytest
import torch

from paper_2311_02293_gb300 import synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = (x.double().cpu().numpy().ravel() for x in (a, b))
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("kernels", ["auto", "generic"])
@pytest.mark.parametrize("ndim,order,dr", [(2, 8, 3), (2, 4, 2), (3, 8, 3), (3, 4, 2)])
def test_decimated_boundaries_in_several_batches(ndim, order, dr, kernels):
    from paper_2311_02293_gb300 import smi
    if ndim == 2:
        w = synth.tiny_2d(nz=60, nx=200, nt=60, order=order, nb=8, src=(5, 20))
    else:
        w = synth.tiny_3d(nz=40, nx=90, ny=30, nt=40, order=order, nb=8)
    nshot, h, nx = 4, w.d[0], w.n[1]
    srcs = np.repeat(w.srcs, nshot, 0)
    srcs[:, 1] = np.round(np.linspace(10, nx - 11, nshot)) * h     # boxes of the shots lie apart at first
    recs = [w.recs[0][k:] for k in range(nshot)]
    dev = torch.device("cuda:0")
    vp, rho, stf = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho, w.stf))
    out = {}
    for cut in (0, 3, 1):
        prob = smi.Problem(w.d, w.nt, w.dt, w.fm, order=order, nb=8, dr=dr, max_batch=cut, kernels=kernels)
        u = smi.smi_forward(vp, rho, prob, srcs, recs, stf, flat=True)
        if cut == 0:
            d = (0.7 * u).contiguous()
        J, g = smi.smi_fwi_gradient(vp, rho, prob, srcs, recs, stf, d)
        img = smi.smi_rtm(vp, rho, prob, srcs, recs, stf, d)
        out[cut] = (u, g, img, torch.as_tensor(J).reshape(-1))
    tol = 4 * w.nt * 2.0 ** -24
    for cut in (3, 1):
        for a, b in zip(out[cut], out[0]):
            assert rel(a, b) <= tol


def test_tape_of_more_shots_than_half_a_grid_dimension():
    """33000 small 2D shots in one batch: the adjoint and the reconstruction
    no longer share a launch along gridDim.z.  Only three shots have an
    adjoint source, so the gradient is that of the three alone."""
    from paper_2311_02293_gb300 import smi
    nshot, n, nt, h = 33000, 9, 30, 10.0
    some = [0, 32767, nshot - 1]
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(3)
    vp = 1800.0 + 600.0 * torch.rand((n, n), generator=gen, device=dev)
    rho = torch.full((n, n), 1500.0, device=dev)
    stf = torch.ones(nt, device=dev)
    srcs = np.stack([3.0 + np.arange(nshot) % 3, 4.0 + np.arange(nshot) % 2, np.zeros(nshot)], 1) * h
    recs = [np.array([[5.0, 2.0 + s % 5, 0.0]]) * h for s in range(nshot)]
    prob = smi.Problem((h, h), nt, 1e-3, 0.0, order=4, nb=2)
    u, tape = smi.smi_forward_tape(vp, rho, prob, srcs, recs, stf)
    adj = torch.zeros_like(u).reshape(nshot, nt)
    adj[some] = u.reshape(nshot, nt)[some]
    g = tape.vjp(adj.reshape(-1))
    tape.free()
    alone = smi.smi_forward_vjp(vp, rho, prob, srcs[some], [recs[s] for s in some], stf, adj[some].reshape(-1).contiguous())
    assert float(alone.abs().max()) > 0
    assert rel(g, alone) <= 4 * nt * 2.0 ** -24


@pytest.mark.parametrize("order,nb,nx", [(8, 8, 150), (4, 6, 141), (8, 10, 170)])
def test_3d_shots_are_the_same_bits_alone(order, nb, nx):
    """Two shots far apart in x, whose boxes start at different nodes: their
    seismograms in one batch and one after the other."""
    from paper_2311_02293_gb300 import smi
    w = synth.tiny_3d(nz=40, nx=nx, ny=34, nt=60, order=order, nb=nb)
    h = w.d[0]
    srcs = np.repeat(w.srcs, 2, 0)
    srcs[:, 1] = [3 * h, (nx - 4) * h]
    recs = [w.recs[0], w.recs[0]]
    dev = torch.device("cuda:0")
    vp, rho, stf = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho, w.stf))
    u = [smi.smi_forward(vp, rho, smi.Problem(w.d, w.nt, w.dt, w.fm, order=order, nb=nb, max_batch=k), srcs, recs, stf,
                         flat=True) for k in (0, 1)]
    assert float(u[0].abs().max()) > 0 and torch.equal(u[0], u[1])
