"""Set-up time of smi_forward_noalloc with many receivers between nodes: like
smi_forward it evaluates the weights of a coordinate once, however many
receivers share it (19600 receivers, host time: 4.7 ms a call; with every
receiver by itself 120 ms)."""
import time

import numpy as np
import pytest
import torch

from paper_2311_02293_gb300 import synth

pytestmark = pytest.mark.gpu


def test_set_up_of_a_receiver_carpet():
    from paper_2311_02293_gb300 import smi
    w = synth.tiny_3d(nz=24, nx=60, ny=60, nt=2, order=8, nb=6)
    h = w.d[0]
    ix, iy = np.meshgrid(5.0 + 0.35 * np.arange(140), 5.0 + 0.35 * np.arange(140))
    rec = np.stack([np.full(ix.size, 3.4), ix.ravel() + 0.07, iy.ravel() + 0.07], 1) * h
    dev = torch.device("cuda:0")
    vp, rho, stf = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho, w.stf))
    prob = smi.Problem(w.d, w.nt, w.dt, w.fm, order=8, nb=6)
    out = torch.empty(w.nt * len(rec), device=dev)

    def best(fn):
        t = []
        for _ in range(4):
            t0 = time.perf_counter()
            fn()
            t.append(time.perf_counter() - t0)
        return min(t)

    u = smi.smi_forward(vp, rho, prob, w.srcs, [rec], stf, flat=True)
    plain = best(lambda: smi.smi_forward(vp, rho, prob, w.srcs, [rec], stf, flat=True))
    noalloc = best(lambda: smi.smi_forward_noalloc(vp, rho, prob, w.srcs, [rec], stf, out=out))
    assert torch.linalg.norm((out - u).double()) <= 4 * w.nt * 2.0 ** -24 * torch.linalg.norm(u.double())
    print(f"noalloc {1e3 * noalloc:.1f} ms, smi_forward {1e3 * plain:.1f} ms")
    assert noalloc <= 4 * plain + 0.05
