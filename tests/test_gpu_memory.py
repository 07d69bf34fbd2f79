"""Device memory between calls: what the library keeps mapped goes back with
smi_release_memory, and by itself where the device is short of memory."""
import numpy as np
import pytest
import torch

from paper_2311_02293_gb300 import synth

pytestmark = pytest.mark.gpu


def _gradient(smi, w, dev):
    vp, rho, stf = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho, w.stf))
    prob = smi.Problem(w.d, w.nt, w.dt, w.fm, order=w.order, nb=w.nb)
    d = torch.zeros(w.nt * sum(len(r) for r in w.recs), device=dev)
    J, g = smi.smi_fwi_gradient(vp, rho, prob, w.srcs, w.recs, stf, d)
    return g


def _free():
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_release_memory_gives_everything_back():
    from paper_2311_02293_gb300 import smi
    dev = torch.device("cuda:0")
    w = synth.layered_fault_2d(nz=150, nx=400, nt=400, nshot=8)
    w.srcs[:, 1] = np.linspace(300.0, 4500.0, 8)
    _gradient(smi, w, dev)                   # loads the kernels
    smi.smi_release_memory()
    before = _free()
    _gradient(smi, w, dev)
    smi.smi_release_memory()
    assert _free() == before


def test_nothing_is_kept_on_a_crowded_device():
    from paper_2311_02293_gb300 import smi
    dev = torch.device("cuda:0")
    w = synth.layered_fault_2d(nz=150, nx=400, nt=400, nshot=8)
    w.srcs[:, 1] = np.linspace(300.0, 4500.0, 8)
    _gradient(smi, w, dev)                   # loads the kernels, and may leave memory with the library
    total = torch.cuda.mem_get_info()[1]
    filler = torch.empty(int(0.6 * total), dtype=torch.uint8, device=dev)
    smi.smi_release_memory()
    before = _free()
    _gradient(smi, w, dev)
    assert _free() == before
    del filler
    torch.cuda.empty_cache()
