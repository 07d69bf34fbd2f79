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


@pytest.mark.parametrize("ndim", [2, 3])
def test_tape_that_fits_only_without_the_tile_kernels_state(ndim):
    """A tape needs all its shots at once.  The tile kernels' state is larger
    than the generic kernels' (2D: two copies); where only the smaller one fits,
    the tape runs the generic kernels.  Against the same shots in batches."""
    from paper_2311_02293_gb300 import smi
    dev = torch.device("cuda:0")
    if ndim == 2:
        w = synth.tiny_2d(nz=400, nx=500, nt=20, order=8, nb=20, src=(10, 250))
        nshot = 300
    else:
        w = synth.tiny_3d(nz=60, nx=60, ny=60, nt=8, order=8, nb=20)
        nshot = 220
    srcs = np.repeat(w.srcs, nshot, 0)
    srcs[:, 1] += 10.0 * (np.arange(nshot) % 20)
    recs = [w.recs[0]] * nshot
    vp, rho, stf = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho, w.stf))
    P = lambda **kw: smi.Problem(w.d, w.nt, w.dt, w.fm, order=8, nb=20, **kw)
    u = smi.smi_forward(vp, rho, P(max_batch=20), srcs, recs, stf, flat=True)
    ref = smi.smi_forward_vjp(vp, rho, P(max_batch=20), srcs, recs, stf, u)
    need = [smi.smi_footprint(vp, rho, P(kernels=k), srcs, recs, stf, kind="gradient") for k in ("auto", "generic")]
    assert need[0] > 1.02 * need[1]
    smi.smi_release_memory()
    torch.cuda.synchronize()
    # 80 % of what is left free lies between the two
    filler = torch.empty(torch.cuda.mem_get_info()[0] - int(0.5 * (need[0] + need[1]) / 0.8), dtype=torch.uint8, device=dev)
    v, tape = smi.smi_forward_tape(vp, rho, P(), srcs, recs, stf)
    g = tape.vjp(u)
    tape.free()
    del filler
    torch.cuda.empty_cache()
    tol = 4 * w.nt * 2.0 ** -24
    assert torch.linalg.norm((v - u).double()) <= tol * torch.linalg.norm(u.double())
    # the shots' sum adds a rounding a shot
    assert torch.linalg.norm((g - ref).double()) <= (4 * tol + nshot * 2.0 ** -24) * torch.linalg.norm(ref.double())
