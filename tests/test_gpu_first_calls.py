"""The library's first calls from several threads at once (a server's slots):
every thread runs the tile kernels, also while another one is still looking up
the tensor-map encoder.  In a child process, where no call has been made."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import threading
import torch
from paper_2311_02293_gb300 import smi, synth
w = synth.tiny_2d(nz=60, nx=70, nt=50, order=8, nb=8)
dev = torch.device("cuda:0")
vp, rho, stf = (torch.from_numpy(a).to(dev) for a in (w.vp, w.rho, w.stf))
torch.cuda.synchronize()
n, launches, start = 8, [0] * 8, threading.Barrier(8)

def call(k):
    st = torch.cuda.Stream()
    start.wait()
    smi.smi_forward(vp, rho, smi.Problem(w.d, w.nt, w.dt, w.fm, order=8, nb=8), w.srcs, w.recs, stf,
                    stream=st.cuda_stream)
    launches[k] = smi.smi_last_stats()["kernel_launches"]

t = [threading.Thread(target=call, args=(k,)) for k in range(n)]
[x.start() for x in t]
[x.join() for x in t]
assert min(launches) == max(launches) < 2 * w.nt, launches     # one launch a step; the generic kernels take four
"""


def test_first_calls_from_several_threads():
    for _ in range(2):
        r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
