"""Performance cases of the library: what is timed, on which inputs, and the
results those inputs have in 64-bit arithmetic.

A case is one call (or one autograd step) through the public Python entry
points on a seeded synthetic model, with the inputs already on the GPU as an
inversion or migration program holds them.  The sizes are those of this
repository's workloads and serving mix, some with fewer time steps so that a
pass stays below two seconds, and ragged sizes between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_02293_gb300 import autograd, smi, synth

NB = 20                                    # CPML layers, the library's default
FIELDS = dict(ny=1, order=8, shots=1, rec_step=1, h=10.0, dt=8e-4, fm=12.0, prec="f32", dr=1, box=True,
              freesurf=False, off=False, corner=False, per_shot=False, model="smooth", vlo=1600.0, vhi=4000.0)


def _case(**kw):
    return {**FIELDS, **kw}


def listed():
    return [
        # one small 2D shot, the two-layer workload's size: a quick modelling call,
        # where launches and latency count
        _case(name="fwd2d_201", kind="forward", nz=201, nx=201, nt=1000, order=4, dt=1e-3, fm=10.0, vlo=2000.0,
              vhi=3000.0, model="layers"),
        # a marine line: free surface, sources and receivers between nodes (every
        # stencil has all its Kaiser-sinc taps), ragged sizes, a few shots a call
        _case(name="fwd2d_marine", kind="forward", nz=187, nx=429, nt=900, shots=6, rec_step=2, dt=1e-3, fm=10.0,
              freesurf=True, off=True, vlo=1500.0, vhi=3500.0),
        # one request of the serving mix: a single-shot 2D gradient with 16-bit boundaries
        _case(name="grad2d_shot", kind="gradient", nz=257, nx=903, nt=1500, h=12.5, dt=1e-3, fm=8.0, prec="f16",
              vlo=1500.0, vhi=4500.0),
        # the 2D inversion workload: the gradient of a whole 40-shot survey
        _case(name="grad2d_survey", kind="gradient", nz=301, nx=1001, nt=800, shots=40, h=12.5, dt=1e-3, fm=8.0,
              vlo=1500.0, vhi=4500.0),
        # one mini-batch step of a torch inversion: misfit and backward through the tape
        _case(name="step2d_autograd", kind="autograd", nz=201, nx=601, nt=700, shots=8, rec_step=4, order=4,
              dt=1e-3, fm=10.0, vlo=1500.0, vhi=4000.0),
        # a small 3D shot at order 4, ragged: survey design, tests of a setting
        _case(name="fwd3d_small", kind="forward", nz=93, nx=101, ny=87, nt=400, rec_step=2, order=4),
        # the large 3D forward workload: corner source and the growing computing box
        _case(name="fwd3d_corner", kind="forward", nz=200, nx=400, ny=400, nt=900, rec_step=2, corner=True,
              vlo=1500.0),
        # the smallest 3D migration request of the serving mix: order 4, 16-bit boundaries
        _case(name="rtm3d_160", kind="rtm", nz=160, nx=160, ny=160, nt=500, rec_step=2, order=4, prec="f16",
              model="salt", vlo=2000.0, vhi=4500.0),
        # a migration with decimated boundaries, flat ragged grid, the box soon filling it
        _case(name="rtm3d_dr", kind="rtm", nz=131, nx=243, ny=205, nt=450, rec_step=3, dr=8, model="layers",
              vlo=2000.0, vhi=4500.0),
        # the benchmark's 3D salt migration, one shot
        _case(name="rtm3d_salt", kind="rtm", nz=300, nx=300, ny=300, nt=600, rec_step=2, fm=15.0, prec="f16",
              model="salt", vlo=2000.0, vhi=4500.0),
        # multiparameter 3D inversion: the (Vp, Ip) gradient of two shots, box off
        _case(name="family3d", kind="family", nz=90, nx=110, ny=100, nt=300, shots=2, rec_step=4, box=False,
              vhi=3500.0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = dict(order=rng.choice([4, 8]), off=rng.random() < 0.25, freesurf=rng.random() < 0.2, box=rng.random() < 0.85,
             model=rng.choice(["smooth", "layers", "salt"]), vhi=round(rng.uniform(2800.0, 4500.0), 1))
    if rng.random() < 0.5:
        c.update(kind=rng.choice(["forward", "gradient", "gradient", "rtm", "autograd"]), nz=size(81, 401),
                 nx=size(81, 1601), nt=size(250, 1500), shots=size(1, 40), rec_step=rng.randint(1, 4), dt=1e-3,
                 fm=10.0, vlo=1600.0)
    else:
        c.update(kind=rng.choice(["forward", "forward", "rtm", "rtm", "gradient", "family"]), nz=size(61, 300),
                 nx=size(61, 400), ny=size(61, 400), nt=size(120, 700), shots=rng.choice([1, 1, 1, 2]),
                 rec_step=rng.randint(2, 4), vlo=1700.0, corner=rng.random() < 0.3)
    if c["kind"] != "forward":
        c.update(prec=rng.choice(["f32", "f16", "f16", "bf16"]), freesurf=False, dr=rng.choice([1, 1, 1, 4]))
    if c["kind"] in ("family", "autograd"):
        c.update(prec="f32", dr=1)
    if c.get("ny", 1) > 1:
        c["off"] = False                    # receiver carpets lie on nodes
    c = _case(**c)
    top = max(_points(k) * _cost(k) for k in listed())
    while _points(c) * _cost(c) > top:
        c["nt"] = int(c["nt"] * 0.8)
    return c


# ---------------------------------------------------------------------------
# Inputs

def _dims(c):
    """Sizes along z, x(, y)."""
    return [c["nz"], c["nx"]] + ([c["ny"]] if c["ny"] > 1 else [])


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _smooth_noise(rng, shape, cells, dev):
    """Smooth noise in about [-1, 1]: a coarse random grid, interpolated."""
    coarse = [max(3, int(round(s / cells)) + 2) for s in shape]
    t = torch.from_numpy(rng.uniform(-1.0, 1.0, coarse).astype(np.float32)).to(dev)
    mode = "bilinear" if len(shape) == 2 else "trilinear"
    return torch.nn.functional.interpolate(t[None, None], size=shape, mode=mode, align_corners=True)[0, 0]


def _models(c, seed):
    """(vp, rho): velocities from vlo to vhi rising with depth, smooth, in
    dipping layers, or layers with a fast body; Gardner's densities."""
    dev = _device()
    rng = np.random.default_rng(seed)
    shape = tuple(reversed(_dims(c)))       # z fastest
    depth = torch.linspace(0.0, 1.0, c["nz"], device=dev)
    f = depth + 0.18 * _smooth_noise(rng, shape, 24, dev)
    if c["model"] != "smooth":
        nl = int(rng.integers(7, 14))
        f = torch.floor(f * nl) / nl
        if c["model"] == "salt":
            f = f * 0.6
    f = f.clamp(0.0, 1.0)
    if c["model"] == "salt":
        r2 = ((depth - rng.uniform(0.5, 0.65)) / 0.28) ** 2
        for ax in range(1, len(shape)):
            x = torch.linspace(0.0, 1.0, shape[-1 - ax], device=dev).reshape([-1] + [1] * ax)
            r2 = r2 + ((x - rng.uniform(0.4, 0.6)) / 0.2) ** 2
        f = torch.where(r2 < 1.0, torch.ones_like(f), f)
    vp = (c["vlo"] + (c["vhi"] - c["vlo"]) * f).float().contiguous()
    rho = (310.0 * vp ** 0.25).contiguous()
    return vp, rho


def _geometry(c):
    """Source positions (nshot, 3) and one receiver array (nrec, 3), metres (z, x, y)."""
    h, ns = c["h"], c["shots"]
    zs = zr = 2.0
    fx = 0.0
    if c["off"]:
        zs, zr, fx = 6.37, 5.71, 0.43
    ix = np.arange(0, c["nx"] - 1, c["rec_step"]) + fx
    sx = np.round((np.arange(ns) + 0.5) / ns * (c["nx"] - 2)) + fx
    if c["ny"] == 1:
        srcs = np.stack([np.full(ns, zs), sx, np.zeros(ns)], 1)
        recs = np.stack([np.full(ix.size, zr), ix, np.zeros(ix.size)], 1)
    else:
        sy = np.full(ns, float(c["ny"] // 2))
        if c["corner"]:
            sx, sy = np.arange(ns) * 10.0, np.zeros(ns)
        iy = np.arange(0, c["ny"] - 1, c["rec_step"]) + fx
        gx, gy = np.meshgrid(ix, iy, indexing="xy")
        srcs = np.stack([np.full(ns, zs), sx, sy], 1)
        recs = np.stack([np.full(gx.size, zr), gx.ravel(), gy.ravel()], 1)
    return srcs * h, recs * h


def _wavelet(c):
    return synth.ricker(c["nt"], c["dt"], c["fm"])


def _observed(c, seed, dev):
    """Recorded data, flat: the direct arrival and a few reflections as
    hyperbolas with the source's amplitude and spreading, plus weak noise."""
    rng = np.random.default_rng(seed + 1)
    srcs, recs = _geometry(c)
    d3 = c["ny"] > 1
    v0 = 0.5 * (c["vlo"] + c["vhi"])
    zmax = c["nz"] * c["h"]
    events = [(0.0, c["vlo"], 1.0)]
    for _ in range(4):
        z = rng.uniform(0.15, 0.95) * zmax
        events.append((z, c["vlo"] + (v0 - c["vlo"]) * z / zmax, rng.uniform(0.05, 0.25) * rng.choice([-1.0, 1.0])))
    t = (torch.arange(c["nt"], device=dev, dtype=torch.float32) * c["dt"] - 1.2 / c["fm"])[:, None]
    rec = torch.from_numpy(recs.astype(np.float32)).to(dev)
    g = torch.Generator(device="cpu").manual_seed(seed + 2)
    noise = torch.randn(c["nt"], generator=g).to(dev)
    out = []
    w0 = 2.0 * math.pi * c["fm"]
    for s in srcs:
        off2 = ((rec - torch.tensor(s, device=dev, dtype=torch.float32)) ** 2).sum(1) + c["h"] ** 2
        tr = torch.zeros(c["nt"], len(recs), device=dev)
        for z, v, a in events:
            r = torch.sqrt(off2 + 4.0 * z * z)
            amp = a * w0 / (4.0 * math.pi * v * v * r) if d3 else \
                a * math.sqrt(math.pi * w0) / (2.0 * math.pi * v * v) * torch.sqrt(v / (2.0 * r))
            q = (math.pi * c["fm"] * (t - r / v)) ** 2
            tr += amp * (1.0 - 2.0 * q) * torch.exp(-q)
        tr += 0.02 * float(tr.abs().mean()) * noise[:, None]
        out.append(tr.reshape(-1))
    return torch.cat(out)


def _problem(c):
    return smi.Problem(tuple([c["h"]] * len(_dims(c))), c["nt"], c["dt"], c["fm"], order=c["order"], nb=NB,
                       use_box=c["box"], shell_prec=c["prec"], dr=c["dr"], freesurf=c["freesurf"],
                       per_shot=c["per_shot"])


def prepare(case, seed):
    vp, rho = _models(case, seed)
    srcs, recs = _geometry(case)
    st = {"case": case, "vp": vp, "rho": rho, "prob": _problem(case), "srcs": srcs, "recs": [recs] * len(srcs),
          "stf": torch.from_numpy(_wavelet(case)).to(vp.device)}
    if case["kind"] != "forward":
        st["dobs"] = _observed(case, seed, vp.device)
    return st


def run(state):
    s = state
    args = (s["vp"], s["rho"], s["prob"], s["srcs"], s["recs"], s["stf"])
    kind = s["case"]["kind"]
    if kind == "forward":
        return smi.smi_forward(*args)
    if kind == "rtm":
        return smi.smi_rtm(*args, s["dobs"])
    if kind == "gradient":
        return smi.smi_fwi_gradient(*args, s["dobs"])
    if kind == "family":
        return smi.smi_fwi_gradient_family(*args, s["dobs"], family=2)
    vp = s["vp"].detach().requires_grad_()
    J = autograd.misfit(vp, *args[1:], s["dobs"])
    grad, = torch.autograd.grad(J, vp)
    return J.detach(), grad


# ---------------------------------------------------------------------------
# Work

def _cost(c):
    """Propagations of a pass, by their bytes."""
    return {"forward": 1.0, "family": 5.0}.get(c["kind"], 3.5)


def _points(c):
    """Grid points advanced by one propagation, all steps and shots (whole grid)."""
    v = float(c["nt"]) * c["shots"]
    for n in _dims(c):
        v *= n + 2 * NB
    return v


def _box_points(c, extents, reach):
    """Points inside the computing box summed over the steps: the box grows
    around the extent by vmax dt a step (physical nodes only for reach = 0)."""
    total = 0.0
    N = c["order"] // 2
    steps = np.arange(1, c["nt"] + 1)
    grow = np.ceil(c["vhi"] * c["dt"] * steps / c["h"]) + 3 * N
    for lo, hi in extents:
        v = np.ones(c["nt"])
        for a, n in enumerate(_dims(c)):
            l0, h0 = lo[a] / c["h"], hi[a] / c["h"]
            g = grow if c["box"] else 10 * n + grow
            v = v * (np.minimum(h0 + g, n - 1 + reach) - np.maximum(l0 - g, -reach) + 1)
        total += float(v.sum())
    return total


def work(case):
    """Bytes and operations of one pass, taken from the scheme: every step of
    a propagation reads and writes its state (pressure, one velocity a
    dimension) once and reads the model (two arrays) once, on the nodes that
    the wave can have reached; reconstruction adds the adjoint pressure and
    the accumulator; boundaries are written and read once; the model is read
    and the results are written once."""
    c = case
    d = len(_dims(c))
    N = c["order"] // 2
    srcs, recs = _geometry(c)
    src = [(s, s) for s in srcs]
    rec = [(recs.min(0), recs.max(0))] * len(srcs)
    pf, pa, pr = _box_points(c, src, NB), _box_points(c, rec, NB), _box_points(c, src, 0)
    step = 4 * (2 * (1 + d) + 2)
    flops = d * 2 * (3 * N) + 4 * d + 2
    nsv = c["nt"] * len(recs) * len(srcs)
    phys = float(np.prod(_dims(c)))
    b = pf * step + 8 * phys + 4 * nsv
    f = pf * flops
    if c["kind"] != "forward":
        band = sum(2 * (2 * N - 1) * phys / n for n in _dims(c)) * c["nt"] * len(srcs) / c["dr"]
        b += pa * step + pr * (step + 12) + 2 * band * (4 if c["prec"] == "f32" else 2) + 4 * phys + 2 * 4 * nsv
        f += pa * flops + pr * (flops + 2)
    if c["kind"] == "family":
        b += pr * 4 * d * 4 + 4 * phys      # both velocities, adjoint velocity, accumulator, per axis
        f += pr * 3 * d
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# The same results in 64 bits: the scheme of the method (staggered leap-frog,
# CPML, image-method free surface, exact discrete adjoint, stored source field)
# written with plain torch operations on whole arrays.

class _Scheme:
    def __init__(self, c, seed):
        self.c = c
        vp32, rho32 = _models(c, seed)
        self.dev = vp32.device
        self.n = _dims(c)
        self.d = len(self.n)
        self.ne = [n + 2 * NB for n in self.n]
        self.N = N = c["order"] // 2
        self.coef = [9.0 / 8, -1.0 / 24] if N == 2 else [1225.0 / 1024, -245.0 / 3072, 49.0 / 5120, -5.0 / 7168]
        self.coef = [v / c["h"] for v in self.coef]
        self.dt = c["dt"]
        self.vp, self.rho = vp32.double(), rho32.double()
        self.K = self._extend(self.rho * self.vp ** 2)
        r = self._extend(self.rho)
        self.b = []
        for a in range(self.d):
            nx = torch.cat([self._cut(r, a, 1, self.ne[a]), self._cut(r, a, self.ne[a] - 1, self.ne[a])],
                           self._ax(a))
            self.b.append(2.0 / (r + nx))    # the last node of an axis: 1 / rho
        vmax = float(vp32.max())
        self.tab = [[self._cpml(a, vg, vmax) for vg in (False, True)] for a in range(self.d)]

    def _ax(self, a):
        return -1 - a

    def _cut(self, x, a, lo, hi):
        return x.narrow(self._ax(a), lo, hi - lo)

    def _extend(self, x):
        for a in range(self.d):
            i = torch.arange(self.ne[a], device=self.dev) - NB
            x = x.index_select(x.dim() - 1 - a, i.clamp(0, self.n[a] - 1))
        return x

    def _slabs(self, a):
        return ((0, NB), (self.ne[a] - NB - 1, self.ne[a]))

    def _cpml(self, a, vgrid, vmax):
        h, L = self.c["h"], NB * self.c["h"]
        d0 = -3.0 * vmax * math.log(1e-3) / (2.0 * L)
        x = np.arange(self.ne[a]) + (0.5 if vgrid else 0.0)
        q = np.minimum(np.maximum(np.maximum(NB - x, x - (self.ne[a] - NB - 1)), 0.0) * h, L) / L
        damp, al = d0 * q * q, math.pi * self.c["fm"] * (1.0 - q)
        bb = np.exp(-(damp + al) * self.dt)
        out = []
        for v in (np.where(q > 0, damp * (bb - 1.0) / (damp + al), 0.0), np.where(q > 0, bb, 0.0)):
            if a == 0 and self.c["freesurf"]:
                v = v.copy()
                v[:NB] = 0.0
            v = torch.from_numpy(v).to(self.dev).reshape([-1] + [1] * a)
            out.append([v[lo:hi] for lo, hi in self._slabs(a)])
        return out                          # [A pieces, B pieces]

    def zeros(self, ns):
        return torch.zeros([ns] + self.ne[::-1], dtype=torch.float64, device=self.dev)

    def memory(self, ns):
        out = []
        for a in range(self.d):
            out.append([])
            for lo, hi in self._slabs(a):
                s = self.ne[::-1]
                s[len(s) - 1 - a] = hi - lo
                out[a].append(torch.zeros([ns] + s, dtype=torch.float64, device=self.dev))
        return out

    def state(self, ns):
        return {"p": self.zeros(ns), "v": [self.zeros(ns) for _ in range(self.d)], "mv": self.memory(ns),
                "mp": self.memory(ns)}

    def D(self, x, a, up):
        """Staggered derivative along a: p nodes to v nodes (up), or back."""
        o, n = torch.zeros_like(x), self.ne[a]
        for l, cl in enumerate(self.coef, 1):
            f, g = (l, l - 1) if up else (l - 1, l)
            self._cut(o, a, 0, n - f).add_(self._cut(x, a, f, n), alpha=cl)
            self._cut(o, a, g, n).sub_(self._cut(x, a, 0, n - g), alpha=cl)
        return o

    def _absorb(self, Dx, a, mem, tab):
        for k, (lo, hi) in enumerate(self._slabs(a)):
            m, part = mem[a][k], self._cut(Dx, a, lo, hi)
            m.mul_(tab[1][k]).addcmul_(tab[0][k].expand_as(m), part)
            part.add_(m)

    def forward_step(self, s, it, src, stf):
        for a in range(self.d):
            g = self.D(s["p"], a, True)
            self._absorb(g, a, s["mv"], self.tab[a][1])
            s["v"][a].sub_(g.mul_(self.b[a]), alpha=self.dt)
        if self.c["freesurf"]:
            for j in range(self.N):
                s["v"][0][..., NB - 1 - j] = s["v"][0][..., NB + j]
        div = 0
        for a in range(self.d):
            g = self.D(s["v"][a], a, False)
            self._absorb(g, a, s["mp"], self.tab[a][0])
            div = g if a == 0 else div.add_(g)
        s["p"].sub_(div.mul_(self.K), alpha=self.dt)
        idx, w = src
        s["p"].view(-1).index_add_(0, idx, w * (stf[it] * self.dt / self.c["h"] ** self.d))
        if self.c["freesurf"]:
            s["p"][..., NB] = 0.0
            for j in range(1, self.N + 1):
                s["p"][..., NB - j] = -s["p"][..., NB + j]

    def _operand(self, x, a, mem, tab):
        """x + A (x + mem) on the slabs (the transposed CPML term)."""
        y = x.clone()
        for k, (lo, hi) in enumerate(self._slabs(a)):
            y_, x_ = self._cut(y, a, lo, hi), self._cut(x, a, lo, hi)
            y_.addcmul_(tab[0][k].expand_as(x_), x_ + mem[a][k])
        return y

    def _recur(self, x, a, mem, tab):
        for k, (lo, hi) in enumerate(self._slabs(a)):
            mem[a][k].add_(self._cut(x, a, lo, hi)).mul_(tab[1][k])

    def adjoint_step(self, s):
        for a in range(self.d):
            g = self.D(self._operand(s["p"], a, s["mp"], self.tab[a][0]), a, True)
            self._recur(s["p"], a, s["mp"], self.tab[a][0])
            s["v"][a].sub_(g.mul_(self.b[a]), alpha=self.dt)
        div = 0
        for a in range(self.d):
            g = self.D(self._operand(s["v"][a], a, s["mv"], self.tab[a][1]), a, False)
            self._recur(s["v"][a], a, s["mv"], self.tab[a][1])
            div = g if a == 0 else div.add_(g)
        s["p"].sub_(div.mul_(self.K), alpha=self.dt)

    def points(self, pos):
        """Flat node indices and weights (k, taps) of positions, Kaiser-windowed sinc of radius N, shape 4."""
        idx = torch.zeros(len(pos), 1, dtype=torch.int64, device=self.dev)
        w = torch.ones(len(pos), 1, dtype=torch.float64, device=self.dev)
        stride = 1
        for a in range(self.d):
            x = pos[:, a] / self.c["h"] + NB
            if np.all(np.abs(x - np.round(x)) < 1e-6):
                node, wt = np.round(x)[:, None], np.ones((len(pos), 1))
            else:
                node = np.floor(x)[:, None] + np.arange(1 - self.N, self.N + 1)[None]
                u = node - x[:, None]
                wt = np.sinc(u) * np.i0(4.0 * np.sqrt(np.maximum(1.0 - (u / self.N) ** 2, 0.0))) / np.i0(4.0)
                wt = np.where(np.abs(u) < self.N, wt, 0.0)
                if a == 0 and self.c["freesurf"]:
                    out = np.zeros_like(wt)  # weights above the surface fold, negated, onto their mirrors
                    first = node[:, 0]
                    for k in range(node.shape[1]):
                        t = np.where(node[:, k] < NB, 2 * NB - node[:, k], node[:, k]) - first
                        sg = np.sign(node[:, k] - NB)
                        np.add.at(out, (np.arange(len(pos)), t.astype(int)), sg * wt[:, k])
                    wt = out
            node = torch.from_numpy(node.astype(np.int64)).to(self.dev)
            wt = torch.from_numpy(wt).to(self.dev)
            idx = (idx[:, :, None] + stride * node[:, None, :]).reshape(len(pos), -1)
            w = (w[:, :, None] * wt[:, None, :]).reshape(len(pos), -1)
            stride *= self.ne[a]
        return idx, w

    def phys(self, x):
        for a in range(self.d):
            x = self._cut(x, a, NB, NB + self.n[a])
        return x


def _clone(s):
    def cp(x):
        return [cp(y) for y in x] if isinstance(x, list) else x.clone()
    return {k: cp(v) for k, v in s.items()}


def _exact_group(S, shots, recs, stf, dobs, kind):
    """Seismograms, misfit and accumulators of a group of shots: (seis, acc, [G per axis])."""
    c, ns, nt = S.c, len(shots), S.c["nt"]
    ntot = int(np.prod(S.ne))
    base = torch.arange(ns, device=S.dev)[:, None]
    si, sw = S.points(shots)
    src = ((si + base * ntot).reshape(-1), sw.reshape(-1))
    ri, rw = S.points(recs)
    ri = ri[None] + base[:, :, None] * ntot
    seis = torch.zeros(ns, nt, len(recs), dtype=torch.float64, device=S.dev)
    seg = nt if kind == "forward" else max(1, min(nt, int(6e9 / (8.0 * ns * ntot * (1 + S.d * (kind == "family"))))))
    s, saved = S.state(ns), []
    for it in range(nt):
        if kind != "forward" and it % seg == 0:
            saved.append(_clone(s))
        S.forward_step(s, it, src, stf)
        seis[:, it] = (s["p"].reshape(-1)[ri] * rw).sum(-1)
    if kind == "forward":
        return seis, None, None
    res = dobs if kind == "rtm" else seis - dobs
    s = None
    adj = S.state(ns)
    acc = torch.zeros([ns] + S.n[::-1], dtype=torch.float64, device=S.dev)
    G = [S.zeros(1)[0] for _ in range(S.d)] if kind == "family" else None
    rk = rw * S.K.reshape(-1)[S.points(recs)[0]]
    for k in reversed(range(len(saved))):
        f, keep, vel = saved[k], [], []
        for it in range(k * seg, min(nt, (k + 1) * seg)):
            old = [v.clone() for v in f["v"]] if G else None
            S.forward_step(f, it, src, stf)
            if kind == "rtm":
                keep.append(S.phys(f["p"]).clone())
            else:
                keep.append(sum(S.phys(S.D(f["v"][a], a, False)) for a in range(S.d)))
            if G:
                vel.append([f["v"][a] - old[a] for a in range(S.d)])
        saved[k] = None
        for it in reversed(range(k * seg, min(nt, (k + 1) * seg))):
            adj["p"].view(-1).index_add_(0, ri.reshape(-1), (rk[None] * res[:, it, :, None]).reshape(-1))
            acc.addcmul_(S.phys(adj["p"]), keep.pop())
            S.adjoint_step(adj)
            if G:
                dv = vel.pop()
                for a in range(S.d):
                    G[a].add_((adj["v"][a] * dv[a]).sum(0))
    return seis, acc, G


def exact(case, seed):
    c = case
    est = _points(c) * (1 if c["kind"] == "forward" else 3.5) * len(_dims(c)) / 3.0 * 2.6e-10
    est += c["nt"] * (1 if c["kind"] == "forward" else 3.5) * 1.2e-3
    if est > 17.0 or c["dr"] > 1 and c["kind"] == "family":
        return None
    with torch.no_grad():
        S = _Scheme(c, seed)
        srcs, recs = _geometry(c)
        stf = _wavelet(c).astype(np.float64)
        kind = "gradient" if c["kind"] == "autograd" else c["kind"]
        nrec = len(recs)
        dobs = None
        if kind != "forward":
            dobs = _observed(c, seed, S.dev).double().reshape(len(srcs), c["nt"], nrec)
        group = max(1, int(6e8 / (8.0 * np.prod(S.ne))))
        seis, acc, G, J = [], 0, None, 0.0
        for k in range(0, len(srcs), group):
            d = None if dobs is None else dobs[k:k + group]
            u, a, g = _exact_group(S, srcs[k:k + group], recs, stf, d, kind)
            if kind == "forward":
                seis += list(u)
                continue
            J = J + 0.5 * ((u - d) ** 2).sum()
            acc = acc + a.sum(0)
            if g:
                G = g if G is None else [x + y for x, y in zip(G, g)]
        if kind == "forward":
            return seis
        if kind == "rtm":
            return acc
        grad = -2.0 * S.dt * acc / S.vp
        if c["kind"] == "autograd":
            return J, grad
        if kind == "gradient":
            return J.reshape(1), grad
        gb = 0                               # half of each half node's sum goes to both of its nodes
        for a in range(S.d):
            lo = G[a]
            for e in range(S.d):
                lo = S._cut(lo, e, NB - (e == a), NB + S.n[e])
            gb = gb + S._cut(lo, a, 1, S.n[a] + 1) + S._cut(lo, a, 0, S.n[a])
        gr = -S.dt * acc / S.rho + 0.5 * gb
        return J.reshape(1), grad - gr * S.rho / S.vp, gr / S.vp
