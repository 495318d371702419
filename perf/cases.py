"""Performance cases: the work that a program using this library has it do.

A case is a dict of plain values.  ``listed()`` names the fixed ones, ``draw(rng)`` makes
another of the same ranges, ``prepare`` builds what a program has in hand before the call
(velocity grid, acquisition, wavelets, observed data on the GPU, a model handle), ``run``
is one pass through the public entry points, ``exact`` is the same computation in 64 bits
with plain torch.

Kinds of case
  forward   FwiModel.forward: traces, with ``final`` also the last two wavefields, with
            ``misfit`` also fwi_misfit of the traces against observed data (the evaluation
            a line search makes)
  gradient  FwiModel.gradient: misfit and gradient; with ``loop`` the call an FWI iteration
            makes, WaveFwi.apply (installs a new velocity) and its backward
  serve     fwi_serve on a list of host requests (2-D and 3-D, forward and gradient)
  codec     fwi_snapshot_encode and fwi_snapshot_decode of one state pair

Step counts are shorter than a survey's, so that a pass takes seconds at most; a gradient
then keeps the ratio of checkpoints to steps of the long run (``slots``).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1912_08063_gb300 import fwi

VMIN, VMAX = 1500.0, 4500.0
ESIZE = {"fp32": 4, "bf16": 2, "fp16": 2}


# ---------------------------------------------------------------- the cases

def _wave(name, kind, shape, nt, order=8, shots=1, snap="fp32", slots=0, nb=20, h=10.0, rec=1,
          aniso=False, offgrid=False, final=False, misfit=False, loop=False):
    """shape (nz, nx) or (nz, ny, nx); slots: checkpoint budget in codes of one field of
    all shots (0: the library's default budget); rec: receiver spacing in cells."""
    nz, ny, nx = shape if len(shape) == 3 else (shape[0], 0, shape[1])
    c = {"kind": kind, "nz": nz, "ny": ny, "nx": nx, "nt": nt, "order": order, "shots": shots,
         "snap": snap, "slots": slots, "nb": nb, "h": h, "rec": rec, "aniso": aniso,
         "offgrid": offgrid, "final": final, "misfit": misfit, "loop": loop}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one shot on the two-layer model's grid: a single small request, where launches count
        _wave("forward 2d 201", "forward", (201, 201), 500),
        # its gradient with lossless checkpoints
        _wave("gradient 2d 201", "gradient", (201, 201), 500, snap="fp32"),
        # one shot of a mid-size 2-D model at 16th order, wavefields returned
        _wave("forward 2d 517x900 o16", "forward", (517, 900), 500, order=16, final=True),
        # observed data of a 64-shot line and its misfit: a line-search evaluation
        _wave("forward 2d 400x1024x64", "forward", (400, 1024), 500, shots=64, misfit=True),
        # the FWI iteration on that line: new velocity, misfit, gradient, BF16 checkpoints
        _wave("fwi 2d 400x1024x64", "gradient", (400, 1024), 500, shots=64, snap="bf16",
              slots=500, loop=True),
        # the 96^3 twin of the salt model, 16th order, FP16 checkpoints with recomputation
        _wave("gradient 3d 96 o16", "gradient", (96, 96, 96), 400, order=16, snap="fp16",
              slots=60, h=66.7, rec=2),
        # two shots with off-grid sources and receivers on a ragged 3-D grid
        _wave("gradient 3d 90x75x110 off", "gradient", (90, 75, 110), 150, shots=2, snap="fp32",
              slots=300, rec=4, offgrid=True),
        # the 256^3 layered model, 8th order, BF16 checkpoints with recomputation
        _wave("gradient 3d 256", "gradient", (256, 256, 256), 400, snap="bf16", slots=100, rec=2),
        # the paper's benchmark: 1024^3, 8th order, 100 steps
        _wave("forward 3d 1024", "forward", (1024, 1024, 1024), 100, rec=2, final=True),
        # the 512^3 salt model, 16th order, FP16 checkpoints for one step in six
        _wave("gradient 3d 512 o16", "gradient", (512, 512, 512), 200, order=16, snap="fp16",
              slots=33, h=12.5, rec=2),
        # a stream of mixed requests from host memory through the serving loop
        {"name": "serve 10 mixed", "kind": "serve", "n": 10, "mix": 3},
        # one checkpoint of a 256^3 model's state, stored and restored
        {"name": "codec 296^3 fp16", "kind": "codec", "n": 296 * 296 * 296, "snap": "fp16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    r = rng.random()
    if r < 0.08:
        return {"kind": "codec", "n": _log(rng, 2000, 168000000),
                "snap": rng.choice(["fp32", "bf16", "fp16"])}
    if r < 0.14:
        return {"kind": "serve", "n": rng.randint(2, 12), "mix": rng.randint(10, 10000)}
    gradient = rng.random() < 0.55
    order = rng.choice([8, 16])
    nb = rng.choice([20, 20, rng.randint(10, 40)])
    if rng.random() < 0.55:
        # sides 64 .. 1024, one shot or a line of up to 64
        shape = (_log(rng, 64, 1024), _log(rng, 64, 1024))
        shots = 1 if rng.random() < 0.5 else _log(rng, 2, 64)
    else:
        shape = (_log(rng, 48, 400), _log(rng, 48, 400), _log(rng, 48, 400))
        shots = rng.choice([1, 1, 2, 3])
    nt = _log(rng, 100, 600)
    points = shots
    for s in shape:
        points *= s + 2 * nb
    cap = 3.0e9 if gradient else 8.0e9          # point steps, far below the largest listed
    nt = max(40, min(nt, int(cap / points)))
    snap = rng.choice(["fp32", "bf16", "fp16"])
    # every state stored, or checkpoints for a part of the steps (binomial recomputation)
    slots = 2 * nt if rng.random() < 0.5 else max(4, int(nt * rng.uniform(0.08, 0.5)))
    slots = max(4, min(slots, int(40e9 / (points * ESIZE[snap]))))
    rec = rng.choice([1, 2, 3]) if len(shape) == 2 else rng.choice([2, 3, 5])
    return _wave("", "gradient" if gradient else "forward", shape, nt, order=order, shots=shots,
                 snap=snap, slots=slots if gradient else 0, nb=nb, h=rng.choice([5.0, 10.0, 12.5]),
                 rec=rec, aniso=rng.random() < 0.2, offgrid=rng.random() < 0.2,
                 final=not gradient and rng.random() < 0.5,
                 misfit=not gradient and rng.random() < 0.3, loop=gradient and rng.random() < 0.4)


# ---------------------------------------------------------------- inputs

def _shape(c):
    return (c["nz"], c["nx"]) if c["ny"] == 0 else (c["nz"], c["ny"], c["nx"])


def _spacing(c):
    """(hz, hy, hx); the anisotropic option has finer z."""
    h = c["h"]
    return [0.8 * h if c["aniso"] else h, h, h]


def _dt(c):
    """Three quarters to nine tenths of the stability limit at VMAX."""
    hmin = min(_spacing(c))
    return (1.0e-3 if c["ny"] == 0 else 0.8e-3) * hmin / 10.0


def _velocity(shape, seed, device):
    """Layers from 1500 to 4500 m/s with smooth random perturbations of a few per cent."""
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    nz = shape[0]
    tops = torch.sort(torch.rand(7, generator=g, device=device) * 0.9 * nz + 0.05 * nz).values
    vel = torch.linspace(1500.0, 4400.0, 8, device=device)
    z = torch.arange(nz, device=device, dtype=torch.float32)
    layer = vel[torch.bucketize(z, tops)].reshape([-1] + [1] * (len(shape) - 1))
    coarse = [1, 1] + [max(4, n // 16 + 2) for n in shape]
    noise = torch.randn(coarse, generator=g, device=device)
    mode = "bilinear" if len(shape) == 2 else "trilinear"
    pert = torch.nn.functional.interpolate(noise, size=list(shape), mode=mode, align_corners=True)[0, 0]
    return (layer * (1.0 + 0.05 * pert)).clamp_(VMIN, VMAX).contiguous()


def _ricker(t, f0):
    a = (math.pi * f0 * (t - 1.5 / f0)) ** 2
    return (1.0 - 2.0 * a) * (torch.exp(-a) if torch.is_tensor(a) else np.exp(-a))


def _f0(c, seed):
    # a few points per wavelength more or less from call to call
    return (0.9 + 0.02 * (seed % 11)) * 200.0 / c["h"]


def _geometry(c, seed):
    """Source and receiver positions (physical index units): sources near the surface,
    receivers on row or plane 5 (every `rec` cells)."""
    rng = np.random.default_rng([seed, 77])
    ns, nz, nx, ny = c["shots"], c["nz"], c["nx"], max(1, c["ny"])
    sx = (np.arange(ns) + rng.uniform(0.3, 0.7)) * nx / ns
    sy = np.full(ns, ny * rng.uniform(0.4, 0.6) if c["ny"] else 0.0)
    src = np.stack([np.full(ns, 10.0), sy, sx], axis=1)
    yy, xx = np.meshgrid(np.arange(0, ny, c["rec"]), np.arange(0, nx, c["rec"]), indexing="ij")
    rec = np.stack([np.full(yy.size, 5.0), yy.ravel(), xx.ravel()], axis=1)
    if c["offgrid"]:
        src[:, 0] += rng.uniform(0.1, 0.9, ns)
        rec += rng.uniform(0.05, 0.9, rec.shape)
        rec = np.minimum(rec, [nz - 1.0, ny - 1.0, nx - 1.0])
    else:
        src = np.floor(src)
    src = np.minimum(src, [nz - 1.0, ny - 1.0, nx - 1.0])
    if c["ny"] == 0:
        src[:, 1] = 0.0
        rec[:, 1] = 0.0
    return src, rec


def _observed(c, seed, src, rec, f0, device):
    """Traces of a simple recorded shot: the direct wave and two reflections, Ricker
    pulses at their travel times with the amplitude of a point source in a uniform
    medium."""
    h = _spacing(c)
    dt, nt = _dt(c), c["nt"]
    hs = torch.tensor(h, device=device, dtype=torch.float32)
    s = torch.as_tensor(src, device=device, dtype=torch.float32) * hs
    q = torch.as_tensor(rec, device=device, dtype=torch.float32) * hs
    dist = (s[:, None, :] - q[None, :, :]).norm(dim=2) + h[2]           # [shot][rec]
    t = (torch.arange(nt, device=device, dtype=torch.float32) + 1.0) * dt
    rng = np.random.default_rng([seed, 78])
    out = torch.zeros((c["shots"], nt, rec.shape[0]), device=device)
    for depth, amp in ((0.0, 1.0), (rng.uniform(0.2, 0.4), 0.4), (rng.uniform(0.5, 0.8), -0.3)):
        r = torch.sqrt(dist * dist + (2.0 * depth * c["nz"] * h[0]) ** 2)
        v = 1500.0 * (1.0 + depth)
        if c["ny"]:
            a = amp * h[0] * h[1] * h[2] / (4.0 * math.pi * v * v * r)
        else:
            a = amp * h[0] * h[2] / (2.0 * math.pi * v * v) * torch.sqrt(v / (2.0 * f0 * r))
        out += a[:, None, :] * _ricker(t[None, :, None] - (r / v)[:, None, :], f0)
    return out


def _inputs(c, seed, device):
    v = _velocity(_shape(c), seed, device)
    src, rec = _geometry(c, seed)
    f0 = _f0(c, seed)
    t = np.arange(c["nt"], dtype=np.float64) * _dt(c)
    w = np.broadcast_to(_ricker(t, f0), (c["shots"], c["nt"]))
    wav = torch.from_numpy(np.ascontiguousarray(w, dtype=np.float32)).to(device)
    dobs = None
    if c["kind"] == "gradient" or c["misfit"]:
        dobs = _observed(c, seed, src, rec, f0, device)
    return v, src, rec, wav, dobs


def _serve_sizes(c):
    """The requests' kinds and sizes (the case's own, not the seed's): three in four 2-D
    with sides 128 .. 1024, else 3-D with sides 64 .. 192; half of them gradients."""
    rng = np.random.default_rng([c["mix"], 79])
    out = []
    for i in range(c["n"]):
        two = i % 4 != 3 if c["n"] >= 4 else rng.random() < 0.75
        kind = "gradient" if rng.random() < 0.5 else "forward"
        nt = int(rng.integers(100, 601))
        if two:
            shape = tuple(int(x) for x in np.exp(rng.uniform(np.log(128), np.log(1024), 2)))
        else:
            shape = tuple(int(x) for x in np.exp(rng.uniform(np.log(64), np.log(192), 3)))
        out.append(_wave("", kind, shape, nt, snap="bf16", slots=128))
    return out


def _serve_requests(c, seed, device):
    reqs = []
    for i, q in enumerate(_serve_sizes(c)):
        v, src, rec, wav, dobs = _inputs(q, seed + 131 * i, device)
        r = {"kind": q["kind"], "v": v.cpu().numpy(), "h": q["h"], "dt": _dt(q), "nt": q["nt"],
             "order": q["order"], "snap_dtype": q["snap"], "src": src[0].astype(np.int32),
             "rec": rec.astype(np.int32), "wavelet": wav[0].cpu().numpy(), "arrival": 0.0}
        if dobs is not None:
            r["d_obs"] = dobs[0].cpu().numpy()
        reqs.append(r)
    return reqs


def _pair(c, seed, device):
    """A state pair (u^n, u^{n-1}): wavefield-sized values over several decades, the older
    one close to the newer."""
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    n = c["n"]
    a = torch.randn(n, generator=g, device=device) * 1e-7
    a *= torch.exp(-8.0 * torch.rand(n, generator=g, device=device))
    b = a * (1.0 - 0.05 * torch.randn(n, generator=g, device=device))
    return a, b


# ---------------------------------------------------------------- the passes

def prepare(case, seed):
    device = torch.device("cuda", torch.cuda.current_device())
    c = case
    if c["kind"] == "serve":
        return {"case": c, "requests": _serve_requests(c, seed, device)}
    if c["kind"] == "codec":
        a, b = _pair(c, seed, device)
        n, dt = c["n"], fwi.SNAP_DTYPES[c["snap"]]
        code = torch.empty(2 * n, dtype=torch.float32 if dt == 0 else torch.int16, device=device)
        return {"case": c, "a": a, "b": b, "code": code, "dtype": dt,
                "scale": torch.empty(2, device=device), "a2": torch.empty_like(a),
                "b2": torch.empty_like(b)}
    v, src, rec, wav, dobs = _inputs(c, seed, device)
    if c["offgrid"]:
        acq = fwi.Acquisition(src_pos=src, rec_pos=rec)
    else:
        acq = fwi.Acquisition(src.astype(np.int32), rec.astype(np.int32))
    points = c["shots"]
    for s in _shape(c):
        points *= s + 2 * c["nb"]
    budget = int(c["slots"] * 1.02 * points * ESIZE[c["snap"]]) + (1 << 20) if c["slots"] else 0
    model = fwi.FwiModel(v, _spacing(c), _dt(c), c["nt"], order=c["order"], nb=c["nb"],
                         snap_dtype=c["snap"], snap_budget_bytes=budget, sponge_vref=VMAX)
    st = {"case": c, "model": model, "acq": acq, "wav": wav, "dobs": dobs}
    if c["loop"]:
        st["v"] = v
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "serve":
        res, outs = fwi.fwi_serve(state["requests"])
        return {"outputs": outs, "misfit": [float(r["misfit"]) for r in res]}
    if c["kind"] == "codec":
        n, dt = c["n"], state["dtype"]
        fwi.fwi_snapshot_encode(state["a"], state["b"], n, dt, state["code"], state["scale"])
        fwi.fwi_snapshot_decode(state["code"], state["scale"], n, dt, state["a2"], state["b2"])
        return {k: state[k] for k in ("code", "scale", "a2", "b2")}
    model, acq, wav = state["model"], state["acq"], state["wav"]
    if c["kind"] == "forward":
        out = {}
        if c["final"]:
            out["traces"], out["final"] = model.forward(acq, wav, final_state=True)
        else:
            out["traces"] = model.forward(acq, wav)
        if c["misfit"]:
            phi = torch.zeros(1, dtype=torch.float64, device=wav.device)
            fwi.fwi_misfit(out["traces"], state["dobs"], out["traces"].numel(), phi)
            out["misfit"] = phi
        return out
    if c["loop"]:
        v = state["v"].detach().requires_grad_(True)
        phi = fwi.WaveFwi.apply(v, model, acq, wav, state["dobs"])
        phi.backward()
        return {"misfit": phi.detach(), "grad": v.grad}
    phi, grad = model.gradient(acq, wav, state["dobs"])
    return {"misfit": phi, "grad": grad}


# ---------------------------------------------------------------- bytes, flops, tolerances

def work(case):
    """Per point and step: a forward step reads u^n and u^{n-1} and writes u^{n+1} (12
    bytes per shot) and reads W (4 bytes, one field for all shots); a gradient also stores
    u^n and reads it back, and its reverse step reads and writes the accumulated gradient
    (8 bytes).  Recomputed steps are not counted."""
    c = case
    if c["kind"] == "serve":
        parts = [work(q) for q in _serve_sizes(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if c["kind"] == "codec":
        e = ESIZE[c["snap"]]
        return {"bytes": c["n"] * (8 + 2 * e + 2 * e + 8), "flops": c["n"] * 8}
    grid = 1
    for s in _shape(c):
        grid *= s + 2 * c["nb"]
    ns, nt, e = c["shots"], c["nt"], ESIZE[c["snap"]]
    dims = 3 if c["ny"] else 2
    flops = (dims * (c["order"] // 2) * 3 + 8.0) * grid * ns * nt
    nbytes = (12.0 * ns + 4.0) * grid * nt
    nrec = len(_geometry(c, 0)[1])
    nbytes += 4.0 * ns * nt * nrec
    if c["kind"] == "forward":
        if c["final"]:
            nbytes += 8.0 * grid * ns
        if c["misfit"]:
            nbytes += 8.0 * ns * nt * nrec
    else:
        nbytes += (e * ns + (12.0 + 8.0 + e) * ns + 4.0) * grid * nt + 8.0 * ns * nt * nrec
        nbytes += 8.0 * grid
        flops = 2.0 * flops + 2.0 * grid * ns * nt
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the error measured against 64 bits (forward up to 1.9e-5, gradients
    up to 2e-5, 1.9e-4 and 8.3e-4 with FP32, FP16 and BF16 checkpoints): 32-bit time stepping
    over a few hundred steps; gradients carry the rounding of 16-bit checkpoint codes.  The
    largest single error is seen where the field has decayed to nothing beside the peaks."""
    c = case
    if c["kind"] == "codec":
        return "exact"
    if c["kind"] == "serve":
        return {"rel": 4e-3, "max": 0.16}
    if c["kind"] == "forward":
        return {"rel": 8e-5, "max": 4e-3}
    rel = {"fp32": 1e-4, "fp16": 8e-4, "bf16": 4e-3}[c["snap"]]
    return {"rel": rel, "max": 40 * rel}


# ---------------------------------------------------------------- the same in 64 bits

def _weights(M):
    c = [0.0] * (M + 1)
    for k in range(1, M + 1):
        r = math.factorial(M) ** 2 / (math.factorial(M - k) * math.factorial(M + k))
        c[k] = 2.0 * (-1) ** (k + 1) * r / (k * k)
    c[0] = -2.0 * sum(c[1:])
    return c


def _laplacian(u, axes, c, out):
    """Zero outside the grid; axes: (dimension, 1 / h^2)."""
    torch.mul(u, c[0] * sum(a for _, a in axes), out=out)
    for d, ih2 in axes:
        n = u.shape[d]
        for k in range(1, len(c)):
            if k >= n:
                break
            w = c[k] * ih2
            out.narrow(d, k, n - k).add_(u.narrow(d, 0, n - k), alpha=w)
            out.narrow(d, 0, n - k).add_(u.narrow(d, k, n - k), alpha=w)
    return out


def _kaiser_taps(p):
    """Nodes and weights of the windowed sinc of half width 4 at coordinate p."""
    first = math.floor(p) - 3
    x = np.arange(first, first + 8) - p
    r = np.clip(1.0 - (x / 4.0) ** 2, 0.0, None)
    return np.arange(first, first + 8), np.sinc(x) * np.i0(6.31 * np.sqrt(r)) / np.i0(6.31)


def _points(c, pos, dims, device):
    """Index and weight tensors [points][taps] into a flattened field of `dims`."""
    idx, wgt = [], []
    for p in pos:
        if not c["offgrid"]:
            q = [int(p[0]) + c["nb"], int(p[1]) + (c["nb"] if c["ny"] else 0), int(p[2]) + c["nb"]]
            idx.append([(q[0] * dims[1] + q[1]) * dims[2] + q[2]])
            wgt.append([1.0])
            continue
        z, wz = _kaiser_taps(p[0] + c["nb"])
        y, wy = _kaiser_taps(p[1] + c["nb"]) if c["ny"] else (np.array([0]), np.array([1.0]))
        x, wx = _kaiser_taps(p[2] + c["nb"])
        idx.append(((z[:, None, None] * dims[1] + y[:, None]) * dims[2] + x).ravel())
        wgt.append((wz[:, None, None] * wy[:, None] * wx).ravel())
    return (torch.as_tensor(np.asarray(idx), device=device, dtype=torch.int64),
            torch.as_tensor(np.asarray(wgt), device=device, dtype=torch.float64))


class _Exact:
    """The damped leapfrog scheme, its adjoint and the imaging sum in 64 bits."""

    def __init__(self, c, v, src, rec, wav, device, vref):
        self.c, self.dev = c, device
        nb, f64 = c["nb"], torch.float64
        h = [float(np.float32(x)) for x in _spacing(c)]
        self.dt = float(np.float32(_dt(c)))
        v = v.double()
        if not c["ny"]:
            v = v[:, None, :]
        axes = [(1, 1.0 / h[0] ** 2), (3, 1.0 / h[2] ** 2)]
        if c["ny"]:
            axes.append((2, 1.0 / h[1] ** 2))
        self.axes, self.coef = axes, _weights(c["order"] // 2)
        self.fold = []          # physical index of every computed index, per axis
        sig = torch.zeros((1, 1, 1), dtype=f64, device=device)
        for a in range(3):
            n = v.shape[a]
            if a == 1 and not c["ny"]:
                self.fold.append(torch.zeros(1, dtype=torch.int64, device=device))
                continue
            i = torch.arange(n + 2 * nb, device=device)
            self.fold.append((i - nb).clamp(0, n - 1))
            depth = ((nb - i).clamp(min=0) + (i - (nb + n - 1)).clamp(min=0)).double()
            emax = 3.0 * vref * math.log(1.0 / 1e-3) / (2.0 * nb * h[a])
            s = 0.5 * self.dt * emax * (depth / nb) ** 2
            sig = sig + s.reshape([-1 if k == a else 1 for k in range(3)])
        self.v = v
        self.dims = [len(f) for f in self.fold]
        vc = v.index_select(0, self.fold[0]).index_select(1, self.fold[1]).index_select(2, self.fold[2])
        self.W = (vc * self.dt) ** 2
        self.inv_ap = 1.0 / (1.0 + sig)
        self.am = 1.0 - sig
        self.si, self.sw = _points(c, src, self.dims, device)
        self.ri, self.rw = _points(c, rec, self.dims, device)
        self.wav = wav.double()
        self.ns = c["shots"]

    def zeros(self):
        return torch.zeros([self.ns] + self.dims, dtype=torch.float64, device=self.dev)

    def sample(self, u):
        return (u.reshape(self.ns, -1)[:, self.ri.reshape(-1)].reshape([self.ns] + list(self.ri.shape))
                * self.rw).sum(-1)

    def step(self, n, u, up, tmp):
        """u^{n+1}, written over up = u^{n-1}."""
        _laplacian(u, self.axes, self.coef, tmp)
        tmp.mul_(self.W).add_(u, alpha=2.0)
        up.mul_(self.am)
        torch.sub(tmp, up, out=up)
        amp = self.dt ** 2 * self.wav[:, n, None] * self.sw
        up.view(self.ns, -1).scatter_add_(1, self.si, amp)
        up.mul_(self.inv_ap)
        return up

    def forward(self, keep=0):
        """Traces, the last two fields and, with keep, the pair at every keep-th step."""
        u, up, tmp = self.zeros(), self.zeros(), self.zeros()
        nt = self.c["nt"]
        tr = torch.empty((self.ns, nt, self.ri.shape[0]), dtype=torch.float64, device=self.dev)
        kept = []
        for n in range(nt):
            if keep and n % keep == 0:
                kept.append((u.clone(), up.clone()))
            u, up = self.step(n, u, up, tmp), u
            tr[:, n] = self.sample(u)
        return tr, u, up, kept

    def gradient(self, dobs):
        nt = self.c["nt"]
        K = max(1, int(math.ceil(math.sqrt(nt))))
        tr, _, _, kept = self.forward(K)
        res = tr - dobs.double()
        phi = (res * res).sum()
        lam, lam2 = self.zeros(), self.zeros()       # lambda^{m+1}, lambda^{m+2}
        g = self.zeros()[0]
        tmp, t2 = self.zeros(), self.zeros()
        ridx = self.ri.reshape(1, -1).expand(self.ns, -1)
        for seg in range(len(kept) - 1, -1, -1):
            u, up = kept.pop()
            states = [u.clone()]
            last = min(nt, (seg + 1) * K)
            for n in range(seg * K, last - 1):
                u, up = self.step(n, u, up, tmp), u
                states.append(u.clone())
            for m in range(last - 1, seg * K - 1, -1):
                # lambda^{m+1} from lambda^{m+2} (lam) and lambda^{m+3} (lam2)
                torch.mul(lam, self.W, out=t2)
                _laplacian(t2, self.axes, self.coef, tmp)
                tmp.add_(lam, alpha=2.0)
                lam2.mul_(self.am)
                torch.sub(tmp, lam2, out=lam2)
                q = (2.0 * res[:, m, :, None] * self.rw).reshape(self.ns, -1)
                lam2.view(self.ns, -1).scatter_add_(1, ridx, q)
                lam2.mul_(self.inv_ap)
                lam, lam2 = lam2, lam
                _laplacian(states.pop(), self.axes, self.coef, tmp)
                g += (tmp.mul_(lam)).sum(0)
        # fold the replicated cells onto the physical ones, d W / d v = 2 v dt^2
        for a in range(3):
            shape = list(g.shape)
            shape[a] = self.v.shape[a]
            g = torch.zeros(shape, dtype=g.dtype, device=self.dev).index_add_(a, self.fold[a], g)
        g = g * 2.0 * self.v * self.dt ** 2
        return phi, g if self.c["ny"] else g[:, 0, :]


def _exact_cost(c):
    """Point steps of stencil work, in 64 bits about 1.2e9 a second at 8th order in 3-D."""
    if c["kind"] == "serve":
        return sum(_exact_cost(q) for q in _serve_sizes(c))
    points = c["shots"] * c["nt"]
    for s in _shape(c):
        points *= s + 2 * c["nb"]
    per = (3 if c["ny"] else 2) * c["order"] / 24.0
    return points * per * (4.0 if c["kind"] == "gradient" else 1.0) + c["nt"] * 2e6


def _exact_codec(c, seed, device):
    a, b = _pair(c, seed, device)
    if c["snap"] == "fp32":
        return {"code": torch.cat([a, b]).double(), "scale": torch.ones(2, dtype=torch.float64),
                "a2": a.double(), "b2": b.double()}
    half = torch.bfloat16 if c["snap"] == "bf16" else torch.float16
    texp = 0 if c["snap"] == "bf16" else 14
    scale, back = [], []
    for x in (a, a - b):
        m, e = math.frexp(float(x.abs().max()))      # max = m 2^e with 0.5 <= m < 1
        s = 2.0 ** (texp - (e - 1) - (1 if m > 0.5 else 0))
        scale.append(s)
        back.append((x.double() * s).to(half).double() / s)
    return {"code": None, "scale": torch.tensor(scale, dtype=torch.float64),
            "a2": back[0], "b2": back[0] - back[1]}


def exact(case, seed):
    c = case
    device = torch.device("cuda", torch.cuda.current_device())
    if c["kind"] == "codec":
        return _exact_codec(c, seed, device)
    if _exact_cost(c) > 1.8e11:
        return None
    if c["kind"] == "serve":
        outs, phis = [], []
        for i, q in enumerate(_serve_sizes(c)):
            v, src, rec, wav, dobs = _inputs(q, seed + 131 * i, device)
            e = _Exact(q, v, src, rec, wav, device, float(v.max()))
            if q["kind"] == "gradient":
                phi, g = e.gradient(dobs)
                outs.append(g)
                phis.append(float(phi))
            else:
                outs.append(e.forward()[0][0])
                phis.append(0.0)
        return {"outputs": outs, "misfit": phis}
    v, src, rec, wav, dobs = _inputs(c, seed, device)
    e = _Exact(c, v, src, rec, wav, device, VMAX)
    if c["kind"] == "gradient":
        phi, g = e.gradient(dobs)
        return {"misfit": phi if c["loop"] else phi.reshape(1), "grad": g}
    tr, u, up, _ = e.forward()
    out = {"traces": tr}
    if c["final"]:
        out["final"] = torch.stack([u, up], dim=1)
    if c["misfit"]:
        r = tr - dobs.double()
        out["misfit"] = (r * r).sum().reshape(1)
    return out
