"""Performance cases of the acoustic FDTD library: what its users run.

Each case is one call (or one short chain of calls) through the package's
public entry points on seeded synthetic inputs: forward modelling of one shot
and of batches of shots on 2D slices and 3D volumes, velocity gradients
(misfit and autograd forms), the source wavelet and the model-builder warps.
Grids, absorbing widths, acquisition and storage options are those of the
repository's configurations; the number of time steps is a tenth or so of a
production record, enough for the wavefield to reach the absorbing layers.

FP64 handles are left out: they exist for verification only.

`exact` states the same problems in plain torch / numpy in 64 bits.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F
from torch.utils.checkpoint import checkpoint

import paper_2605_30541_gb300 as gs
from paper_2605_30541_gb300.autograd import gathers
from paper_2605_30541_gb300 import model as gm

H = 10.0  # grid spacing of every configuration, m
# (f_lo, f_hi, f0) in Hz of the production frequency bands
BANDS = [(3.0, 6.0, 4.50), (3.0, 8.5, 5.75), (3.0, 12.0, 7.50), (3.0, 17.5, 10.25), (3.0, 25.0, 14.00)]


# ------------------------------------------------------------------ the cases

def _forward(name, **kw):
    c = dict(name=name, kind="forward", ndim=2, nz=0, ny=1, nx=0, nt=0, bc="cpml", width=50, free_surface=True,
             shots=1, nrec=0, rec_side=0, snap_every=0, snap_fp16=False)
    c.update(kw)
    return c


def _gradient(name, **kw):
    return _forward(name, kind="gradient", ckpt_fp16=True, **kw)


def listed():
    return [
        # the source wavelet of a production record (8 s at 1 ms), made once per slice and band: the smallest call
        dict(name="wavelet", kind="wavelet", nt=8001, band=0, order=4),
        # a small two-sided model with absorbing layers on every side: a quick look, a smoke run, one FWI forward
        _forward("small_shot", nz=201, nx=201, nt=1000, width=20, free_surface=False, nrec=201),
        # one shot on a field-scale slice with its gather and its FP32 wavefield every 10 steps (training pairs)
        _forward("slice_wavefield", nz=619, nx=1000, nt=1000, nrec=1000, snap_every=10),
        # the production wavefield: sponge, snapshots every 14 steps in scaled FP16, no receivers
        _forward("slice_wavefield_fp16", nz=619, nx=1000, nt=701, bc="sponge", width=60, snap_every=14,
                 snap_fp16=True),
        # the production shot gathers: 64 shots of one slice in one batch, sponge
        dict(_forward("production_gathers", nz=619, nx=1000, nt=560, bc="sponge", width=60, shots=64, nrec=1000),
             kind="batch", slices=1),
        # a dataset chunk: one field-scale slice with many shots and uneven smaller ones in one batch, CPML
        dict(_forward("uneven_slices", nz=619, nx=1000, nt=400, shots=24, nrec=1000), kind="batch", slices=6),
        # one FWI iteration: misfit and velocity gradient of all shots of a survey, FP16 checkpoints
        _gradient("fwi_gradient", nz=201, nx=201, nt=1000, width=20, free_surface=False, shots=16, nrec=201),
        # the solver inside a torch loss: forward, then backward, a few shots on an odd-sized model, FP32 storage
        dict(_gradient("autograd_loss", nz=151, nx=301, nt=600, bc="sponge", width=40, shots=4, nrec=151),
             kind="autograd", ckpt_fp16=False),
        # two shots on a ragged 3D volume that fits in L2 field by field
        _forward("ragged_volume", ndim=3, nz=150, ny=187, nx=233, nt=200, width=20, shots=2, rec_side=31),
        # the field-scale 3D volume: the largest arrays
        _forward("field_volume", ndim=3, nz=619, ny=1000, nx=1000, nt=40, width=30, rec_side=101),
        # a 3D velocity gradient, FP32 storage (what a volume this size has room for)
        dict(_gradient("volume_gradient", ndim=3, nz=100, ny=120, nx=140, nt=120, width=16, rec_side=21),
             ckpt_fp16=False),
        # model building on the device: deposit, squish and fault warps of a 3D volume with its labels
        dict(name="model_volume", kind="model", nz=619, ny=64, nx=1000),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["wavelet", "forward", "forward", "batch", "gradient", "autograd", "volume", "volume_gradient",
                       "model"])
    if kind == "wavelet":
        return dict(kind=kind, nt=_logint(rng, 1001, 16001), band=rng.randrange(5), order=4)
    if kind == "model":
        ny = 1 if rng.random() < 0.3 else _logint(rng, 8, 64)
        return dict(kind=kind, nz=_logint(rng, 100, 619), ny=ny, nx=_logint(rng, 100, 1000))
    bc = rng.choice(["cpml", "sponge"])
    common = dict(bc=bc, free_surface=rng.random() < 0.7)
    if kind == "volume":
        nz, ny, nx = (_logint(rng, 60, 300) for _ in range(3))
        c = _forward("", ndim=3, nz=nz, ny=ny, nx=nx, nt=_logint(rng, 40, 200), width=rng.randint(10, 30),
                     shots=rng.randint(1, 2), rec_side=rng.randint(5, 31), **common)
    elif kind == "volume_gradient":
        nz, ny, nx = (_logint(rng, 40, 140) for _ in range(3))
        c = dict(_gradient("", ndim=3, nz=nz, ny=ny, nx=nx, nt=_logint(rng, 40, 120), width=rng.randint(6, 20),
                           rec_side=rng.randint(5, 21), **common), ckpt_fp16=False)
    else:
        small = kind in ("gradient", "autograd")
        nz, nx = _logint(rng, 101, 301 if small else 619), _logint(rng, 101, 301 if small else 1000)
        common.update(nz=nz, nx=nx, width=rng.randint(15, 60), nrec=rng.randint(min(nx, 51), nx))
        if kind == "forward":
            snaps = rng.random() < 0.5
            c = _forward("", nt=_logint(rng, 200, 1000), shots=rng.choice([1, 1, 2, 4, 8]),
                         snap_every=rng.randint(7, 20) if snaps else 0, snap_fp16=snaps and rng.random() < 0.3,
                         **common)
        elif kind == "batch":
            c = dict(_forward("", nt=_logint(rng, 200, 560), shots=_logint(rng, 2, 32), **common), kind=kind,
                     slices=rng.randint(1, 5))
        elif kind == "gradient":
            c = _gradient("", nt=_logint(rng, 200, 1000), shots=_logint(rng, 1, 16), **common)
            c["ckpt_fp16"] = rng.random() < 0.7
        else:
            c = dict(_gradient("", nt=_logint(rng, 200, 600), shots=_logint(rng, 1, 6), **common), kind=kind,
                     ckpt_fp16=False)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _problem(c, nz=None, nx=None):
    """Problem dict of the package's Simulator."""
    top = 0 if c["free_surface"] else c["width"]
    w = c["width"]
    d3 = c["ndim"] == 3
    nt = c["nt"]
    return dict(ndim=c["ndim"], nz=nz or c["nz"], ny=c["ny"] if d3 else 1, nx=nx or c["nx"], h=H,
                dt=8e-4 if d3 else 1e-3, nt=nt, bc=c["bc"], nb=[top, w, w if d3 else 0, w if d3 else 0, w, w],
                free_surface=int(c["free_surface"]), R=1e-3, f_ref=10.0, snap_every=c["snap_every"], snap_begin=0,
                snap_end=nt if c["snap_every"] else 0)


def _velocity(p, rng, smooth=False):
    """Layered velocity [nz, (ny,) nx], m/s, FP32: layers growing faster with
    depth, one fold, two normal faults; smooth: a depth trend with a low-wavenumber
    perturbation instead (an inversion's starting model). Built slab by slab."""
    dev = _device()
    nz, ny, nx = p["nz"], p["ny"], p["nx"]
    n = 16
    tops = np.sort((np.arange(1, n) + rng.uniform(-0.3, 0.3, n - 1)) * nz / n)
    lv = np.clip(np.sort(np.linspace(1500.0, 4700.0, n) + rng.uniform(-300.0, 300.0, n)), 1500.0, 5000.0)
    tops, lv = torch.tensor(tops, dtype=torch.float32, device=dev), torch.tensor(lv, dtype=torch.float32, device=dev)
    amp, kx, ky, px, py = rng.uniform(0.01, 0.05) * nz, *(2 * math.pi / rng.uniform(200.0, 800.0, 2)), *rng.uniform(
        0.0, 2 * math.pi, 2)
    faults = [(rng.uniform(0.1, 0.9) * nx, math.tan(math.radians(rng.uniform(50.0, 70.0))), rng.uniform(2.0, 20.0),
               rng.uniform(-0.5, 0.5)) for _ in range(2)]
    x = torch.arange(nx, dtype=torch.float32, device=dev)[None, None]
    y = torch.arange(ny, dtype=torch.float32, device=dev)[None, :, None]
    v = torch.empty((nz, ny, nx), dtype=torch.float32, device=dev)
    slab = max(1, (1 << 25) // (ny * nx))
    for z0 in range(0, nz, slab):
        z = torch.arange(z0, min(nz, z0 + slab), dtype=torch.float32, device=dev)[:, None, None]
        wave = torch.sin(kx * x + px) * torch.cos(ky * y + py)
        if smooth:
            v[z0:z0 + slab] = 1600.0 + 1800.0 * z / nz + 80.0 * wave * torch.sin(6.0 * z / nz)
            continue
        zz = z - amp * wave
        for x0, t, throw, sy in faults:
            zz = zz - throw * ((x - x0 + sy * y) * t > z)
        v[z0:z0 + slab] = lv[torch.bucketize(zz.contiguous(), tops)]
    return v if p["ndim"] == 3 else v[:, 0].contiguous()


def _ricker(p, f0):
    t0 = min(1.0 / f0, p["nt"] * p["dt"] / 3.0)
    a = (math.pi * f0 * (np.arange(p["nt"]) * p["dt"] - t0)) ** 2
    return ((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32)


def _geometry(c, p, shots, rng):
    """Sources and receivers in metres: 2D shots along the surface and receivers
    over the full width at 10 or 20 m; 3D shots near the surface and a receiver
    grid 10 m apart around the first one."""
    depth = 10.0 if c["free_surface"] else 20.0
    xm, ym = (p["nx"] - 1) * H, (p["ny"] - 1) * H
    if c["ndim"] == 2:
        s = np.linspace(0.11 * xm, 0.89 * xm, shots) if shots > 1 else np.array([0.5 * xm])
        src = np.stack([s + rng.uniform(-30.0, 30.0), np.full(shots, depth)], axis=1)
        nrec = min(c["nrec"], p["nx"])
        rec = np.stack([np.linspace(0.0, xm, nrec), np.full(nrec, depth)], axis=1) if nrec else np.zeros((0, 2))
        return src, rec
    k = c["rec_side"]
    cx, cy = (rng.uniform(0.35, 0.65) * m for m in (xm, ym))
    src = np.stack([cx + 70.0 * np.arange(shots), cy - 50.0 * np.arange(shots), np.full(shots, depth)], axis=1)
    off = (np.arange(k) - (k - 1) / 2) * H
    Y, X = np.meshgrid(np.clip(cy + off, 0.0, ym), np.clip(cx + off, 0.0, xm), indexing="ij")
    return src, np.stack([X.ravel(), Y.ravel(), np.full(X.size, depth)], axis=1)


def _observed(p, w, src, rec, rng):
    """Recorded data [nshots, nt, nrec]: a direct arrival per trace and a later
    weaker one, FP32 (what a survey's file would hold)."""
    t = torch.arange(p["nt"], dtype=torch.float64, device=_device()) * p["dt"]
    dist = np.linalg.norm(src[:, None] - rec[None], axis=2) + 30.0
    v, f0 = rng.uniform(1600.0, 1900.0), 10.0
    d = torch.zeros((len(src), p["nt"], len(rec)), dtype=torch.float64, device=_device())
    for amp, delay, vel in ((1.0, 0.1, v), (0.3, 0.25, 1.5 * v)):
        tau = torch.tensor(dist / vel + delay, device=d.device)[:, None] - t[None, :, None]
        a = (math.pi * f0 * tau) ** 2
        d += amp * (1.0 - 2.0 * a) * torch.exp(-a) / torch.tensor(np.sqrt(dist), device=d.device)[:, None]
    return (0.3 * d if p["ndim"] == 2 else 0.02 * d).float()


def _slices(c, rng):
    """The members of a batch: the listed grid with its shots, then smaller ones with 8 shots each."""
    out, size = [], np.random.default_rng([c["nz"], c["nx"]])  # the grids belong to the case, not to the seed
    for j in range(c["slices"]):
        nz = c["nz"] if j == 0 else int(size.integers(max(81, c["nz"] // 2), c["nz"] + 1))
        nx = c["nx"] if j == 0 else int(size.integers(max(81, 2 * c["nx"] // 5), c["nx"] + 1))
        p = _problem(c, nz, nx)
        src, rec = _geometry(c, p, c["shots"] if j == 0 else 8, rng)
        out.append((p, _velocity(p, rng), src, rec))
    return out


def _band(c, rng):
    lo, hi, f0 = BANDS[c["band"]]
    k = rng.uniform(0.95, 1.05)
    return lo * k, hi * k, f0 * k


def _model_inputs(c, rng):
    """Drawn fields of one build: a base model with labels, a deposit of six beds
    with texture, a squish displacement and a curved fault."""
    dev = _device()
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    p = dict(ndim=3, nz=nz, ny=ny, nx=nx)
    t = max(8, nz // 5)
    x, y = np.arange(nx)[None], np.arange(ny)[:, None]

    def wave(a, lx, ly):
        q = rng.uniform(0.0, 2 * math.pi, 2)
        return a * np.sin(2 * math.pi * x / lx + q[0]) * np.cos(2 * math.pi * y / ly + q[1])

    def t32(a):
        return torch.tensor(a, dtype=torch.float32, device=dev)

    base = np.linspace(0.15 * t, 0.85 * t, 5) + rng.uniform(-1.0, 1.0, 5)
    g = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 30)))
    lab = torch.randint(1, 12, (nz // 16 + 1,), generator=g, device=dev, dtype=torch.int32)
    lab = lab[torch.arange(nz, device=dev) // 16][:, None, None].expand(nz, ny, nx).contiguous()
    az = math.pi / 2 if ny == 1 else rng.uniform(0.3, 1.2)
    return dict(
        v=_velocity(p, rng), lab=lab,
        deposit=dict(t=t, bounds=t32(np.stack([b + wave(2.0, 90.0, 70.0) for b in base])),
                     vbed=rng.normal(1900.0, 150.0, 6).astype(np.float32), beta=1.0, a_eta=30.0, f_top=0.1, f_base=0.1,
                     eta=torch.randn((t + 40, ny, nx), generator=g, device=dev), offsets=rng.integers(0, 40, 6),
                     label0=20),
        squish=dict(dz=t32(wave(12.0, 400.0, 300.0)), fill=1500.0, fill_label=0),
        fault=dict(cz=rng.uniform(0.4, 0.6) * nz, cy=0.5 * ny, cx=rng.uniform(0.4, 0.6) * nx, azimuth=az,
                   dip=math.radians(rng.uniform(50.0, 70.0)), radius=rng.uniform(300.0, 900.0),
                   slip=rng.uniform(5.0, 15.0), direction=1, d_die=rng.uniform(40.0, 60.0), d_perp=1e9,
                   theta_die=math.radians(40.0), fill=1500.0, fill_label=0))


def _simulator(c, p, vel, src, rec):
    return gs.Simulator(p, vel, max_shots=len(src), max_rec=len(rec), snap_fp16=c["snap_fp16"])


def prepare(case, seed):
    c, rng = case, np.random.default_rng(seed)
    if c["kind"] == "wavelet":
        return dict(kind="wavelet", nt=c["nt"], order=c["order"], band=_band(c, rng))
    if c["kind"] == "model":
        return dict(kind="model", **_model_inputs(c, rng))
    if c["kind"] == "batch":
        entries = []
        for p, vel, src, rec in _slices(c, rng):
            entries.append(dict(sim=_simulator(c, p, vel, src, rec), src=src, rec=rec,
                                wavelet=torch.tensor(_ricker(p, 10.0), device="cuda")))
        return dict(kind="batch", entries=entries)
    p = _problem(c)
    src, rec = _geometry(c, p, c["shots"], rng)
    vel = _velocity(p, rng, smooth=c["kind"] != "forward")
    w = torch.tensor(_ricker(p, 10.0), device="cuda")
    s = dict(kind=c["kind"], sim=_simulator(c, p, vel, src, rec), wavelet=w, src=src, rec=rec)
    if c["kind"] != "forward":
        s.update(vel=vel, d_obs=_observed(p, w, src, rec, rng), ckpt_fp16=c["ckpt_fp16"])
    return s


# ------------------------------------------------------------------ one pass

def run(state):
    s = state
    if s["kind"] == "wavelet":
        lo, hi, f0 = s["band"]
        return gs.bandpass_ricker(s["nt"], 1e-3, f0, lo, hi, order=s["order"])
    if s["kind"] == "model":
        v, lab = gm.deposit(s["v"], s["lab"], **s["deposit"])
        v, lab = gm.squish(v, lab, **s["squish"])
        v, lab = gm.fault(v, lab, **s["fault"])
        return dict(vel=v, labels=lab)
    if s["kind"] == "batch":
        return gs.batch(s["entries"])
    sim, w, src, rec = s["sim"], s["wavelet"], s["src"], s["rec"]
    if s["kind"] == "forward":
        out = sim.forward(w, src, rec, snapshots=True)
        return {k: v for k, v in out.items() if v is not None}
    if s["kind"] == "autograd":
        vel = s["vel"].detach().requires_grad_()
        g = gathers(vel, sim, w, src, rec, ckpt_fp16=s["ckpt_fp16"])
        loss = 0.5 * (g - s["d_obs"]).square().sum()
        loss.backward()
        return dict(gather=g.detach(), loss=loss.detach(), grad=vel.grad)
    grad, misfit = torch.zeros_like(s["vel"]), np.zeros(1)
    gather = torch.empty_like(s["d_obs"])
    gs.sim_adjoint(sim.handle, len(src), w, src, len(rec), rec, s["d_obs"], gather, misfit, int(s["ckpt_fp16"]), grad)
    return dict(gather=gather, misfit=float(misfit[0]), grad=grad)


# ------------------------------------------------------------------ work of one pass

def _cells(c):
    w = c["width"]
    n = (c["nz"] + w * (1 if c["free_surface"] else 2)) * (c["nx"] + 2 * w)
    return n * (c["ny"] + 2 * w) if c["ndim"] == 3 else n


def work(case):
    """Inputs read once and outputs written once; arithmetic of the steps."""
    c = case
    if c["kind"] == "wavelet":  # two passes of `order` second-order sections
        return dict(bytes=4.0 * c["nt"], flops=2.0 * c["order"] * 9 * c["nt"])
    if c["kind"] == "model":  # three warps, velocities and labels; 8 (squish) and up to 8^3 taps near the fault
        n = float(c["nz"] * c["ny"] * c["nx"])
        return dict(bytes=16.0 * n, flops=16.0 * n)
    per = 12 * c["ndim"] + 6  # a second difference per axis and the update
    nint = c["nz"] * c["nx"] * (c["ny"] if c["ndim"] == 3 else 1)
    nrec = c["rec_side"] ** 2 if c["ndim"] == 3 else min(c["nrec"], c["nx"])
    if c["kind"] == "batch":  # the further slices have 3/4 of the depth and 7/10 of the width on average, 8 shots
        more = (c["slices"] - 1) * 8
        updates = c["nt"] * _cells(c) * (c["shots"] + 0.52 * more)
        return dict(bytes=4.0 * nint * (1 + 0.52 * (c["slices"] - 1)) + 4.0 * c["nt"] * nrec * (c["shots"] + 0.7 * more),
                    flops=per * updates)
    updates = float(c["nt"]) * _cells(c) * c["shots"]
    gather = 4.0 * c["shots"] * c["nt"] * nrec
    if c["kind"] == "forward":
        ns = -(-c["nt"] // c["snap_every"]) if c["snap_every"] else 0
        snaps = float(c["shots"]) * ns * nint * (2 if c["snap_fp16"] else 4)
        return dict(bytes=4.0 * nint + gather + snaps, flops=per * updates)
    # forward, recompute with its imaging term, adjoint sweep
    return dict(bytes=8.0 * nint + 2.0 * gather, flops=(3 * per + 6) * updates)


# ------------------------------------------------------------------ the same in 64 bits

_D2 = [-1 / 560, 8 / 315, -1 / 5, 8 / 5, -205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560]
_D1 = [1 / 280, -4 / 105, 1 / 5, -4 / 5, 0.0, 4 / 5, -1 / 5, 4 / 105, -1 / 280]


def _valid(q, axis, w):
    n = q.shape[axis] - 8
    out = q.narrow(axis, 4, n) * w[4]
    for k in (0, 1, 2, 3, 5, 6, 7, 8):
        out.add_(q.narrow(axis, k, n), alpha=w[k])
    return out


class _Stencil(torch.autograd.Function):
    """Nine-point stencil along one axis of an array padded by 4 there."""

    @staticmethod
    def forward(ctx, q, axis, w):
        ctx.axis, ctx.w = axis, w
        return _valid(q, axis, w)

    @staticmethod
    def backward(ctx, g):
        return _valid(_pad(g, ctx.axis, 8), ctx.axis, ctx.w[::-1]), None, None


def _pad(q, axis, n):
    return F.pad(q, (0, 0) * (q.dim() - 1 - axis) + (n, n))


class _Exact:
    """The leapfrog scheme of one grid for all shots at once; fields
    [shots, z, (y,) x] in FP64 with p = 0 outside the grid."""

    def __init__(self, p, vel, vmax):
        self.p, self.nd = p, p["ndim"]
        nb = p["nb"]
        lo, hi = [nb[0], nb[2], nb[4]], [nb[1], nb[3], nb[5]]
        n = [p["nz"], p["ny"], p["nx"]]
        if self.nd == 2:
            lo, hi, n = [lo[0], lo[2]], [hi[0], hi[2]], [n[0], n[2]]
        self.lo, self.n = lo, n
        self.N = [a + b + m for a, b, m in zip(lo, hi, n)]
        dev = vel.device
        v = vel.double()
        for ax in range(self.nd):  # absorbing cells copy the nearest interior cell
            i = torch.clamp(torch.arange(self.N[ax], device=dev) - lo[ax], 0, n[ax] - 1)
            v = v.index_select(ax, i)
        c = (v * (p["dt"] / H)) ** 2
        if p["free_surface"]:  # p = 0 on the top row
            keep = torch.ones(self.N[0], dtype=torch.float64, device=dev)
            keep[0] = 0.0
            c = c * keep.view([-1] + [1] * (self.nd - 1))
        self.c = c
        self.damp, self.mem = None, [None] * self.nd
        for ax in range(self.nd):
            i = np.arange(self.N[ax], dtype=np.float64)
            rho, w = np.zeros(self.N[ax]), np.ones(self.N[ax])
            rho[:lo[ax]], w[:lo[ax]] = (lo[ax] - i[:lo[ax]]) / max(1, lo[ax]), lo[ax]
            k = self.N[ax] - hi[ax]
            rho[k:], w[k:] = (i[k:] - k + 1) / max(1, hi[ax]), hi[ax]
            on = rho > 0
            shape = [1] * (ax + 1) + [-1] + [1] * (self.nd - 1 - ax)
            t = lambda a: torch.tensor(a, device=dev).view(shape)  # noqa: E731
            if p["bc"] == "sponge":
                cd = 1.5 * math.log(1.0 / p["R"]) / w
                eta = 1e-3 * (cd / H) * (rho - np.sin(2 * math.pi * rho) / (2 * math.pi)) * on
                e = t(eta * H * H / (2.0 * p["dt"]))
                self.damp = e if self.damp is None else self.damp + e
            elif on.any():
                d = 3.0 * vmax * math.log(1.0 / p["R"]) / (2.0 * w * H) * rho * rho
                al = math.pi * p["f_ref"] * (1.0 - rho)
                b = np.exp(-(d + al) * p["dt"])
                a = d * (b - 1.0) / np.where(on, d + al, 1.0)
                self.mem[ax] = (t(a * on), t(b * on))

    def points(self, pos):
        """Flat cells and weights of the linear interpolation at positions in metres."""
        order = [self.nd - 1] + ([1] if self.nd == 3 else []) + [0]
        f = np.stack([pos[:, o] / H + l for o, l in zip(order, self.lo)], axis=1)
        r = np.rint(f)
        f = np.where(np.abs(f - r) < 1e-6, r, f)
        i0 = np.floor(f).astype(np.int64)
        t = f - i0
        cell, wt = [], []
        for m in range(1 << self.nd):
            bit = np.array([(m >> (self.nd - 1 - a)) & 1 for a in range(self.nd)])
            wt.append(np.prod(np.where(bit, t, 1.0 - t), axis=1))
            ix = np.minimum(i0 + bit, np.array(self.N) - 1)
            cell.append(np.ravel_multi_index(tuple(ix.T), self.N))
        dev = self.c.device
        return torch.tensor(np.stack(cell, 1), device=dev), torch.tensor(np.stack(wt, 1), device=dev)

    def diff(self, q, ax, w, mirror=False):
        if mirror:  # odd about the top row
            q = torch.cat([-q[:, 1:5].flip(1), q, torch.zeros_like(q[:, :4])], 1)
        else:
            q = _pad(q, ax + 1, 4)
        return _Stencil.apply(q, ax + 1, w)

    def step(self, state, src, wn):
        p, pm, mem = state[0], state[1], list(state[2:])
        rhs, k = src * wn, 0
        for ax in range(self.nd):
            d2 = self.diff(p, ax, _D2, mirror=ax == 0 and self.p["free_surface"])
            rhs = rhs + d2
            if self.mem[ax] is not None:
                a, b = self.mem[ax]
                psi = b * mem[k] + a * self.diff(p, ax, _D1)
                dps = self.diff(psi, ax, _D1)
                zeta = b * mem[k + 1] + a * (d2 + dps)
                mem[k], mem[k + 1] = psi, zeta
                rhs = rhs + dps + zeta
                k += 2
        if self.damp is None:
            new = 2.0 * p - pm + self.c * rhs
        else:
            a = self.c * self.damp
            new = (2.0 * p - (1.0 - a) * pm + self.c * rhs) / (1.0 + a)
        return [new, p] + mem

    def run(self, src_pos, rec_pos, w, segments=False):
        """gathers [shots, nt, nrec], wavefield snapshots of the interior (or None)."""
        p, dev = self.p, self.c.device
        S = len(src_pos)
        cells, wt = self.points(src_pos)
        src = torch.zeros([S] + self.N, dtype=torch.float64, device=dev)
        src.view(S, -1).scatter_add_(1, cells, wt)
        src *= H ** (2 - self.nd)
        rc, rw = self.points(rec_pos) if len(rec_pos) else (None, None)
        zero = torch.zeros_like(src)
        state = [zero, zero] + [zero] * (2 * sum(m is not None for m in self.mem))
        inner = tuple([slice(None)] + [slice(a, a + m) for a, m in zip(self.lo, self.n)])

        def some(n0, n1, *st):
            st, rows, snaps = list(st), [], []
            for n in range(n0, n1):
                if rc is not None:
                    rows.append((st[0].reshape(S, -1)[:, rc] * rw).sum(2))
                if p["snap_every"] and n % p["snap_every"] == 0:
                    snaps.append(st[0][inner].clone())
                st = self.step(st, src, float(w[n]))
            return st, rows, snaps

        rows, snaps, L = [], [], max(1, math.isqrt(p["nt"])) if segments else p["nt"]
        for n0 in range(0, p["nt"], L):
            n1 = min(p["nt"], n0 + L)
            state, r, s = checkpoint(some, n0, n1, *state, use_reentrant=False) if segments else some(n0, n1, *state)
            rows += r
            snaps += s
        return torch.stack(rows, 1) if rows else None, torch.stack(snaps, 1) if snaps else None


def _crop(p, vel, src, rec):
    """A large volume cut to what the wavefield can reach in nt steps (4 cells a
    step, 8 inside an absorbing layer); the rest stays exactly zero."""
    reach = 8 * p["nt"] + 8
    cut, q = [], dict(p, nb=list(p["nb"]))
    for key, o, pair in (("nz", 2, 0), ("ny", 1, 2), ("nx", 0, 4)):
        at = src[:, o] / H
        i0, i1 = max(0, int(at.min()) - reach), min(p[key], int(at.max()) + reach + 2)
        if i0 > 0:
            q["nb"][pair] = 0
        if i1 < p[key]:
            q["nb"][pair + 1] = 0
        if key == "nz" and i0 > 0:
            q["free_surface"] = 0
        q[key] = i1 - i0
        cut.append((i0, i1))
    (z0, z1), (y0, y1), (x0, x1) = cut
    off = np.array([x0, y0, z0]) * H
    return q, vel[z0:z1, y0:y1, x0:x1], src - off, rec - off


def _exact_model(s):
    v = s["v"].double()
    nz, ny, nx = v.shape
    dev = v.device
    z = torch.arange(nz, dtype=torch.float64, device=dev)[:, None, None]
    y = torch.arange(ny, dtype=torch.float64, device=dev)[None, :, None]
    x = torch.arange(nx, dtype=torch.float64, device=dev)[None, None, :]
    d, t = s["deposit"], s["deposit"]["t"]
    bounds, vbed = d["bounds"].double(), torch.tensor(d["vbed"], device=dev).double()
    eta, off = d["eta"].double(), torch.tensor(d["offsets"], device=dev)
    slab = torch.empty_like(v[:t])
    for k in range(t):
        above = bounds < k
        bed = above.sum(0)
        start = torch.where(above, bounds, torch.zeros_like(bounds)).amax(0)
        top, base = min(k / (d["f_top"] * t), 1.0), min((t - k) / (d["f_base"] * t), 1.0)
        zt = torch.clamp(k - start.floor().long() + off[bed], 0, eta.shape[0] - 1)
        slab[k] = vbed.mean() + d["beta"] * k + top * base * (
            vbed[bed] - vbed.mean() + d["a_eta"] * eta.gather(0, zt[None])[0])
    v = torch.cat([slab, v[:nz - t]])

    def taps(q):
        i0 = q.floor()
        u = (q - i0)[..., None] + 3.0 - torch.arange(8, dtype=torch.float64, device=dev)
        w = torch.where(u.abs() < 4.0, torch.sinc(u) * torch.sinc(u / 4.0), torch.zeros_like(u))
        return i0.long() - 3, w / w.sum(-1, keepdim=True)

    q = s["squish"]
    dz = q["dz"].double().reshape(ny, nx)
    i0, w = taps(dz)
    zi = torch.arange(nz, device=dev)[:, None, None]
    out = torch.zeros_like(v)
    for k in range(8):
        out += w[..., k] * v.gather(0, torch.clamp(zi + i0 + k, 0, nz - 1))
    sz = z + dz
    v = torch.where((sz < -1e-6) | (sz >= nz), torch.full_like(v, q["fill"]), out)

    f = s["fault"]
    ca, sa = math.cos(f["azimuth"]), math.sin(f["azimuth"])
    rz, ra = f["radius"] * math.sin(f["dip"]), f["radius"] * math.cos(f["dip"])
    ct = (f["cz"] - rz, f["cy"] - ra * ca, f["cx"] - ra * sa)
    wz, wy, wx = z - ct[0], y - ct[1], x - ct[2]
    u, along = wy * ca + wx * sa, -wy * sa + wx * ca
    r = torch.hypot(u.expand_as(v), wz.expand_as(v))
    th = torch.atan2(wz.expand_as(v), u.expand_as(v))
    rr, rs = (r - f["radius"]).abs() / f["d_die"], along.abs() / f["d_perp"]
    rt = (th - math.atan2(rz, ra)).abs() / f["theta_die"]
    move = (rr < 1) & (rt < 1) & (rs < 1)
    at = move.nonzero(as_tuple=True)
    pick = lambda a: a.expand_as(v)[at]  # noqa: E731
    taper = torch.cos(0.5 * math.pi * rr[at]) * torch.cos(0.5 * math.pi * rt[at]) * torch.cos(0.5 * math.pi * pick(rs))
    chi = torch.where(r[at] >= f["radius"], 1.0, -1.0)
    thn = th[at] - chi * f["direction"] * taper * (f["slip"] / f["radius"])
    fu, al = r[at] * torch.cos(thn), pick(along)
    sz = 2 * pick(z) - (ct[0] + r[at] * torch.sin(thn))
    sy = 2 * pick(y) - (ct[1] + fu * ca - al * sa)
    sx = 2 * pick(x) - (ct[2] + fu * sa + al * ca)
    del r, th, rr, rt, move
    (iz, tz), (iy, ty), (ix, tx) = taps(sz), taps(sy), taps(sx)
    got = torch.zeros_like(sz)
    for a in range(8):
        za = torch.clamp(iz + a, 0, nz - 1) * (ny * nx)
        for b in range(8):
            yb = za + torch.clamp(iy + b, 0, ny - 1) * nx
            wab = tz[:, a] * ty[:, b]
            for k in range(8):
                got += wab * tx[:, k] * v.view(-1)[yb + torch.clamp(ix + k, 0, nx - 1)]
    got = torch.where((sz < -1e-6) | (sz >= nz), torch.full_like(got, f["fill"]), got)
    v = v.clone()
    v[at] = got
    return dict(vel=v, labels=None)


def _exact_wavelet(c, band):
    lo, hi, f0 = band
    nt, N, fs = c["nt"], c["order"], 1000.0
    t = np.arange(nt) / fs - 1.0 / f0
    a = (math.pi * f0 * t) ** 2
    x = (1.0 - 2.0 * a) * np.exp(-a)
    wl, wh = (2.0 * fs * math.tan(math.pi * f / fs) for f in (lo, hi))
    proto = np.exp(1j * math.pi * (2.0 * np.arange(N) + N + 1) / (2.0 * N))
    half = proto * (wh - wl) / 2.0
    root = np.sqrt(half * half - wl * wh)
    poles = np.concatenate([half + root, half - root])
    zp = (2.0 * fs + poles) / (2.0 * fs - poles)
    gain = ((2.0 * fs * (wh - wl)) ** N / np.prod(2.0 * fs - poles)).real
    up = zp[zp.imag > 0]
    sec = [[gain if k == 0 else 1.0, -2.0 * q.real, abs(q) ** 2] for k, q in enumerate(up)]  # g (1 - z^-2) / (..)
    steady, scale = [], 1.0
    for g, _, _ in sec:  # a constant input leaves a band-pass section at zero: the later ones start at rest
        steady.append((scale * -g, scale * -g))
        scale = 0.0
    pad = 3 * (2 * N + 1)
    x = np.concatenate([2 * x[0] - x[pad:0:-1], x, 2 * x[-1] - x[-2:-pad - 2:-1]])
    for _ in range(2):
        for (g, a1, a2), (s1, s2) in zip(sec, steady):
            z1, z2, out = s1 * x[0], s2 * x[0], np.empty_like(x)
            for i, v in enumerate(x.tolist()):
                y = g * v + z1
                z1, z2 = z2 - a1 * y, -g * v - a2 * y
                out[i] = y
            x = out
        x = x[::-1]
    x = x[pad:pad + nt]
    return x / np.linalg.norm(x) * math.sqrt((hi - lo) / 24.0)


def _pow2(m):
    s = torch.exp2(torch.floor(torch.log2(torch.clamp(m, min=2.0 ** -112))) - 14.0)
    return torch.where(m > 0, s, torch.ones_like(m))


def exact(case, seed):
    c, rng = case, np.random.default_rng(seed)
    if c["kind"] == "wavelet":
        return torch.tensor(_exact_wavelet(c, _band(c, rng)).copy())
    if c["kind"] == "model":
        return _exact_model(_model_inputs(c, rng))
    if c["kind"] == "batch":
        out = []
        with torch.no_grad():
            for p, vel, src, rec in _slices(c, rng):
                out.append(_Exact(p, vel, float(vel.max())).run(src, rec, _ricker(p, 10.0))[0])
        return out
    p = _problem(c)
    src, rec = _geometry(c, p, c["shots"], rng)
    vel = _velocity(p, rng, smooth=c["kind"] != "forward")
    vmax, w = float(vel.max()), _ricker(p, 10.0)
    if c["kind"] == "forward":
        if vel.numel() > 1 << 28:
            p, vel, src, rec = _crop(p, vel, src, rec)
        with torch.no_grad():
            g, snaps = _Exact(p, vel, vmax).run(src, rec, w)
        out = {} if g is None else {"gather": g}
        if snaps is not None and c["snap_fp16"]:
            scale = _pow2(snaps.abs().amax((2, 3)))
            out.update(snaps=snaps / scale[:, :, None, None], snap_scale=scale)
        elif snaps is not None:
            out["snaps"] = snaps
        return out
    d = _observed(p, w, src, rec, rng).double()
    v = vel.double().requires_grad_()
    g, _ = _Exact(p, v, vmax).run(src, rec, w, segments=True)
    J = 0.5 * (g - d).square().sum()
    J.backward()
    if c["kind"] == "autograd":
        return dict(gather=g.detach(), loss=J.detach(), grad=v.grad)
    return dict(gather=g.detach(), misfit=float(J.detach()), grad=v.grad)
