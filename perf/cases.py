"""Performance cases of the k-space time step: what a user of this package has it do, from the
smallest grids (where launches and latency count) to the largest (where HBM does).

A case is a dict of plain values.  `kind` says which public call a pass makes:

  "step"      kwgb.Simulation.step(steps) and the read-back of every sensor output
  "operator"  kwgb.Simulation.apply_operator on device tensors (Eq. 4a gradient, Eq. 8 terms)
  "focal"     autograd.SimulateFocal: J, dJ/dphases and dJ/damplitudes of a phased array

Grids are powers of two in [8, 1024] per axis, the range the library takes.  The tensor-core forms
are not listed: they are slower than the float32 form at every size, so nobody picks them for speed.
All inputs are float32 and come from the seed alone.  Sensor maps are returned in single precision,
the precision they are computed in.
"""

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1408_4675_gb300 import autograd, kwgb

FREQ = 1e6                 # drive frequency [Hz]
ALPHA_POWER = 1.1          # power-law exponent y of the absorbing media
NP_PER_DB = 100.0 / (20.0 * math.log10(math.e)) * (2.0 * math.pi * FREQ) ** (-ALPHA_POWER)


def listed():
    def step(name, shape, steps, **kw):
        nz, ny, nx = shape
        return dict(name=name, kind="step", nz=nz, ny=ny, nx=nx, steps=steps, **kw)

    tissue = dict(medium="smooth", nonlinear=True, absorbing=True)
    return [
        # the first thing a user runs: a tissue block of the smoke check's size, all maps read back
        step("tissue_32", (32, 32, 32), 100, source="plane", sensor="grid", **tissue),
        # a plane wave down a thin tube, pressure held on a plane, the time series recorded
        # (the shape of the one-dimensional physics checks: periodic sides, layers along z only)
        step("tube_8x8x256", (256, 8, 8), 100, source="dirichlet", sensor="series", medium="water",
             nonlinear=False, absorbing=True),
        # photoacoustic-like run: initial pressure ball in water, linear and lossless, peak map
        step("water_64", (64, 64, 64), 100, source="p0", sensor="grid", medium="water", nonlinear=False,
             absorbing=False),
        # a flat tissue slab: three different axis lengths, force source
        step("slab_32x256x128", (32, 256, 128), 50, source="force", sensor="plane", **tissue),
        # bowl-sized water bath with a perturbed sound speed, nonlinear and lossless (EOS fused, 10 FFTs)
        step("bath_128", (128, 128, 128), 60, source="plane", sensor="plane", medium="sound", nonlinear=True,
             absorbing=False),
        # heterogeneous nonlinear absorbing tissue, tone from a plane: the everyday size
        step("tissue_256", (256, 256, 256), 16, source="plane", sensor="plane", **tissue),
        # the benchmark's workload: layered tissue, focal box with intensity and a plane
        step("hifu_512", (512, 512, 512), 8, source="plane", sensor="intensity", medium="layered", nonlinear=True,
             absorbing=True),
        # the largest grid the library takes
        step("hifu_1024", (1024, 1024, 1024), 3, source="plane", sensor="box", medium="layered", nonlinear=True,
             absorbing=True),
        # treatment planning: focal pressure of a phased array and its gradient, every step kept
        dict(name="focal_128", kind="focal", nz=128, ny=128, nx=128, steps=150, every=150, absorbing=False),
        # the same through an absorbing medium, with checkpoints
        dict(name="focal_64_absorbing", kind="focal", nz=64, ny=64, nx=64, steps=120, every=40, absorbing=True),
        # the staggered gradient alone, on a caller's field
        dict(name="gradient_256", kind="operator", nz=256, ny=256, nx=256, op="gradient"),
        # the dispersion operator of Eq. 8 on a long, uneven grid
        dict(name="eta_64x512x1024", kind="operator", nz=64, ny=512, nx=1024, op="eta"),
    ]


def draw(rng):
    kind = rng.choices(["step", "operator", "focal"], [6, 2, 1])[0]
    if kind == "focal":
        n = [rng.choice([32, 64, 128]) for _ in range(2)]
        steps = rng.randrange(130, 200)
        return dict(kind="focal", nz=64, ny=n[0], nx=n[1], steps=steps, every=rng.choice([steps, 20, 33]),
                    absorbing=rng.random() < 0.5)
    while True:
        e = [rng.randrange(3, 11) for _ in range(3)]
        if 13 <= sum(e) <= 27:
            break
    nz, ny, nx = (1 << v for v in e)
    if kind == "operator":
        return dict(kind="operator", nz=nz, ny=ny, nx=nx, op=rng.choice(["gradient", "backward", "tau", "eta"]))
    medium = rng.choice(["smooth", "smooth", "layered", "sound", "water"])
    most = max(3, min(60, (1 << 28) // (nz * ny * nx)))
    return dict(kind="step", nz=nz, ny=ny, nx=nx, steps=rng.randrange(max(2, most // 2), most + 1), medium=medium,
                nonlinear=rng.random() < 0.7, absorbing=rng.random() < 0.7,
                source=rng.choice(["plane", "plane", "p0", "force", "dirichlet"]),
                sensor=rng.choice(["plane", "box", "intensity", "series"] + (["grid"] if sum(e) <= 20 else [])))


# ------------------------------------------------------------------ inputs
def _smooth(shape, lo, hi, gen, sigma=4.0):
    """Periodic Gaussian-filtered noise scaled into [lo, hi] (float32, on the GPU)."""
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, device="cuda"))
    for a, n in enumerate(shape):
        k = 2.0 * math.pi * (torch.fft.rfftfreq(n, device="cuda") if a == 2 else torch.fft.fftfreq(n, device="cuda"))
        f *= torch.exp(-0.5 * (sigma * k) ** 2).view([-1 if b == a else 1 for b in range(3)])
    f = torch.fft.irfftn(f, s=shape)
    f = (f - f.min()) / (f.max() - f.min())
    return lo + (hi - lo) * f


# typical soft tissue: sound speed, density, absorption in dB/(MHz^y cm), B/A
TISSUE = [(1500.0, 1000.0, 0.0025, 5.0), (1450.0, 950.0, 0.6, 10.0), (1580.0, 1050.0, 1.1, 7.4),
          (1450.0, 950.0, 0.6, 10.0), (1560.0, 1050.0, 1.0, 7.0)]


def _medium(case, shape, gen, rng):
    """c0, rho0, B/A, alpha0: float32 device fields or numbers."""
    kind = case["medium"]
    if kind == "water":
        return [1500.0, 1000.0, 5.0, 5.0 * NP_PER_DB]
    if kind == "sound":
        return [_smooth(shape, 1455.0, 1545.0, gen), 1000.0, 5.0, 0.5 * NP_PER_DB]
    if kind == "smooth":
        return [_smooth(shape, 1450.0, 1650.0, gen), _smooth(shape, 950.0, 1100.0, gen), _smooth(shape, 5.0, 9.0, gen),
                _smooth(shape, 0.3, 1.0, gen) * NP_PER_DB]
    edges = np.sort(rng.uniform(0.3, 0.9, 4)) * shape[0]                 # layered: along z
    layer = np.searchsorted(edges, np.arange(shape[0]))
    out = []
    for j in (0, 1, 3, 2):
        v = torch.tensor([TISSUE[i][j] * (NP_PER_DB if j == 2 else 1.0) for i in layer], device="cuda")
        out.append(v.float().view(-1, 1, 1).expand(shape).contiguous())
    return out


def _run_inputs(case, seed):
    """Everything a run is made of: grid, medium, sources (mode, idx, signals), sensors (idx, records)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    nz, ny, nx = shape
    dx = 0.2e-3
    c_ref = 1650.0
    dt = 0.3 * dx / c_ref
    thin = [n < 16 for n in shape]                                       # periodic, no layer
    pml = [0 if t else min(10, n // 4) for t, n in zip(thin, shape)]
    r = dict(shape=shape, dx=dx, dt=dt, c_ref=c_ref, pml=pml, alpha=2.0, sources=[], sensors=[], p0=None,
             medium=_medium(case, shape, gen, rng), nonlinear=case["nonlinear"], absorbing=case["absorbing"])
    src, phase = case["source"], rng.uniform(-0.5, 0.5)
    t = (np.arange(4000) + 0.5) * dt
    zs = pml[0] + 1
    inner = [np.arange(p, n - p) for p, n in zip(pml, shape)]
    plane = (inner[2][None, :] + nx * (inner[1][:, None] + ny * zs)).ravel().astype(np.int64)
    wave = np.sin(2.0 * math.pi * FREQ * t + phase)
    if thin[0]:                                                          # no layer along z: a burst, or the wave would build up
        wave[int(4.0 / (FREQ * dt)):] = 0.0
    if src == "p0":
        z, y, x = np.meshgrid(*[np.arange(n) for n in shape], indexing="ij", sparse=True)
        c = [n / 2 + rng.uniform(-2, 2) for n in shape]
        s = 4.0 if min(shape) >= 32 else 2.0
        r["p0"] = (2e5 * np.exp(-((z - c[0]) ** 2 + (y - c[1]) ** 2 + (x - c[2]) ** 2) / (2 * s * s))).astype(np.float32)
    elif src == "force":
        r["sources"] = [(kwgb.FORCE_Z, plane, (1e9 * wave).astype(np.float32))]
    elif src == "dirichlet":
        r["sources"] = [(kwgb.DIRICHLET_P, plane, (2e5 * wave).astype(np.float32))]
    else:
        r["sources"] = [(kwgb.ADDITIVE_MASS, plane, (4e5 * wave).astype(np.float32))]
    zc = nz // 2 if src == "p0" else min(nz - 1, zs + 24)                  # where the waves are
    zf, yf, xf = (np.arange(max(0, c - 32), min(n, c + 33)) for c, n in zip((zc, ny // 2, nx // 2), shape))
    box = (xf[None, None, :] + nx * (yf[None, :, None] + ny * zf[:, None, None])).ravel().astype(np.int64)
    xz = (np.arange(nx)[None, :] + nx * (ny // 2 + ny * np.arange(nz)[:, None])).ravel().astype(np.int64)
    kind = case["sensor"]
    if kind == "grid":
        r["sensors"] = [(None, kwgb.P_MAX | kwgb.P_RMS)]
    elif kind == "plane":
        r["sensors"] = [(xz, kwgb.P_MAX | kwgb.P_RMS)]
    elif kind == "box":
        r["sensors"] = [(box, kwgb.P_MAX | kwgb.P_RMS)]
    elif kind == "intensity":
        r["sensors"] = [(box, kwgb.P_MAX | kwgb.P_RMS | kwgb.I_AVG), (xz, kwgb.P_MAX | kwgb.P_RMS)]
    else:
        r["sensors"] = [(xz.reshape(nz, nx)[:, nx // 2 - 4:nx // 2 + 4].ravel(), kwgb.P_SERIES | kwgb.P_MIN)]
    return r


RECORDS = (kwgb.P_MAX, kwgb.P_RMS, kwgb.I_AVG, kwgb.P_MIN, kwgb.P_SERIES)


def _focal_inputs(case, seed):
    """A planar 8 x 8 phased array facing a focal box 28 cells away (the waves arrive well within the run)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    nz, ny, nx = shape
    dx, pml = 0.15e-3, 8
    medium = [_smooth(shape, 1455.0, 1545.0, gen), 1000.0, 5.0,
              _smooth(shape, 0.3, 1.0, gen) * NP_PER_DB if case["absorbing"] else 0.0]
    by, bx = (np.array_split(np.arange(pml, n - pml), 8) for n in (ny, nx))
    zs = pml + 1
    elements = [(bx[j][None, :] + nx * (by[i][:, None] + ny * zs)).ravel().astype(np.int64) for i in range(8) for j in range(8)]
    zf, yf, xf = (np.arange(c - 2, c + 3) for c in (zs + 28, ny // 2, nx // 2))
    focal = (xf[None, None, :] + nx * (yf[None, :, None] + ny * zf[:, None, None])).ravel().astype(np.int64)
    c_ref = 1550.0
    return dict(shape=shape, dx=dx, dt=0.3 * dx / c_ref, c_ref=c_ref, pml=[pml] * 3, alpha=2.0, medium=medium,
                nonlinear=True, absorbing=case["absorbing"], elements=elements, focal=focal,
                phases=rng.uniform(-0.6, 0.6, 64).astype(np.float32),
                amps=rng.uniform(0.8e5, 1.2e5, 64).astype(np.float32))


def _flags(r):
    return (kwgb.NONLINEAR if r["nonlinear"] else 0) | (kwgb.ABSORBING if r["absorbing"] else 0)


# ------------------------------------------------------------------ the measured interface
def prepare(case, seed):
    if case["kind"] == "focal":
        r = _focal_inputs(case, seed)
        c0, rho0, bona, alpha0 = r["medium"]
        cfg = dict(shape=r["shape"], d=(r["dx"],) * 3, dt=r["dt"], c_ref=r["c_ref"], pml_size=r["pml"],
                   pml_alpha=(r["alpha"],) * 3, flags=_flags(r), alpha_power=ALPHA_POWER, c0=c0, rho0=rho0, bona=bona,
                   alpha0=alpha0, elements=r["elements"], focal=r["focal"], freq=FREQ, n_steps=case["steps"])
        problem = autograd.FocalProblem(cfg, case["steps"], case["every"])
        return dict(kind="focal", problem=problem, phases=torch.from_numpy(r["phases"]).requires_grad_(True),
                    amps=torch.from_numpy(r["amps"]).requires_grad_(True))
    if case["kind"] == "operator":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        shape = (case["nz"], case["ny"], case["nx"])
        sim = kwgb.Simulation(shape, (2e-4,) * 3, 0.3 * 2e-4 / 1650.0, 1650.0, flags=kwgb.ABSORBING,
                              alpha_power=ALPHA_POWER)
        sim.set_medium(1500.0, 1000.0, 5.0, 1e-9)
        field = _smooth(shape, -1.0, 1.0, gen, sigma=1.0)
        n = 3 if case["op"] in ("gradient", "backward") else 1
        return dict(kind="operator", sim=sim, field=field, outs=[torch.empty_like(field) for _ in range(n)],
                    op={"gradient": kwgb.OP_GRAD_FWD, "backward": kwgb.OP_GRAD_BWD, "tau": kwgb.OP_ABS_TAU,
                        "eta": kwgb.OP_ABS_ETA}[case["op"]])
    r = _run_inputs(case, seed)
    sim = kwgb.Simulation(r["shape"], (r["dx"],) * 3, r["dt"], r["c_ref"], r["pml"][::-1], (r["alpha"],) * 3, _flags(r),
                          ALPHA_POWER)
    sim.set_medium(*r["medium"])
    if r["p0"] is not None:
        sim.set_initial_pressure(r["p0"])
    for mode, idx, signal in r["sources"]:
        sim.add_source(idx, signal, mode)
    reads = []
    for idx, record in r["sensors"]:
        sid = sim.add_sensor(idx, record)
        if record & kwgb.P_SERIES:
            sim.set_series_capacity(sid, case["steps"])
        reads += [(sid, w) for w in RECORDS if record & w]
    return dict(kind="step", sim=sim, steps=case["steps"], reads=reads)


def run(state):
    if state["kind"] == "focal":
        ph, am = state["phases"], state["amps"]
        ph.grad = am.grad = None
        J = autograd.SimulateFocal.apply(ph, am, state["problem"])
        J.backward()
        return {"J": J.detach(), "phases": ph.grad, "amps": am.grad}
    sim = state["sim"]
    stream = torch.cuda.current_stream()
    if state["kind"] == "operator":
        sim.apply_operator(state["op"], state["field"], state["outs"], stream)
        return state["outs"]
    sim.step(state["steps"], stream)
    return [sim.read(sid, which).astype(np.float32) for sid, which in state["reads"]]


def work(case):
    """Bytes: the state (u, rho and p, read and written) and the medium's fields once per step; the
    reverse pass reads the density fields of a step and reads and writes the seven adjoint fields.  FFTs
    at 2.5 N log2 N (real data) and about 60 operations a point for the updates."""
    n = case["nz"] * case["ny"] * case["nx"]
    fft = 2.5 * n * math.log2(n)
    if case["kind"] == "operator":
        outs = 3 if case["op"] in ("gradient", "backward") else 1
        return {"bytes": 4.0 * n * (1 + outs), "flops": fft * (1 + outs) + 10.0 * n}
    ffts = 14 if case["absorbing"] else 10
    if case["kind"] == "focal":
        fields = 14 + 1 + int(case["absorbing"])
        return {"bytes": 4.0 * n * case["steps"] * (fields + 7 + 14 + 7 + 1), "flops": 2.0 * case["steps"] * (fft * ffts + 60.0 * n)}
    fields = 14 + {"water": 0, "sound": 1, "smooth": 2, "layered": 2}[case["medium"]]
    if case["medium"] in ("smooth", "layered"):
        fields += int(case["nonlinear"]) + int(case["absorbing"])
    sensors = (4 + 8 + 4 + 8) if case["sensor"] == "grid" else 0          # peak (4 bytes) and sum of squares (8), in and out
    return {"bytes": float(n * case["steps"] * (4 * fields + sensors)), "flops": case["steps"] * (fft * ffts + 60.0 * n)}


# ------------------------------------------------------------------ 64-bit values
class _Step64:
    """The time step in float64 with torch.fft (Eqs. 4a-4d, 6 and 8 with the split-field layer)."""

    def __init__(self, r):
        f64 = dict(dtype=torch.float64, device="cuda")
        self.r, shape, dx, dt = r, r["shape"], r["dx"], r["dt"]
        self.s, self.dt = shape, dt
        self.c0, self.rho0, self.ba, self.a0 = [v.double() if torch.is_tensor(v) else torch.tensor(np.float32(v), **f64)
                                                for v in r["medium"]]
        k2, self.df = 0.0, []
        for a, n in enumerate(shape):
            k = 2.0 * math.pi / dx * (torch.fft.rfftfreq(n, **f64) if a == 2 else torch.fft.fftfreq(n, **f64))
            k = k.view([-1 if b == a else 1 for b in range(3)])
            d = 1j * k * torch.exp(0.5j * k * dx)
            half = (k.abs() * dx - math.pi).abs() < 1e-6
            self.df.append(torch.where(half, d.real.to(d.dtype), d))
            k2 = k2 + k * k
        k = torch.sqrt(k2)
        h = r["c_ref"] * dt / 2.0 * k
        self.kappa = torch.where(h > 0, torch.sin(h) / h.clamp(min=1e-300), torch.ones_like(h))
        y = ALPHA_POWER
        if r["absorbing"] or "op" in r:
            safe = torch.where(k > 0, k, torch.ones_like(k))
            self.k1, self.k2 = (torch.where(k > 0, safe ** e, torch.zeros_like(k)) for e in (y - 2.0, y - 1.0))
        self.f, self.fs = [], []
        for a, n in enumerate(shape):
            for off, out in ((0.0, self.f), (0.5, self.fs)):
                s, p = torch.arange(n, **f64) + off, r["pml"][a]
                depth = torch.clamp(torch.maximum(p - s, s - (n - 1 - p)), min=0.0) / max(p, 1)
                v = torch.exp(-r["alpha"] * r["c_ref"] / dx * depth ** 4 * dt / 2.0) if p > 0 else torch.ones_like(s)
                out.append(v.view([-1 if b == a else 1 for b in range(3)]))
        zero = torch.zeros(shape, **f64)
        self.u, self.rho, self.p = [zero] * 3, [zero] * 3, zero
        if r.get("p0") is not None:
            self.p = torch.from_numpy(r["p0"]).cuda().double()
            self.rho = [self.p / (3.0 * self.c0 ** 2)] * 3
            self.u = [0.5 * dt * g / self.staggered(a) for a, g in enumerate(self.grad(self.p))]
        self.tau = -2.0 * self.a0 * self.c0 ** (y - 1.0)
        self.eta = 2.0 * self.a0 * self.c0 ** y * math.tan(math.pi * y / 2.0)

    def staggered(self, a):
        return self.rho0 if self.rho0.dim() == 0 else 0.5 * (self.rho0 + torch.roll(self.rho0, -1, a))

    def inv(self, f):
        return torch.fft.irfftn(f, s=self.s)

    def grad(self, p):
        q = torch.fft.rfftn(p) * self.kappa
        return [self.inv(self.df[a] * q) for a in range(3)]

    def velocity(self, force=None):
        out = []
        for a, g in enumerate(self.grad(self.p)):
            v = self.fs[a] * (self.fs[a] * self.u[a] - self.dt * g / self.staggered(a))
            if force is not None and force[0] == a:
                w = torch.zeros(self.s, dtype=torch.float64, device="cuda")
                w.view(-1)[force[1]] = self.dt * force[2]
                v = v + w / self.staggered(a)
            out.append(v)
        return out

    def step(self, force=None, mass=None, held=None):
        """force (axis, idx, value), mass: field added to every split density, held (idx, value)."""
        self.u = self.velocity(force)
        total, rho = 0.0, []
        for a in range(3):
            d = self.inv(torch.conj(-self.df[a]) * self.kappa * torch.fft.rfftn(self.u[a]))
            total = total + self.rho0 * d
            v = self.f[a] * (self.f[a] * self.rho[a] - self.dt * self.rho0 * d)
            if self.r["nonlinear"]:
                v = v / (1.0 + 2.0 * self.dt * d)
            v = v if mass is None else v + mass
            if held is not None:
                v = v.clone()
                c = self.c0 if self.c0.dim() == 0 else self.c0.view(-1)[held[0]]
                v.view(-1)[held[0]] = held[1] / (3.0 * c * c)
            rho.append(v)
        self.rho, s = rho, rho[0] + rho[1] + rho[2]
        p = s + (0.5 * self.ba * s * s / self.rho0 if self.r["nonlinear"] else 0.0)
        if self.r["absorbing"]:
            p = p + self.tau * self.inv(self.k1 * torch.fft.rfftn(total)) - self.eta * self.inv(self.k2 * torch.fft.rfftn(s))
        p = self.c0 ** 2 * p
        if held is not None:
            p = p.clone()
            p.view(-1)[held[0]] = held[1]
        self.p = p

    def mean_u(self, idx):
        return torch.stack([(0.5 * (v + torch.roll(v, 1, a))).view(-1)[idx] for a, v in ((2, self.u[2]), (1, self.u[1]), (0, self.u[0]))])


def _exact_operator(case, seed):
    st = prepare(case, seed)
    field = st["field"].double()
    st["sim"].close()
    e = _Step64(dict(shape=tuple(field.shape), dx=2e-4, dt=0.3 * 2e-4 / 1650.0, c_ref=1650.0, pml=[0] * 3, alpha=0.0, absorbing=True,
                     nonlinear=False, medium=[1500.0, 1000.0, 5.0, 1e-9]))
    f = torch.fft.rfftn(field)
    if case["op"] in ("tau", "eta"):
        return [e.inv(f * (e.k1 if case["op"] == "tau" else e.k2))]
    d = [e.df[a] if case["op"] == "gradient" else torch.conj(-e.df[a]) for a in (2, 1, 0)]
    return [e.inv(f * e.kappa * v) for v in d]


def _exact_focal(case, seed):
    r = _focal_inputs(case, seed)
    e = _Step64(r)
    ph, am = (torch.from_numpy(r[k]).double().cuda().requires_grad_(True) for k in ("phases", "amps"))
    which = torch.full((int(np.prod(r["shape"])),), 64, device="cuda")
    for i, idx in enumerate(r["elements"]):
        which[torch.from_numpy(idx).cuda()] = i
    which = which.view(r["shape"])
    focal, J = torch.from_numpy(r["focal"]).cuda(), 0.0

    def advance(q, uz, uy, ux, rz, ry, rx, p):
        e.u, e.rho, e.p = [uz, uy, ux], [rz, ry, rx], p
        s = torch.cat([q, torch.zeros_like(q[:1])])
        e.step(mass=s[which] * (e.dt * 2.0 / (3.0 * r["dx"])) / e.c0)
        return (*e.u, *e.rho, e.p)

    v = (*e.u, *e.rho, e.p)
    for n in range(case["steps"]):
        q = am * torch.sin(2.0 * math.pi * FREQ * (n + 0.5) * r["dt"] + ph)
        v = checkpoint(advance, q, *v, use_reentrant=False)
        J = J + v[6].view(-1)[focal].abs().sum()
    J = J / (len(focal) * case["steps"])
    J.backward()
    return {"J": J.detach(), "phases": ph.grad, "amps": am.grad}


def exact(case, seed):
    n = case["nz"] * case["ny"] * case["nx"]
    if n > 1 << 27:                     # 64-bit fields of the largest grid do not fit the card
        return None
    if case["kind"] == "operator":
        return _exact_operator(case, seed)
    if case["kind"] == "focal":
        return _exact_focal(case, seed)
    r = _run_inputs(case, seed)
    e = _Step64(r)
    src = [(m, torch.from_numpy(i).cuda(), s) for m, i, s in r["sources"]]
    sensors = [(None if i is None else torch.from_numpy(i).cuda(), rec) for i, rec in r["sensors"]]
    acc = [dict() for _ in sensors]
    for n in range(case["steps"] + 1):
        last = n == case["steps"]
        force = mass = held = None
        for mode, idx, sig in src:
            v = float(sig[n])
            if mode == kwgb.FORCE_Z:
                force = (0, idx, v)
            elif mode == kwgb.DIRICHLET_P:
                held = (idx, v)
            else:
                w = torch.zeros(r["shape"], dtype=torch.float64, device="cuda")
                w.view(-1)[idx] = v * e.dt * 2.0 / (3.0 * r["dx"])
                mass = w / e.c0
        means = [e.mean_u(i) if rec & kwgb.I_AVG else None for i, rec in sensors]
        pold = e.p
        if last:
            if not any(rec & kwgb.I_AVG for _, rec in sensors):
                break
            e.u = e.velocity(force)
        else:
            e.step(force, mass, held)
        for (idx, rec), a, before in zip(sensors, acc, means):
            if rec & kwgb.I_AVG and n > 0:
                a["i"] = a.get("i", 0.0) + pold.view(-1)[idx] * 0.5 * (before + e.mean_u(idx))
            if last:
                continue
            p = e.p.view(-1) if idx is None else e.p.view(-1)[idx]
            a["max"] = torch.maximum(a["max"], p) if "max" in a else p
            a["min"] = torch.minimum(a["min"], p) if "min" in a else p
            a["sq"] = a.get("sq", 0.0) + p * p
            if rec & kwgb.P_SERIES:
                a.setdefault("series", []).append(p)
    out = []
    for (idx, rec), a in zip(sensors, acc):
        for w in RECORDS:
            if rec & w:
                v = {kwgb.P_MAX: lambda: a["max"], kwgb.P_MIN: lambda: a["min"], kwgb.P_RMS: lambda: torch.sqrt(a["sq"] / case["steps"]),
                     kwgb.I_AVG: lambda: a["i"] / case["steps"], kwgb.P_SERIES: lambda: torch.stack(a["series"])}[w]()
                out.append(v.cpu().numpy())
    return out
