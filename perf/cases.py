"""The work this solver is used for, as timed cases.

A case is a dict of plain values.  `kind` says which call of the package it stands for:

  step    advance a batch that is already on the GPU: Solver.step, then the profiles of
          every instance on the host and a checkpoint of the state on the device
  upload  one whole round trip of a coupled program: the state of every instance from
          pinned host memory, steps, profiles back on the host (and the checkpoint)
  steady  the batched parameter sweep: seed every instance (predicted profiles below
          Kn = 1, the free-molecular state above), march to the steady state
  train   one epoch of the warm-start network: minibatches of loss, gradients and Adam
  infer   the warm-start network's forward pass

`mix` says which instances a batch holds: `same` (copies of one problem, each with a state
of its own), `tables` (the 20 half-channel runs of the paper's He / Ar tables), `luo` (its
four low-Mach runs) or `sweep` (instances of mixed sizes drawn from `params_seed`).

Results of FP32 storage are returned as float32: the profiles come out of the library as
float64 numbers that carry FP32 storage's accuracy.
"""
import math

import numpy as np
import torch

import paper_1702_01335_gb300 as lbs
from paper_1702_01335_gb300 import warmstart

TOL = 1e-5           # residual target of the steady case
CHECK_EVERY = 50
PROFILE_ROWS = 8     # n, ux, T, qx, qz, Pxx, Pxz, Pzz
NET_SIZES = (6, 256, 256, 512)


def _step(name, mix, prec, batch, steps, **kw):
    c = dict(kind="step", mix=mix, prec=prec, batch=batch, steps=steps)
    c.update(kw)
    c["name"] = name
    return c


C1 = dict(Qx=4, Qy=4, Qz=4, N_eq=3, Nz=32, A=0.0, half=0, Kn=0.1, u_w=0.1, Pr=1.0, law=0, visc=1.0)
C2 = dict(Qx=8, Qy=8, Qz=16, N_eq=4, Nz=128, A=0.98, half=0, Kn=1.0, u_w=0.5, Pr=2.0 / 3.0, law=0, visc=1.0)
C3 = dict(Qx=16, Qy=4, Qz=64, N_eq=4, Nz=256, A=0.0, half=0, Kn=100.0, u_w=0.05, Pr=2.0 / 3.0, law=0, visc=0.5)


def listed():
    return [
        # the smallest call: one step of one small channel in FP64, as a program that
        # couples to it step by step makes it (launches and latency)
        _step("one_small_f64", "same", "f64", 1, 1, **C1),
        # one channel of ordinary size marched between two looks at its profiles
        _step("one_channel_f32", "same", "f32", 1, 10, **C2),
        # the paper's published tables: 20 small half channels of two sizes, odd Q
        _step("tables_f32", "tables", "f32", 20, 16, reduced=False),
        # the paper's low-Mach runs: the phi / chi model in FP64, half channels of mixed sizes
        _step("low_mach_f64", "luo", "f64", 4, 16),
        # a parameter sweep: 64 channels of mixed Nz, Qx, Qz and viscosity laws
        _step("sweep_f32", "sweep", "f32", 64, 4, params_seed=1702, reduced=False),
        # high-Knudsen channels: many velocities
        _step("high_kn_f32", "same", "f32", 32, 4, **C3),
        # the throughput batch, the largest call
        _step("batch_f32", "same", "f32", 256, 4, **C2),
        # the same problem in FP64
        _step("batch_f64", "same", "f64", 16, 2, **C2),
        # a coupled program's round trip: state from pinned host memory, one step, profiles back
        dict(_step("upload_f32", "same", "f32", 64, 1, **C2), kind="upload"),
        # the batched solve to the steady state from seeds (the sizes the network is trained on)
        dict(kind="steady", mix="sweep", prec="f32", batch=48, params_seed=1704, reduced=False, small=True,
             name="steady_f32"),
        # training the warm-start network: minibatches of 256 over 1000 samples (a ragged last one)
        dict(kind="train", samples=1000, batch=256, hidden=256, outputs=512, name="train"),
        # predicting the profiles of a held-out sweep
        dict(kind="infer", batch=2000, hidden=256, outputs=512, name="infer"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["upload", "steady", "train", "infer"])
    if kind == "train":
        return dict(kind=kind, samples=_log_int(rng, 100, 1000), batch=rng.choice([64, 100, 256]),
                    hidden=rng.choice([64, 128, 200, 256]), outputs=rng.choice([256, 384, 512]))
    if kind == "infer":
        return dict(kind=kind, batch=_log_int(rng, 1, 2000), hidden=rng.choice([64, 128, 200, 256]),
                    outputs=rng.choice([256, 384, 512]))
    if kind == "steady":
        return dict(kind=kind, mix="sweep", prec="f32", batch=rng.randint(4, 40),
                    params_seed=rng.randrange(1 << 20), reduced=False, small=True)
    prec = "f32" if kind == "upload" else rng.choice(["f32", "f32", "f64"])
    if kind == "step" and rng.random() < 0.25:
        return dict(kind=kind, mix="sweep", prec=prec, batch=_log_int(rng, 2, 64 if prec == "f32" else 8),
                    steps=rng.randint(1, 4), params_seed=rng.randrange(1 << 20), reduced=rng.random() < 0.3,
                    small=prec == "f64")
    Qy = rng.choice([0, 0, 2, 3, 4, 5, 7, 8])
    c = dict(kind=kind, mix="same", prec=prec, Qx=rng.randint(2, 16), Qy=Qy, Qz=_log_int(rng, 3, 64),
             N_eq=rng.choice([3, 4, 6]), A=rng.choice([0.0, 0.98]), half=rng.choice([0, 0, 1]),
             Kn=10.0 ** rng.uniform(-1.7, 2.0), u_w=rng.uniform(0.05, 1.0), Pr=rng.choice([1.0, 2.0 / 3.0]),
             law=rng.choice([0, 0, 1]))
    if prec == "f64" and c["Qz"] > 16:
        # the half-range coefficients of order 6 carry 1e-9 of rounding at the largest
        # nodes of such a rule, whatever the order of the operations
        c["N_eq"] = min(c["N_eq"], 4)
    c["visc"] = rng.choice([0.27, 0.52]) if c["law"] else rng.choice([0.5, 0.75, 1.0])
    c["Nz"] = 2 * _log_int(rng, 8, 128) if rng.random() < 0.5 else 2 * _log_int(rng, 8, 128) + 1
    per = c["Nz"] * 2 * c["Qx"] * (Qy if Qy else 2) * c["Qz"]
    most = {"f32": 6e7, "f64": 4e6}[prec] if kind == "step" else 1.6e7
    c["batch"] = max(1, min(256, _log_int(rng, 1, max(1.0, most / per))))
    c["steps"] = rng.randint(1, 4 if prec == "f32" else 2)
    return c


# ---------------------------------------------------------------- the instances ----
def _tables(reduced):
    out = []
    for S in (0.5239, 0.3101):  # Ar, He
        for delta in (0.1, 1.0, 10.0, 20.0, 40.0):
            Qz, dt = (30, 2.5e-4) if delta < 1.0 else (7, 5e-4)
            for u_w in (2.0 ** 0.5, 0.1 * 2.0 ** 0.5):
                out.append(dict(Qx=7, Qy=0 if reduced else 7, Qz=Qz, N_eq=6, Nz=16, A=0.98, half=1,
                                Kn=1.0 / (delta * 2.0 ** 0.5), u_w=u_w, Pr=2.0 / 3.0, law=1, visc=S, dt=dt))
    return out


def _luo():
    runs = ((0.03, 3, 4, 64), (0.1, 6, 7, 32), (1.0, 6, 21, 32), (10.0, 6, 80, 32))
    return [dict(Qx=2, Qy=0, Qz=Qz, N_eq=N, Nz=Nz, A=0.98, half=1, Kn=k / 2.0 ** 0.5, u_w=1e-5, Pr=1.0, law=0,
                 visc=1.0, dt=0.0) for k, N, Qz, Nz in runs]


def _sweep(n, seed, reduced, small):
    rng = np.random.Generator(np.random.PCG64(seed))
    nzs, qxs, qzs = ((32, 48, 64), (4, 6, 8), (4, 8)) if small else \
        ((32, 48, 64, 96, 128, 192, 256, 384, 512), (4, 6, 8, 12, 16), (4, 8, 12, 16, 24, 32, 48))
    out = []
    for b in range(n):
        Kn, u_w = float(10.0 ** rng.uniform(-2.0, 2.0)), float(rng.uniform(0.05, 1.0))
        law, visc = (0, float(rng.uniform(0.5, 1.0))) if b < n // 2 else (1, (0.27, 0.52)[b % 2])
        if small:  # the distribution the network is trained on
            Kn = float(min(max(Kn, 0.05), 20.0))
        out.append(dict(Qx=int(rng.choice(qxs)), Qy=0 if reduced else 4, Qz=int(rng.choice(qzs)), N_eq=4,
                        Nz=int(rng.choice(nzs)), A=0.0, half=0, Kn=Kn, u_w=u_w, Pr=2.0 / 3.0, law=law,
                        visc=visc, dt=0.0))
    return out


def instances(case):
    if case["mix"] == "tables":
        return _tables(case["reduced"])
    if case["mix"] == "luo":
        return _luo()
    if case["mix"] == "sweep":
        return _sweep(case["batch"], case["params_seed"], case["reduced"], case.get("small", False))
    p = {k: case[k] for k in ("Qx", "Qy", "Qz", "N_eq", "Nz", "A", "half", "Kn", "u_w", "Pr", "law", "visc")}
    return [dict(p, dt=0.0) for _ in range(case["batch"])]


def _values(p):
    return p["Nz"] * 2 * p["Qx"] * (p["Qy"] if p["Qy"] else 2) * p["Qz"]


# ---------------------------------------------------------------- the inputs ----
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _waves(gen, z, n, amplitude, lead=()):
    """n smooth random profiles per leading index on the centres z: three harmonics each."""
    a = torch.randn(*lead, n, 3, generator=gen, dtype=torch.float64) * amplitude
    ph = torch.rand(*lead, n, 3, generator=gen, dtype=torch.float64) * 2 * math.pi
    k = torch.arange(1, 4, dtype=torch.float64)
    arg = math.pi * k[:, None] * z + ph[..., None]
    return (a[..., None] * torch.sin(arg) / k[:, None]).sum(-2)


def start_states(case, seed):
    """Each group of alike instances' start state d = f / w - 1, [members, Nz, Q] in the
    storage type: smooth density, velocity and temperature waves about the linear Couette
    profile, linearised in the departure from rest."""
    dtype = torch.float32 if case["prec"] == "f32" else torch.float64
    gen = torch.Generator().manual_seed(seed)
    dev = _device()
    out = []
    for members, p in _groups(instances(case)):
        V = Velocities(p, dev)
        z = V.zc.cpu()
        uw = torch.tensor([q["u_w"] for q in members["p"]], dtype=torch.float64)[:, None]
        size = torch.clamp(uw, max=0.3)  # the departures scale with the wall speed
        w = _waves(gen, z, 4, 0.08, (len(members["p"]),)) * size[:, :, None]
        n, T, uz = w[:, 0], w[:, 1], 0.3 * w[:, 2]
        ux = 0.8 * torch.clamp(uw, max=0.6) * 2 * z + w[:, 3]
        n, T, ux, uz = (t.to(dev)[..., None] for t in (n, T, ux, uz))
        d = n + ux * V.X + uz * V.Z + 0.5 * T * (V.P2 - V.dim)
        if V.reduced:
            d = d + T * V.chi
        out.append((members, p, d.to(dtype)))
    return out


def _groups(ps):
    """Instances alike in sizes and grid: ({"index": [...], "p": [...]}, parameters of the first)."""
    groups = {}
    for b, p in enumerate(ps):
        key = tuple(p[k] for k in ("Qx", "Qy", "Qz", "N_eq", "Nz", "A", "half"))
        groups.setdefault(key, dict(index=[], p=[]))["index"].append(b)
        groups[key]["p"].append(p)
    return [(g, g["p"][0]) for g in groups.values()]


def _packed(case, seed):
    """Every instance's state back to back in instance order, as the library takes it:
    d, then (FP32 storage) the 16-bit rounding residuals, zero.  As bytes."""
    parts = [None] * sum(1 for _ in instances(case))
    for members, _, d in start_states(case, seed):
        for m, b in enumerate(members["index"]):
            parts[b] = d[m].reshape(-1)
    d = torch.cat(parts)
    if case["prec"] == "f64":
        return d.view(torch.uint8)
    return torch.cat([d.view(torch.uint8), torch.zeros(2 * d.numel(), dtype=torch.uint8, device=d.device)])


def _solver(case):
    ps = [lbs.Instance(Qx=p["Qx"], Qy=p["Qy"], Qz=p["Qz"], N_eq=p["N_eq"], Nz=p["Nz"], A=p["A"], half=p["half"],
                       Kn=p["Kn"], u_w=p["u_w"], Pr=p["Pr"], visc_law=p["law"], visc_param=p["visc"], dt=p["dt"])
          for p in instances(case)]
    return lbs.Solver(ps, precision=lbs.LBS_FP32 if case["prec"] == "f32" else lbs.LBS_FP64)


def _seeds(case, seed):
    """Profiles an instance is seeded with ([8, Nz]), None above Kn = 1."""
    gen = torch.Generator().manual_seed(seed)
    out = []
    for p in instances(case):
        z = (torch.arange(p["Nz"], dtype=torch.float64) + 0.5) / p["Nz"] - 0.5
        w = _waves(gen, z, 5, 0.02)
        prof = torch.zeros(PROFILE_ROWS, p["Nz"], dtype=torch.float64)
        prof[0], prof[2] = 1.0 + w[0] - w[0].mean(), 1.0 + 0.1 * p["u_w"] ** 2 + w[1] * p["u_w"] ** 2
        prof[1] = 2 * p["u_w"] * z / (1 + 2 * p["Kn"]) * (1 + w[2])
        prof[3], prof[4] = w[3] * p["u_w"], w[4] * p["u_w"] ** 2
        out.append(prof.numpy() if p["Kn"] < warmstart.WARM_KN_MAX else None)
    return out


def _net_params(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    sizes = (NET_SIZES[0], case["hidden"], case["hidden"], case["outputs"])
    parts = []
    for a, b in zip(sizes[:-1], sizes[1:]):
        parts.append((rng.standard_normal((b, a)) * math.sqrt(2.0 / a)).ravel())
        parts.append(0.1 * rng.standard_normal(b))
    return sizes, np.concatenate(parts).astype(np.float32)


def _net_data(case, seed):
    """Standardised network inputs and targets (a smooth map of the inputs plus noise)."""
    rows = case["samples"] if case["kind"] == "train" else case["batch"]
    gen = torch.Generator().manual_seed(seed + 1)
    x = torch.randn(rows, NET_SIZES[0], generator=gen, dtype=torch.float64)
    M = torch.randn(NET_SIZES[0], case["outputs"], generator=gen, dtype=torch.float64) * 0.4
    t = torch.sin(x @ M) + 0.05 * torch.randn(rows, case["outputs"], generator=gen, dtype=torch.float64)
    return x.float(), t.float()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("train", "infer"):
        sizes, flat = _net_params(case, seed)
        net = warmstart.Mlp(sizes, max_batch=case["batch"])
        net.set_params(flat)
        x, t = _net_data(case, seed)
        return dict(kind=kind, net=net, x=x.to(_device()), t=t.to(_device()), batch=case["batch"])
    s = _solver(case)
    st = dict(kind=kind, solver=s, fp32=case["prec"] == "f32")
    cells = sum(i.Nz for i in s.instances)
    st["profiles"] = torch.zeros(PROFILE_ROWS * cells, dtype=torch.float64).pin_memory()
    if kind == "steady":
        st["seeds"] = _seeds(case, seed)
        return st
    st["steps"] = case["steps"]
    st["checkpoint"] = torch.empty(s.state_bytes(), dtype=torch.uint8, device=_device())
    start = _packed(case, seed)
    if kind == "upload":
        st["start"] = start.cpu().pin_memory()
    else:
        torch.cuda.current_stream().synchronize()
        s.set_state_all_ptr(start.data_ptr(), from_host=False)
    return st


# ---------------------------------------------------------------- one pass ----
def _profiles(st):
    st["solver"].moments_all_ptr(st["profiles"].data_ptr())
    return st["profiles"].to(torch.float32) if st["fp32"] else st["profiles"].clone()


def run(st):
    kind = st["kind"]
    if kind == "infer":
        return st["net"].forward(st["x"])
    if kind == "train":
        net, loss = st["net"], []
        for i in range(0, st["x"].shape[0], st["batch"]):
            loss.append(net.loss_grad(st["x"][i:i + st["batch"]], st["t"][i:i + st["batch"]])[0])
            net.adam(1e-3)
        return dict(loss=np.array(loss, dtype=np.float32), params=net.get_params())
    s = st["solver"]
    if kind == "steady":
        for b, prof in enumerate(st["seeds"]):
            if prof is None:
                s.init_free_molecular(b)
            else:
                s.init_from_profiles(b, prof)
        s.run_to_steady(TOL, max_steps=20000, check_every=CHECK_EVERY, raise_on_fail=False)
        return _profiles(st)
    if kind == "upload":
        s.set_state_all_ptr(st["start"].data_ptr(), from_host=True)
    s.step(st["steps"])
    prof = _profiles(st)
    buf = st["checkpoint"]
    s.get_state_all_ptr(buf.data_ptr(), to_host=False)
    n = buf.numel() // (6 if st["fp32"] else 8)
    # FP64: as normalised populations f / w = 1 + d, the form Solver.populations gives
    state = buf[:4 * n].view(torch.float32) if st["fp32"] else 1.0 + buf.view(torch.float64)
    return dict(profiles=prof, state=state)


# ---------------------------------------------------------------- its work ----
def work(case):
    """Bytes: a step reads the state (d and, FP32, the 16-bit residual) once and writes it
    once; an upload reads it from the host once.  Flops: about 100 per velocity, cell and
    Runge-Kutta stage (the WENO-5 flux 55, the Shakhov target and relaxation 25, the
    moments 20)."""
    if case["kind"] in ("train", "infer"):
        H, O = case["hidden"], case["outputs"]
        rows = case["samples"] if case["kind"] == "train" else case["batch"]
        P = NET_SIZES[0] * H + H * H + H * O + 2 * H + O
        io = 4 * rows * (NET_SIZES[0] + O)
        mac = 2 * rows * (NET_SIZES[0] * H + H * H + H * O)
        if case["kind"] == "infer":
            return dict(bytes=io + 4 * P, flops=mac)
        batches = -(-rows // case["batch"])
        return dict(bytes=io + 24 * P * batches, flops=3 * mac)  # masters and both moments, in and out
    values = sum(_values(p) for p in instances(case))
    size = 6 if case["prec"] == "f32" else 8
    steps = case.get("steps", 500)  # a steady march of these sizes takes some hundred steps
    return dict(bytes=size * values * (2 * steps + (1 if case["kind"] == "upload" else 0)), flops=300 * values * steps)


# ---------------------------------------------------------------- in 64 bits ----
def _gauss(alpha, beta):
    """Nodes and weights of a Gauss rule from its monic recurrence, beta[0] the weight's
    mass: eigenvalues (Golub and Welsch), weights by the Christoffel numbers, which keep
    their relative accuracy where the weights are small."""
    r = np.sqrt(beta)
    x = np.linalg.eigvalsh(np.diag(alpha) + np.diag(r[1:], 1) + np.diag(r[1:], -1))
    p0, p1 = np.zeros_like(x), np.full_like(x, 1.0 / r[0])
    total = p1 * p1
    for k in range(len(alpha) - 1):
        p0, p1 = p1, ((x - alpha[k]) * p1 - (r[k] * p0 if k else 0.0)) / r[k + 1]
        total += p1 * p1
    return x, 1.0 / total


def _half_recurrence(n):
    """alpha, beta of the monic polynomials orthogonal under exp(-p^2/2) / sqrt(2 pi) on
    p > 0, by the Stieltjes procedure on a fine composite Gauss-Legendre rule."""
    t, v = np.polynomial.legendre.leggauss(32)
    edges = np.linspace(0.0, 36.0, 73)
    x = np.concatenate([0.5 * (b - a) * t + 0.5 * (a + b) for a, b in zip(edges[:-1], edges[1:])])
    w = np.tile(0.25 * v, 72) * np.exp(-0.5 * x * x) / math.sqrt(2.0 * math.pi)
    alpha, beta = np.zeros(n), np.zeros(n)
    beta[0] = 0.5
    p0, p1 = np.zeros_like(x), np.full_like(x, math.sqrt(2.0))  # orthonormal
    for k in range(n):
        alpha[k] = np.sum(w * x * p1 * p1)
        q = (x - alpha[k]) * p1 - (math.sqrt(beta[k]) * p0 if k else 0.0)
        h = np.sum(w * q * q)
        if k + 1 < n:
            beta[k + 1] = h
        p0, p1 = p1, q / math.sqrt(h)
    return alpha, beta


_RULES = {}


def _rule(kind, Q):
    if (kind, Q) not in _RULES:
        if kind == "full":
            x, w = _gauss(np.zeros(Q), np.maximum(np.arange(Q, dtype=np.float64), [1.0] + [0.0] * (Q - 1)))
        else:
            x, w = _gauss(*_half_recurrence(Q))
        _RULES[kind, Q] = (x, w)
    return _RULES[kind, Q]


class Velocities:
    """Velocity set and grid of an instance, as float64 tensors: one entry per velocity in
    storage order ((sign of p_z, Qz node, Qx node, Qy node), the last fastest)."""

    def __init__(self, p, dev):
        Qx, Qz = p["Qx"], p["Qz"]
        self.reduced = p["Qy"] == 0
        Qy = 2 if self.reduced else p["Qy"]
        px, wx = _rule("full", Qx)
        py, wy = (np.zeros(2), np.ones(2)) if self.reduced else _rule("full", Qy)
        xi, wz = _rule("half", Qz)
        pz, wz2 = np.concatenate([xi, -xi]), np.concatenate([wz, wz])
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        shape = (2 * Qz, Qx, Qy)
        spread = lambda a, axis: t(a).reshape([-1 if i == axis else 1 for i in range(3)]).expand(shape).reshape(-1)  # noqa: E731
        self.X, self.Y, self.Z = spread(px, 1), spread(py, 2), spread(pz, 0)
        self.w = spread(wx, 1) * spread(wy, 2) * spread(wz2, 0)
        self.chi = spread(np.arange(Qy) == 1, 2) if self.reduced else torch.zeros_like(self.X)
        self.P2 = self.X ** 2 + self.Y ** 2 + self.Z ** 2
        self.dim = 2 if self.reduced else 3
        self.shape, self.px, self.py, self.xi = shape, t(px), t(py), t(xi)
        self.N = min(p["N_eq"], Qx - 1), min(p["N_eq"], Qy - 1), min(p["N_eq"], Qz - 1)
        # cells: interfaces and centres with three ghosts on each side
        Nz, A = p["Nz"], p["A"]
        n, s0 = (2 * Nz, Nz) if p["half"] else (Nz, 0)
        E = math.atanh(A) if A else 0.0
        pos = lambda s: np.tanh(-E + s * 2 * E / n) / (2 * A) if A else -0.5 + s / n  # noqa: E731
        self.dz = t(np.diff(pos(s0 + np.arange(Nz + 1.0))))
        centres = pos(s0 + np.arange(-3, Nz + 3) + 0.5)
        self.zc, self.zg = t(centres[3:-3]), centres


def _full_basis(x, N):
    """He_l(x) / l!, [N + 1, nodes]."""
    H = [torch.ones_like(x), x]
    for k in range(1, N):
        H.append(x * H[k] - k * H[k - 1])
    return torch.stack([H[k] / math.factorial(k) for k in range(N + 1)])


def _half_basis(x, N):
    """pi_l(x) / h_l of the monic half-range polynomials, [N + 1, nodes]."""
    a, b = _half_recurrence(N + 1)
    pi, h = [torch.ones_like(x)], [0.5]
    for k in range(N):
        pi.append((x - a[k]) * pi[k] - (b[k] * pi[k - 1] if k else 0.0))
        h.append(h[k] * b[k + 1])
    return torch.stack([q / s for q, s in zip(pi, h)])


def _full_coeffs(u, T, N):
    a = [torch.ones_like(u), u]
    for k in range(1, N):
        a.append(u * a[k] + k * (T - 1.0) * a[k - 1])
    return torch.stack(a[:N + 1], -1)


def _half_coeffs(u, T, N):
    """int_0^inf of the Maxwellian times pi_l, by the recurrence of its mixed moments."""
    al, be = _half_recurrence(N + 1)
    M = [0.5 * torch.erfc(-u / torch.sqrt(2 * T))]
    M.append(u * M[0] + T * torch.exp(-u * u / (2 * T)) / torch.sqrt(2 * math.pi * T))
    for k in range(1, N):
        M.append(u * M[k] + k * T * M[k - 1])
    out, prev, row = [M[0]], None, M[:N + 1]
    for k in range(N):
        nxt = [row[j + 1] - al[k] * row[j] - (be[k] * prev[j] if k else 0.0) for j in range(len(row) - 1)]
        prev, row = row, nxt
        out.append(row[0])
    return torch.stack(out, -1)


def _lagrange(x, a, b, c):
    return ((x - b) * (x - c) / ((a - b) * (a - c)), (x - a) * (x - c) / ((b - a) * (b - c)),
            (x - a) * (x - b) / ((c - a) * (c - b)))


def _weno(v0, v1, v2, v3, v4):
    s = (13.0 / 12.0 * (v0 - 2 * v1 + v2) ** 2 + 0.25 * (v0 - 4 * v1 + 3 * v2) ** 2,
         13.0 / 12.0 * (v1 - 2 * v2 + v3) ** 2 + 0.25 * (v1 - v3) ** 2,
         13.0 / 12.0 * (v2 - 2 * v3 + v4) ** 2 + 0.25 * (3 * v2 - 4 * v3 + v4) ** 2)
    top = torch.maximum(torch.maximum(s[0], s[1]), s[2])
    top = torch.where(top == 0, torch.ones_like(top), top)
    w = [g / torch.clamp(q / top, min=1e-140) ** 2 for g, q in zip((0.1, 0.6, 0.3), s)]
    c = ((2 * v0 - 7 * v1 + 11 * v2) / 6, (-v1 + 5 * v2 + 2 * v3) / 6, (2 * v2 + 5 * v3 - v4) / 6)
    return (w[0] * c[0] + w[1] * c[1] + w[2] * c[2]) / (w[0] + w[1] + w[2])


class Scheme:
    """The scheme in plain float64 tensors, for one group of alike instances; f is the
    normalised population f / w, [members, Nz, Q]."""

    def __init__(self, ps, dev):
        p = ps[0]
        self.V = V = Velocities(p, dev)
        col = lambda k: torch.tensor([q[k] for q in ps], dtype=torch.float64, device=dev)[:, None]  # noqa: E731
        self.Kn, self.uw, self.Pr, self.visc, self.law = col("Kn"), col("u_w"), col("Pr"), col("visc"), col("law")
        self.half, self.Nz, self.Q = p["half"], p["Nz"], V.X.numel()
        dt = []
        for q in ps:  # an instance without a dt of its own: CFL 0.5, at most half of tau at n = 2, T = 1
            cfl = min(0.5 * float(V.dz.min()) / float(V.xi.max()), 0.25 * q["Kn"])
            dt.append(q["dt"] if q["dt"] > 0 else cfl)
        self.dt = torch.tensor(dt, dtype=torch.float64, device=dev)[:, None, None]
        Nx, Ny, Nq = V.N
        self.Bx, self.By, self.Bz = _full_basis(V.px, max(Nx, 1)), _full_basis(V.py, max(Ny, 1)), _half_basis(V.xi, Nq)
        one, zero = torch.ones_like(self.uw), torch.zeros_like(self.uw)
        self.g_top = self.equilibrium(one, self.uw, zero, zero, one)
        self.g_bot = self.equilibrium(one, -self.uw, zero, zero, one)
        up = V.Z > 0
        self.up = up
        mass = V.w * V.Z * (1 - V.chi)
        self.mass = mass
        self.D_top = (mass * self.g_top)[..., ~up].sum(-1)
        self.D_bot = (mass * self.g_bot)[..., up].sum(-1)
        z = V.zg
        N = self.Nz
        self.ext_top = _lagrange(z[N + 3], z[N + 2], z[N + 1], z[N]), _lagrange(z[N + 4], z[N + 3], z[N + 2], z[N + 1])
        self.ext_bot = _lagrange(z[2], z[3], z[4], z[5]), _lagrange(z[1], z[2], z[3], z[4])

    def equilibrium(self, n, ux, uy, uz, T):
        """n times the product of the truncated expansions, [..., Q], for states [...]."""
        V = self.V
        Nx, Ny, Nq = V.N
        gx = _full_coeffs(ux, T, max(Nx, 1))[..., :Nx + 1] @ self.Bx[:Nx + 1]
        if V.reduced:
            gy = torch.stack([torch.ones_like(T), T], -1)
        else:
            gy = _full_coeffs(uy, T, max(Ny, 1))[..., :Ny + 1] @ self.By[:Ny + 1]
        gz = torch.cat([_half_coeffs(uz, T, max(Nq, 1))[..., :Nq + 1] @ self.Bz,
                        _half_coeffs(-uz, T, max(Nq, 1))[..., :Nq + 1] @ self.Bz], -1)
        g = gz[..., :, None, None] * gx[..., None, :, None] * gy[..., None, None, :]
        return n[..., None] * g.reshape(*g.shape[:-3], -1)

    def macro(self, f):
        V = self.V
        g = f * V.w
        phi = g * (1 - V.chi)
        n = phi.sum(-1)
        ux, uy, uz = ((phi * c).sum(-1) / n for c in (V.X, V.Y, V.Z))
        x, y, z = V.X - ux[..., None], V.Y - uy[..., None], V.Z - uz[..., None]
        c2 = x * x + y * y + z * z if not V.reduced else x * x + z * z
        chi = g * V.chi  # carries the p_y^2 parts of the reduced model
        P = dict(xx=(phi * x * x).sum(-1), yy=(phi * y * y).sum(-1) if not V.reduced else chi.sum(-1),
                 zz=(phi * z * z).sum(-1), xz=(phi * x * z).sum(-1))
        T = (P["xx"] + P["yy"] + P["zz"]) / (3 * n)
        q = [0.5 * (phi * c2 * c + (chi * c if V.reduced else 0.0)).sum(-1) for c in (x, y, z)]
        return n, (ux, uy, uz), T, q, P

    def target(self, m):
        V = self.V
        n, u, T, q, _ = m
        x, y, z = V.X - u[0][..., None], V.Y - u[1][..., None], V.Z - u[2][..., None]
        Tc, qs = T[..., None], [c[..., None] for c in q]
        pre = ((1 - self.Pr) / (n * T * T))[..., None]
        if V.reduced:
            S = pre * ((x * x + z * z) / (5 * Tc) - torch.where(V.chi > 0, 0.4, 0.8)) * (x * qs[0] + z * qs[2])
        else:
            S = pre * ((x * x + y * y + z * z) / (5 * Tc) - 1) * (x * qs[0] + y * qs[1] + z * qs[2])
        zero = torch.zeros_like(u[1])
        return self.equilibrium(n, u[0], zero if V.reduced else u[1], u[2], T) * (1 + S)

    def itau(self, n, T):
        power = n * T ** (1 - self.visc) / self.Kn
        suth = n * (T + self.visc) / (self.Kn * torch.sqrt(T) * (1 + self.visc))
        return torch.where(self.law == 0, power, suth)

    def outgoing(self, f):
        """The ghost values next to each wall of the populations that leave through it."""
        t, b = self.ext_top, self.ext_bot
        a, c, e = f[:, -1], f[:, -2], f[:, -3]
        t0 = t[0][0] * a + t[0][1] * c + t[0][2] * e
        t1 = t[1][0] * t0 + t[1][1] * a + t[1][2] * c
        a, c, e = f[:, 0], f[:, 1], f[:, 2]
        b0 = b[0][0] * a + b[0][1] * c + b[0][2] * e
        b1 = b[1][0] * b0 + b[1][1] * a + b[1][2] * c
        return t0, t1, b0, b1

    def rate(self, f):
        """L[F] of every cell."""
        V, up = self.V, self.up
        t0, t1, b0, b1 = self.outgoing(f)
        out_top = _weno(f[:, -3], f[:, -2], f[:, -1], t0, t1)
        nw_top = -(self.mass * out_top)[:, up].sum(-1, keepdim=True) / self.D_top
        top = torch.stack([torch.where(up, g, nw_top * self.g_top[:, 0]) for g in (t0, t1, t1)], 1)
        if self.half:  # bounce-back on the centre line: p_z and p_x reversed
            m = f[:, :3].reshape(f.shape[0], 3, 2, V.shape[0] // 2, V.shape[1], V.shape[2])
            bot = m.flip(2).flip(4).reshape(f.shape[0], 3, -1).flip(1)
        else:
            out_bot = _weno(f[:, 2], f[:, 1], f[:, 0], b0, b1)
            nw_bot = -(self.mass * out_bot)[:, ~up].sum(-1, keepdim=True) / self.D_bot
            bot = torch.stack([torch.where(up, nw_bot * self.g_bot[:, 0], g) for g in (b1, b1, b0)], 1)
        e = torch.cat([bot, f, top], 1)
        N = self.Nz
        flux = torch.empty(f.shape[0], N + 1, self.Q, dtype=torch.float64, device=f.device)
        v = [e[:, k:k + N + 1] for k in range(6)]
        Q2 = self.Q // 2  # the first half has p_z > 0
        flux[..., :Q2] = _weno(*(a[..., :Q2] for a in v[:5]))
        flux[..., Q2:] = _weno(*(a[..., Q2:] for a in v[:0:-1]))
        m = self.macro(f)
        relax = (f - self.target(m)) * self.itau(m[0], m[2])[..., None]
        return -V.Z * (flux[:, 1:] - flux[:, :-1]) / V.dz[:, None] - relax

    def step(self, f):
        f1 = f + self.dt * self.rate(f)
        f2 = 0.75 * f + 0.25 * (f1 + self.dt * self.rate(f1))
        return f / 3 + 2.0 / 3.0 * (f2 + self.dt * self.rate(f2))


def _exact_steps(case, seed):
    ps = instances(case)
    states, profs = [None] * len(ps), [None] * len(ps)
    for members, _, d in start_states(case, seed):
        part = max(1, int(4e7 // (d.shape[1] * d.shape[2])))
        for k in range(0, d.shape[0], part):
            S = Scheme(members["p"][k:k + part], d.device)
            f = 1.0 + d[k:k + part].double()
            for _ in range(case["steps"]):
                f = S.step(f)
            n, u, T, q, P = S.macro(f)
            rows = torch.stack([n, u[0], T, q[0], q[2], P["xx"], P["xz"], P["zz"]], 1)
            for m, b in enumerate(members["index"][k:k + part]):
                states[b], profs[b] = (f[m] - 1.0).reshape(-1), rows[m].reshape(-1)
    out = dict(profiles=torch.cat(profs).cpu(), state=torch.cat(states))
    if case["prec"] == "f32":
        return {k: v.float() for k, v in out.items()}
    return dict(profiles=out["profiles"], state=1.0 + out["state"])


def _layers(flat, sizes):
    out, o = [], 0
    for a, b in zip(sizes[:-1], sizes[1:]):
        W = flat[o:o + a * b].reshape(b, a)
        o += a * b
        out.append((W, flat[o:o + b]))
        o += b
    return out


def _net(flat, sizes, x):
    h = x
    for k, (W, b) in enumerate(_layers(flat, sizes)):
        h = h @ W.T + b
        if k < 2:
            h = 0.5 * h * (1 + torch.erf(h / math.sqrt(2.0)))
    return h


def _exact_net(case, seed):
    sizes, flat = _net_params(case, seed)
    x, t = (a.double().to(_device()) for a in _net_data(case, seed))
    p = torch.tensor(flat, dtype=torch.float64, device=_device(), requires_grad=True)
    if case["kind"] == "infer":
        return _net(p.detach(), sizes, x)
    opt = torch.optim.Adam([p], lr=1e-3)
    loss = []
    for i in range(0, x.shape[0], case["batch"]):
        opt.zero_grad()
        e = ((_net(p, sizes, x[i:i + case["batch"]]) - t[i:i + case["batch"]]) ** 2).mean()
        e.backward()
        opt.step()
        loss.append(e.item())
    return dict(loss=np.array(loss), params=p.detach())


def exact(case, seed):
    if case["kind"] in ("train", "infer"):
        return _exact_net(case, seed)
    if case["kind"] == "steady":  # some hundred steps of each instance: too long here
        return None
    return _exact_steps(case, seed)
