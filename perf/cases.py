"""Workloads of the framework as its users run them, for timing and comparison.

A case is a dict of plain values.  ``prepare`` builds what a program has in
hand before the call (windows with a loaded particle, networks, marker
arrays), ``run`` makes one pass through the public entry points and returns
whole outputs, ``work`` counts what a pass cannot do without, and ``exact``
gives the same outputs in 64 bits from the reference solver at the end of this
file (plain torch, nothing of the library).

Kinds of case:
  settle    a particle in a prepared window: step(n), then the particle state
            and the density and velocity of every cell (a monitoring interval
            of a settling run)
  monitor   the same, but one step at a time with the particle state read
            after each (a program that logs or couples every step)
  session   a whole short run from host arrays: context, initial fields,
            surface, steps, state, fields
  ensemble  many settling runs advanced as one batch
  fluid     the collide+stream alone (no particle): channel, shear, periodic
  train     one epoch of the force/torque network on logged pairs
  infer     the network's predictions for a set of rows
  spread    the standalone spreading operator
"""
import functools
import math

import numpy as np
import torch

from paper_2408_15115_gb300 import configs
from paper_2408_15115_gb300 import inputs as I
from paper_2408_15115_gb300 import surrogate
from paper_2408_15115_gb300 import turret as T

DEV = "cuda:0"
STATE_KEYS = ("r", "d", "v", "w", "F", "T", "L", "Fp", "origin")
PARTICLE = dict(force_eval=0, predictor="paper", sround=0)
TURRET_BC = dict(bc_x=0, bc_y=0, bc_bottom=1, bc_top=2, slide=1)   # the settling window of the paper
CLOSED_BC = dict(bc_x=1, bc_y=1, bc_bottom=1, bc_top=1, slide=0)   # a closed box


def _window(kind, name, nx, ny, nz, storage, steps, nu, re, d, shape, **kw):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, nu=nu, re=re, d=d, shape=shape,
             kappa=2.0, sponge=int(round(0.08 * nz)), anchor=0.25, **PARTICLE, **TURRET_BC)
    c.update(kw)
    return c


def listed():
    return [
        # a first look at a particle: a short closed-box run from host arrays to results
        _window("session", "session_sphere_32x32x64", 32, 32, 64, "f32", 100, 0.05, 0.2, 8.0, "sphere", kappa=2.5,
                sponge=0, **CLOSED_BC),
        # a controller or logger that reads the body after every step of a small window
        _window("monitor", "monitor_sphere_64x64x64", 64, 64, 64, "f32", 16, 0.02, 10.0, 10.0, "sphere"),
        # the paper's settling set-up at the size of one particle study
        _window("settle", "settle_prolate_96x96x192_f32", 96, 96, 192, "f32", 24, 0.02, 10.0, 10.08, "prolate", sponge=15),
        # a window whose sides are no multiples of anything, with the predictor and warm-started cycles
        _window("settle", "settle_ragged_93x70x151_f16", 93, 70, 151, "f16", 24, 0.02, 20.0, 12.0, "irregular",
                predictor="linear_warm"),
        # the 16-bit storages on a production window
        _window("settle", "settle_irregular_192x192x384_f16", 192, 192, 384, "f16", 16, 0.0024, 200.0, 24.0, "irregular", sponge=30),
        _window("settle", "settle_irregular_192x192x384_bf16_sr", 192, 192, 384, "bf16", 16, 0.0024, 200.0, 24.0, "irregular",
                sponge=30, sround=1),
        # the largest single run: a 33.6-million-cell window at Re ~ 1000
        _window("settle", "settle_irregular_256x256x512_f32", 256, 256, 512, "f32", 16, 0.00064, 1000.0, 32.0, "irregular", sponge=40),
        # a parameter sweep: 32 different particles at once, FP32 and FP16 windows mixed
        dict(name="ensemble_32_mixed", kind="ensemble", runs=32, pick=4, storage="alternate", steps=8, d_max=24.0, predictor="paper"),
        # the fluid alone between two sliding walls, before a particle is put in
        dict(name="shear_75x101x143_f32", kind="fluid", nx=75, ny=101, nz=143, storage="f32", steps=24, nu=0.03, bc_x=0, bc_y=0,
             bc_bottom=3, bc_top=3, sponge=0, sround=0),
        # training the force/torque network on a collected trajectory set, and using it on the set
        dict(name="train_16384_batch_4096", kind="train", rows=16384, batch=4096, precision="bf16"),
        dict(name="infer_15967", kind="infer", rows=15967, precision="bf16"),
        # the spreading operator called by another code on its own grid
        dict(name="spread_6252_on_96x80x72", kind="spread", nx=96, ny=80, nz=72, freq=25, radius=16.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["settle", "settle", "settle", "monitor", "session", "ensemble", "fluid", "train", "infer", "spread"])
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    if kind in ("settle", "monitor", "session"):
        small = kind != "settle"
        d = math.exp(rng.uniform(math.log(6.0), math.log(12.0 if small else 32.0)))
        base = max(32, int(3.5 * d))
        top = 72 if small else 256
        nx = min(top, _log_int(rng, base, max(base + 1, top)))
        ny = min(top, max(base, int(nx * rng.uniform(0.75, 1.25))))
        nz = min(144 if small else 512, max(64, int(max(nx, ny) * rng.uniform(1.3, 2.0))))
        if rng.random() < 0.5:  # sides that the fast layouts like, as users pick them
            nx, ny, nz = min(top, -(-nx // 32) * 32), -(-ny // 4) * 4, -(-nz // 4) * 4
        closed = kind == "session" and rng.random() < 0.5
        re = math.exp(rng.uniform(math.log(0.5), math.log(1.0 + 0.9 * d * d)))
        kw = dict(CLOSED_BC, sponge=0) if closed else {}
        kw["force_eval"] = rng.choice([0, 0, 0, 1])
        kw["predictor"] = rng.choice(["paper", "paper", "linear", "linear_warm"])
        kw["sround"] = rng.choice([0, 1]) if storage == "bf16" else 0
        nu = min(0.1, 0.02 * d / re)
        c = _window(kind, "", nx, ny, nz, storage, rng.choice([50, 100]) if kind == "session" else rng.randint(1, 16),
                    nu, re, round(d, 2), rng.choice(["sphere", "oblate", "prolate", "irregular"]), **kw)
    elif kind == "ensemble":
        c = dict(kind=kind, runs=rng.randint(2, 28), pick=rng.randint(0, 1000), storage=rng.choice(["alternate", "f32", "f16"]),
                 steps=rng.randint(1, 8), d_max=rng.choice([14.0, 20.0]), predictor=rng.choice(["paper", "linear_warm"]))
    elif kind == "fluid":
        nx, ny, nz = (_log_int(rng, 17, 200) for _ in range(3))
        walls = rng.choice([(0, 0, 0, 0), (0, 0, 3, 3), (1, 1, 1, 1), (0, 0, 1, 2), (1, 0, 1, 2)])
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, steps=rng.randint(1, 32), nu=rng.choice([0.003, 0.03, 0.1]),
                 bc_x=walls[0], bc_y=walls[1], bc_bottom=walls[2], bc_top=walls[3], sponge=rng.choice([0, nz // 8]) if walls[3] == 2 else 0,
                 sround=rng.choice([0, 1]) if storage == "bf16" else 0)
    elif kind == "train":
        batch = rng.choice([256, 1000, 1024, 4096, 5000])
        c = dict(kind=kind, rows=batch * rng.randint(1, 6) + rng.randint(0, 200), batch=batch, precision=rng.choice(["bf16", "bf16", "fp32"]))
    elif kind == "infer":
        c = dict(kind=kind, rows=_log_int(rng, 1, 40000), precision=rng.choice(["bf16", "bf16", "fp32"]))
    else:
        freq = rng.randint(4, 25)
        r = round(0.62 * freq * rng.uniform(0.8, 1.2), 2)
        lo = int(2 * r) + 8
        c = dict(kind=kind, nx=_log_int(rng, lo, 128), ny=_log_int(rng, lo, 128), nz=_log_int(rng, lo, 128), freq=freq, radius=r)
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# Inputs

@functools.lru_cache(maxsize=64)
def _mesh(shape, d):
    """Surface of volume-equivalent diameter d with markers about 0.9 cells apart."""
    R = 0.5 * d
    freq = lambda r: max(4, int(math.ceil(1.2 * r / 0.9)))  # noqa: E731
    if shape == "sphere":
        return I.sphere(freq(R), d)
    if shape == "oblate":
        a = R * 2.0 ** (1.0 / 3.0)
        return I.ellipsoid(freq(a), (a, a, 0.5 * a))
    if shape == "prolate":
        b = R / 2.0 ** (1.0 / 3.0)
        return I.ellipsoid(freq(2.0 * b), (2.0 * b, b, b))
    return I.sh_particle(freq(1.2 * R), d, seed=3)


@functools.lru_cache(maxsize=8)
def _ensemble(runs, pick, storage, d_max):
    return configs.ensemble(runs, seed=pick, storage=storage, d_range=(8.0, d_max))


def _fields(nz, ny, nx, seed):
    """Smooth seeded density and velocity (as host arrays): a few Fourier modes per component, |u| <= 0.01, |rho - 1| <= 1e-3."""
    rng = np.random.default_rng([seed, 1])
    ax = [torch.arange(n, device=DEV, dtype=torch.float64) / n for n in (nz, ny, nx)]
    rho, u = torch.empty((nz, ny, nx), device=DEV, dtype=torch.float64), torch.empty((nz, ny, nx, 3), device=DEV, dtype=torch.float64)
    for c in range(4):
        acc = torch.zeros((nz, ny, nx), device=DEV, dtype=torch.float64)
        for _ in range(4):
            k, ph, a = rng.integers(-3, 4, size=3), rng.uniform(0, 2 * math.pi), rng.standard_normal()
            z, y, x = (2 * math.pi * float(kk) * v for kk, v in zip(k, ax))
            acc += a * torch.cos(z[:, None, None] + (y[:, None] + x[None, :] + ph)[None])
        acc *= (0.01 if c < 3 else 1e-3) / float(acc.abs().max().clamp(min=1e-30))
        if c < 3:
            u[..., c] = acc
        else:
            rho.copy_(1.0 + acc)
    return rho.cpu().numpy(), u.cpu().numpy()


def _body(case, seed):
    """Mesh (turned by the seed), start position, velocities and gravity of a case's particle."""
    rng = np.random.default_rng([seed, 2])
    V, Tr = _mesh(case["shape"], case["d"])
    if case["shape"] != "sphere":
        V = I.rotate(I.rotate(V, "x", float(rng.uniform(0.0, 45.0))), "z", float(rng.uniform(0.0, 90.0)))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    z0 = case["anchor"] * nz if case["slide"] else 0.65 * nz
    r0 = np.array([0.5 * nx - 0.5, 0.5 * ny - 0.5, z0]) + rng.uniform(-0.4, 0.4, 3)
    vt = case["re"] * case["nu"] / case["d"]
    v0 = np.array([0.0, 0.0, -0.3 * vt]) + 0.02 * vt * rng.standard_normal(3)
    w0 = 0.05 * vt / case["d"] * rng.standard_normal(3)
    g = (0.0, 0.0, -configs.gravity_for(case["re"], case["d"], case["nu"], case["kappa"]))
    return V, Tr, tuple(r0), tuple(v0), tuple(w0), g


def _walls(case):
    """Velocities of sliding bottom and top walls (bc 3)."""
    return ((-0.02, 0.0, 0.0) if case["bc_bottom"] == 3 else (0.0, 0.0, 0.0),
            (0.02, 0.005, 0.0) if case["bc_top"] == 3 else (0.0, 0.0, 0.0))


def _flags(case):
    f = {}
    if case.get("force_eval"):
        f["force_eval"] = 1
    if case.get("sround"):
        f["stochastic_rounding"] = 1
    return f


def _set_predictor(t, mode):
    if mode != "paper":
        t.set_predictor("linear", warm=mode == "linear_warm", slip_eps=1e-4)


def _open(case, g):
    return T.Turret(case["nx"], case["ny"], case["nz"], case["nu"], case.get("kappa", 1.0), g, case["bc_x"], case["bc_y"],
                    case["bc_bottom"], case["bc_top"], sponge=case["sponge"], slide=case.get("slide", 0),
                    anchor_frac=case.get("anchor", 0.25), storage=case["storage"], flags=_flags(case) or None, device=DEV)


def _pairs(rows, seed):
    """Rows of the network's inputs and targets with the spread of logged trajectories: unit-scale scaled forces and
    quaternions, small velocities, targets a smooth function of them plus noise (host float32)."""
    rng = np.random.default_rng([seed, 3])
    scale = np.concatenate([np.full(4, 0.5), np.full(3, 1e-2), np.full(3, 1e-3), np.full(24, 0.6)])
    x = rng.standard_normal((rows, T.MLP_IN)) * scale + 0.2 * scale
    A = rng.standard_normal((T.MLP_IN, T.MLP_OUT)) / scale[:, None] / math.sqrt(T.MLP_IN)
    y = 1e-3 * (np.tanh(x @ A) + 0.3 * np.sin(x @ A[:, ::-1]) + 0.05 * rng.standard_normal((rows, T.MLP_OUT)))
    return x.astype(np.float32), y.astype(np.float32)


def _norm(x, y):
    return x.mean(0), x.std(0), y.mean(0), y.std(0)


def _markers(case, seed):
    """Positions, forces and areas of markers on a sphere inside the grid (host arrays)."""
    rng = np.random.default_rng([seed, 4])
    V, Tr = _unit_sphere(case["freq"])
    room = np.array([case["nx"], case["ny"], case["nz"]]) - 2.0 * case["radius"] - 6.0
    X = case["radius"] * V + (0.5 * np.array([case["nx"], case["ny"], case["nz"]]) - 0.5 + 0.4 * room * rng.uniform(-1, 1, 3))
    h = 1e-3 * rng.standard_normal(X.shape)
    dS = np.full(len(X), 4 * math.pi * case["radius"] ** 2 / len(X)) * rng.uniform(0.8, 1.2, len(X))
    return X.astype(np.float32), h.astype(np.float32), dS.astype(np.float32)


@functools.lru_cache(maxsize=32)
def _unit_sphere(freq):
    return I.icosphere(freq)


# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("settle", "monitor"):
        V, Tr, r0, v0, w0, g = _body(case, seed)
        s["t"] = t = _open(case, g)
        t.set_fields(*_fields(case["nz"], case["ny"], case["nx"], seed))
        _set_predictor(t, case["predictor"])
        t.load_surface(V, Tr, r0, v0, w0)
    elif kind == "session":
        s["body"] = _body(case, seed)
        s["fields"] = _fields(case["nz"], case["ny"], case["nx"], seed)
    elif kind == "ensemble":
        s["runs"] = []
        rng = np.random.default_rng([seed, 5])
        for k, c in enumerate(_ensemble(case["runs"], case["pick"], case["storage"], case["d_max"])):
            t = configs.make_turret(c, device=DEV)
            t.set_fields(*_fields(c["nz"], c["ny"], c["nx"], seed + 1000 * k))
            _set_predictor(t, case["predictor"])
            t.load_surface(c["verts"], c["tris"], c["r0"], (0.0, 0.0, -0.02 * float(rng.uniform(0.1, 0.5))))
            s["runs"].append(t)
        s["batch"] = T.Batch(s["runs"], device=DEV)
    elif kind == "fluid":
        s["t"] = t = _open(case, (0.0, 0.0, 0.0))
        if 3 in (case["bc_bottom"], case["bc_top"]):
            t.set_wall_velocity(*_walls(case))
        t.set_fields(*_fields(case["nz"], case["ny"], case["nx"], seed))
    elif kind in ("train", "infer"):
        x, y = _pairs(case["rows"], seed)
        s["net"] = net = T.MLP(I.mlp_init_params(seed).astype(np.float32), batch_cap=case.get("batch", 4096),
                               precision=case["precision"], device=DEV)
        net.set_norm(*_norm(x, y))
        s["x"], s["y"] = torch.as_tensor(x, device=DEV), torch.as_tensor(y, device=DEV)
    else:
        X, h, dS = _markers(case, seed)
        s.update(X=torch.as_tensor(np.ascontiguousarray(X.T), device=DEV), h=torch.as_tensor(np.ascontiguousarray(h.T), device=DEV),
                 dS=torch.as_tensor(dS, device=DEV))
    return s


def _read(t):
    st = t.state()
    return {k: st[k] for k in STATE_KEYS}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "settle":
        s["t"].step(case["steps"])
        return {"state": _read(s["t"]), "fields": s["t"].macro()}
    if kind == "monitor":
        log = []
        for _ in range(case["steps"]):
            s["t"].step(1)
            log.append(_read(s["t"]))
        return {"state": {k: np.stack([e[k] for e in log]) for k in STATE_KEYS}, "fields": s["t"].macro()}
    if kind == "session":
        V, Tr, r0, v0, w0, g = s["body"]
        t = _open(case, g)
        t.set_fields(*s["fields"])
        _set_predictor(t, case["predictor"])
        t.load_surface(V, Tr, r0, v0, w0)
        t.step(case["steps"])
        out = {"state": _read(t), "fields": t.macro()}
        t.close()
        return out
    if kind == "ensemble":
        s["batch"].step(case["steps"])
        states = [_read(t) for t in s["runs"]]
        return {"state": {k: np.stack([e[k] for e in states]) for k in STATE_KEYS}, "fields": [t.macro() for t in s["runs"]]}
    if kind == "fluid":
        s["t"].fluid_step(case["steps"])
        return s["t"].populations()
    if kind == "train":
        net, history = surrogate.train(s["x"], s["y"], epochs=1, batch=case["batch"], net=s["net"])
        return {"loss": history[0], "params": net.params()}
    if kind == "infer":
        return s["net"].infer(s["x"])
    return T.ibm_spread(s["X"], s["h"], s["dS"], (case["nz"], case["ny"], case["nx"]))


FLOPS_PER_CELL = 500  # moments, equilibrium and off-equilibrium rebuild of one D3Q27 cell


def _window_work(nx, ny, nz, storage, steps, markers, out_planes):
    cells = nx * ny * nz
    pop = 4 if storage == "f32" else 2
    # the state in and out once, the requested fields once; every step's arithmetic
    return (2 * 27 * pop * cells + 4 * out_planes * cells + 200 * markers, steps * (FLOPS_PER_CELL * cells + 64 * 100 * markers))


def work(case):
    kind = case["kind"]
    if kind in ("settle", "monitor", "session"):
        b, f = _window_work(case["nx"], case["ny"], case["nz"], case["storage"], case["steps"], int(3.9 * case["d"] ** 2), 4)
        if kind == "session":  # fields from host memory instead of the populations
            b = 32 * case["nx"] * case["ny"] * case["nz"] + 16 * case["nx"] * case["ny"] * case["nz"]
    elif kind == "ensemble":
        b = f = 0
        for c in _ensemble(case["runs"], case["pick"], case["storage"], case["d_max"]):
            wb, wf = _window_work(c["nx"], c["ny"], c["nz"], c["storage"], case["steps"], len(c["verts"]), 4)
            b, f = b + wb, f + wf
    elif kind == "fluid":
        b, f = _window_work(case["nx"], case["ny"], case["nz"], case["storage"], case["steps"], 0, 27)
    elif kind in ("train", "infer"):
        weights = 34 * 128 + 2 * 128 * 128 + 6 * 128
        steps = case["rows"] // case["batch"] if kind == "train" else 1
        rows = steps * case["batch"] if kind == "train" else case["rows"]
        b = rows * 40 * 4 + steps * 4 * weights * (6 if kind == "train" else 1)
        f = rows * weights * (6 if kind == "train" else 2)
    else:
        markers = 10 * case["freq"] ** 2 + 2
        b, f = 12 * case["nx"] * case["ny"] * case["nz"] + 28 * markers, markers * 64 * 9
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# The same results in 64 bits: a dense solver of the method in plain torch.

def exact(case, seed):
    kind = case["kind"]
    if kind in ("settle", "monitor", "session"):
        V, Tr, r0, v0, w0, g = _body(case, seed)
        sim = _Solver(case, g, *_fields(case["nz"], case["ny"], case["nx"], seed))
        sim.load(V, Tr, r0, v0, w0)
        log = []
        for _ in range(case["steps"]):
            sim.step()
            log.append(sim.state())
        state = {k: np.stack([e[k] for e in log]) for k in STATE_KEYS} if kind == "monitor" else log[-1]
        return {"state": state, "fields": sim.macro()}
    if kind == "ensemble":
        states, fields = [], []
        rng = np.random.default_rng([seed, 5])
        for k, c in enumerate(_ensemble(case["runs"], case["pick"], case["storage"], case["d_max"])):
            bc = dict(zip(("bc_x", "bc_y", "bc_bottom", "bc_top"), c["bc"]))
            sim = _Solver(dict(c, **bc, predictor=case["predictor"]), c["g"], *_fields(c["nz"], c["ny"], c["nx"], seed + 1000 * k))
            sim.load(c["verts"], c["tris"], c["r0"], (0.0, 0.0, -0.02 * float(rng.uniform(0.1, 0.5))), (0.0, 0.0, 0.0))
            for _ in range(case["steps"]):
                sim.step()
            states.append(sim.state())
            fields.append(sim.macro())
        return {"state": {k: np.stack([e[k] for e in states]) for k in STATE_KEYS}, "fields": fields}
    if kind == "fluid":
        sim = _Solver(case, (0.0, 0.0, 0.0), *_fields(case["nz"], case["ny"], case["nx"], seed))
        for _ in range(case["steps"]):
            sim.step()
        return sim.q
    if kind in ("train", "infer"):
        return _exact_net(case, seed)
    X, h, dS = (torch.as_tensor(a, device=DEV).double() for a in _markers(case, seed))
    idx, w = _stencil(X, (case["nx"], case["ny"], case["nz"]), (False, False, False))
    return _spread(idx, w, h * dS[:, None], case["nx"] * case["ny"] * case["nz"]).reshape(3, case["nz"], case["ny"], case["nx"])


def _exact_net(case, seed):
    x32, y32 = _pairs(case["rows"], seed)
    mx, sx, my, sy = (torch.as_tensor(np.asarray(a, np.float32), device=DEV).double() for a in _norm(x32, y32))
    x, y = (torch.as_tensor(x32, device=DEV).double() - mx) / sx, (torch.as_tensor(y32, device=DEV).double() - my) / sy
    flat = torch.as_tensor(I.mlp_init_params(seed).astype(np.float32), device=DEV).double()
    shapes, mats, at = ((128, 34), (128, 128), (128, 128), (6, 128)), [], 0
    decay = torch.zeros_like(flat)
    for o, i in shapes:
        decay[at:at + o * i] = 1.0
        mats.append((at, o, i))
        at += o * i + o

    def net(p, rows):
        for l, (a, o, i) in enumerate(mats):
            rows = rows @ p[a:a + o * i].reshape(o, i).T + p[a + o * i:a + o * i + o]
            rows = torch.nn.functional.gelu(rows) if l < 3 else rows
        return rows

    if case["kind"] == "infer":
        return net(flat, x) * sy + my
    lr, wd, b1, b2, eps, losses = 1e-3, 1e-4, 0.9, 0.999, 1e-8, []
    m, v = torch.zeros_like(flat), torch.zeros_like(flat)
    perm = torch.as_tensor(np.random.default_rng(0).permutation(case["rows"]), device=DEV)
    for k in range(case["rows"] // case["batch"]):
        at = perm[k * case["batch"]:(k + 1) * case["batch"]]
        p = flat.clone().requires_grad_(True)
        loss = (net(p, x[at]) - y[at]).square().mean()
        g, = torch.autograd.grad(loss, p)
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        flat = flat - lr * ((m / (1 - b1 ** (k + 1))) / ((v / (1 - b2 ** (k + 1))).sqrt() + eps) + wd * decay * flat)
        losses.append(float(loss.detach()))
    return {"loss": float(np.mean(losses)), "params": flat.float().double().cpu().numpy()}


def _peskin(r):
    a = r.abs()
    inner = 0.125 * (3 - 2 * a + (1 + 4 * a - 4 * a * a).clamp(min=0).sqrt())
    outer = 0.125 * (5 - 2 * a - (-7 + 12 * a - 4 * a * a).clamp(min=0).sqrt())
    return torch.where(a < 1, inner, torch.where(a < 2, outer, torch.zeros_like(a)))


def _stencil(X, n, periodic):
    """Flat cell indices and weights [markers][64] of the 4-point kernel around X [markers][3]."""
    base = X.floor().long() - 1
    off = torch.arange(4, device=X.device)
    idx, w = None, None
    for a in (2, 1, 0):
        c = base[:, a, None] + off
        wa = _peskin(c - X[:, a, None])
        c = c % n[a] if periodic[a] else c
        idx = c if idx is None else (idx[:, :, None] * n[a] + c[:, None, :]).reshape(len(X), -1)
        w = wa if w is None else (w[:, :, None] * wa[:, None, :]).reshape(len(X), -1)
    return idx, w


def _spread(idx, w, f, cells):
    out = torch.zeros((3, cells), device=f.device, dtype=f.dtype)
    for c in range(3):
        out[c].index_add_(0, idx.reshape(-1), (w * f[:, c, None]).reshape(-1))
    return out


def _axis(u):
    """w1(xi) (1 + 3 xi u + 9/2 (xi^2 - 1/3) u^2) for xi = -1, 0, 1 and its first two derivatives in u."""
    return (((1 - 3 * u + 3 * u * u) / 6, 2 / 3 - u * u, (1 + 3 * u + 3 * u * u) / 6), (u - 0.5, -2 * u, u + 0.5), (1.0, -2.0, 1.0))


W1 = (1 / 6, 2 / 3, 1 / 6)
XI = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)]
WEIGHT = [W1[x + 1] * W1[y + 1] * W1[z + 1] for x, y, z in XI]


def _mesh_properties(V, Tr):
    """Marker areas, outward normals, offset-surface areas, volume, centre of mass and J/m of a closed surface."""
    p = V[Tr]
    cr = np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    area = 0.5 * np.linalg.norm(cr, axis=1)
    dS, nrm, dSo = np.zeros(len(V)), np.zeros((len(V), 3)), np.zeros(len(V))
    for e in range(3):
        np.add.at(dS, Tr[:, e], area / 3)
        np.add.at(nrm, Tr[:, e], 0.5 * cr)
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    po = (V + 2.0 * nrm)[Tr]
    ao = 0.5 * np.linalg.norm(np.cross(po[:, 1] - po[:, 0], po[:, 2] - po[:, 0]), axis=1)
    for e in range(3):
        np.add.at(dSo, Tr[:, e], ao / 3)
    tv = np.einsum("ij,ij->i", p[:, 0], np.cross(p[:, 1], p[:, 2])) / 6
    s = p.sum(1)
    vol = tv.sum()
    com = (tv[:, None] * s).sum(0) / 4 / vol
    S = np.einsum("t,tea,teb->ab", tv, p, p) / 20 + np.einsum("t,ta,tb->ab", tv, s, s) / 20 - vol * np.outer(com, com)
    return dS, nrm, dSo, vol, com, (np.trace(S) * np.eye(3) - S) / vol


class _Solver:
    """Dense D3Q27 recursive-regularized lattice Boltzmann with an immersed rigid body, one step after another
    (arXiv 2408.15115, Table 1), on the deviations q_i = f_i - w_i."""

    def __init__(self, case, g, rho, u):
        self.case, self.n = case, (case["nx"], case["ny"], case["nz"])
        self.bc = case["bc_x"], case["bc_y"], case["bc_bottom"], case["bc_top"]
        self.periodic = self.bc[0] == 0, self.bc[1] == 0, self.bc[2] == 0
        tau0, L, nz = 3 * case["nu"] + 0.5, case["sponge"], case["nz"]
        z = torch.arange(nz, device=DEV, dtype=torch.float64)
        self.tau = torch.where(z >= nz - L, tau0 + (1 - tau0) * (z - (nz - L) + 1) / max(L, 1), torch.full_like(z, tau0))[:, None, None]
        self.walls = _walls(case) if 3 in self.bc else None
        self.g, self.body, self.h = np.array(g), False, None
        u = torch.as_tensor(u, device=DEV).movedim(-1, 0)
        rho = torch.as_tensor(rho, device=DEV)
        self.utop = u[:, -1].clone()
        post = torch.empty((27,) + tuple(rho.shape), device=DEV, dtype=torch.float64)
        self._equilibrium(rho, u, post)
        self.q = torch.empty_like(post)
        self._stream(post)
        self.spare = post

    def _equilibrium(self, rho, u, out, factor=1.0, add=False):
        ax = [_axis(u[a])[0] for a in range(3)]
        for i, (x, y, z) in enumerate(XI):
            e = factor * (rho * ax[0][x + 1] * ax[1][y + 1] * ax[2][z + 1] - WEIGHT[i])
            if add:
                out[i] += e
            else:
                out[i] = e

    def _moments(self):
        q = self.q
        drho = q.sum(0)
        j = [sum(XI[i][a] * q[i] for i in range(27) if XI[i][a]) for a in range(3)]
        u = torch.stack(j) / (1 + drho)
        P = {}
        for a in range(3):
            for b in range(a, 3):
                s = sum(XI[i][a] * XI[i][b] * q[i] for i in range(27) if XI[i][a] * XI[i][b])
                P[a, b] = s - (drho / 3 if a == b else 0) - j[a] * u[b]
        return drho, u, P

    def _collide(self, post):
        drho, u, P = self._moments()
        om = 1 / self.tau
        self._equilibrium(1 + drho, u, post, 1 - om if self.body else 1.0)
        if self.body:
            self._equilibrium(1 + drho, u + self.tau * self.h, post, om, add=True)
        f, d1, d2 = zip(*(_axis(u[a]) for a in range(3)))
        for i, (x, y, z) in enumerate(XI):
            x, y, z = x + 1, y + 1, z + 1
            f1 = 0.5 * (P[0, 0] * d2[0][x] * f[1][y] * f[2][z] + P[1, 1] * f[0][x] * d2[1][y] * f[2][z]
                        + P[2, 2] * f[0][x] * f[1][y] * d2[2][z])
            f1 += P[0, 1] * d1[0][x] * d1[1][y] * f[2][z] + P[0, 2] * d1[0][x] * f[1][y] * d1[2][z] + P[1, 2] * f[0][x] * d1[1][y] * d1[2][z]
            post[i] += (1 - om) * f1
        self.utop = u[:, -1].clone()

    def _stream(self, post):
        bx, by, bottom, top = self.bc
        for i, (x, y, z) in enumerate(XI):
            g, opp = torch.roll(post[i], (z, y, x), (0, 1, 2)), post[26 - i]
            if top == 2 and z == -1:  # ghost plane: rest density with the top plane's velocity
                ug = torch.roll(self.utop, (y, x), (1, 2))
                a = [_axis(ug[c])[0] for c in range(3)]
                g[-1] = a[0][x + 1] * a[1][y + 1] * a[2][z + 1] - WEIGHT[i]
            if bx == 1 and x:
                g[:, :, 0 if x > 0 else -1] = opp[:, :, 0 if x > 0 else -1]
            if by == 1 and y:
                g[:, 0 if y > 0 else -1] = opp[:, 0 if y > 0 else -1]
            for face, bc, at in ((1, bottom, 0), (-1, top, -1)):
                if z == face and bc in (1, 3):
                    uw = self.walls[0 if face > 0 else 1] if bc == 3 else (0, 0, 0)
                    g[at] = opp[at] + 6 * WEIGHT[i] * (x * uw[0] + y * uw[1] + z * uw[2])
            self.q[i] = g

    def load(self, V, Tr, r0, v0, w0):
        dS, nrm, dSo, self.vol, com, self.J = _mesh_properties(np.asarray(V, dtype=np.float64), np.asarray(Tr))
        dev = lambda a: torch.as_tensor(a, device=DEV)  # noqa: E731
        self.Xb, self.nb, self.dS, self.dSo = dev(V - com), dev(nrm), dev(dS), dev(dSo)
        self.m = self.case["kappa"] * self.vol
        self.r, self.v, self.w = (np.array(a, dtype=np.float64) for a in (r0, v0, w0))
        self.d, self.origin, self.L = np.eye(3), np.zeros(3, dtype=np.int64), self.m * self.J @ self.w
        self.body, self.hl, self.hist = True, None, []
        self._couple(self.v, self.w, warm=False)

    def _couple(self, vel, om, warm):
        """Force and torque at the new time level, then the immersed-boundary cycles."""
        drho, u, P = self._moments()
        k = 0.5 / self.tau - 1
        C = torch.as_tensor(self.r - self.origin, device=DEV)
        M = torch.as_tensor(self.d, device=DEV)
        arm, nn = self.Xb @ M, self.nb @ M
        X = C + arm
        U = torch.as_tensor(vel, device=DEV) + torch.linalg.cross(torch.as_tensor(om, device=DEV).expand_as(arm), arm)
        off = 0.0 if self.case.get("force_eval") else 2.0
        area = self.dS if self.case.get("force_eval") else self.dSo
        idx, w = _stencil(X + off * nn, self.n, self.periodic)
        at = lambda a: (a.reshape(-1)[idx] * w).sum(1)  # noqa: E731
        p = at(drho) / 3
        s = {ab: at(k * P[ab]) for ab in P}
        tr = torch.stack([sum(s[min(a, b), max(a, b)] * nn[:, b] for b in range(3)) - p * nn[:, a] for a in range(3)], 1) * area[:, None]
        self.F = tr.sum(0).cpu().numpy()
        self.T = torch.linalg.cross(arm + off * nn, tr).sum(0).cpu().numpy()
        self.Fp = -(area[:, None] * p[:, None] * nn).sum(0).cpu().numpy()
        self.hist = [(self.F, self.T)] + self.hist[:1]
        idx, w = _stencil(X, self.n, self.periodic)
        cells = self.n[0] * self.n[1] * self.n[2]
        interp = lambda a: torch.stack([(a[c].reshape(-1)[idx] * w).sum(1) for c in range(3)], 1)  # noqa: E731
        r0 = U - interp(u)
        h, cycles = (self.hl, 4) if warm else (r0, 3)
        for _ in range(cycles):
            res = r0 - interp(_spread(idx, w, h * self.dS[:, None], cells))
            h = h + res
            if warm and float(res.abs().max()) < 1e-4:
                break
        self.hl = h
        self.h = _spread(idx, w, h * self.dS[:, None], cells).reshape(3, *self.q.shape[1:])

    def step(self):
        post = self.spare
        self._collide(post)
        if self.body:
            mode = self.case.get("predictor", "paper")
            (F0, T0), (F1, T1) = self.hist[0], self.hist[-1]
            ge = (1 - 1 / self.case["kappa"]) * self.g
            self.v = self.v + ge + self.F / self.m
            self.r = self.r + self.v
            self.L = self.L + self.T
            Ji, d = np.linalg.inv(self.J), self.d
            self.w = d.T @ Ji @ d @ self.L / self.m
            self.d = d + np.cross(self.w, d + 0.5 * np.cross(self.w, d))
            if self.case.get("slide"):
                dz = self.r[2] - self.origin[2] - self.case.get("anchor", 0.25) * self.n[2]
                move = -1 if dz <= -1 else 1 if dz >= 1 else 0
                if move:  # the window follows by one plane; the entering plane is at rest
                    post.copy_(torch.roll(post, -move, 1))
                    post[:, 0 if move < 0 else -1] = 0.0
                    self.origin[2] += move
        self._stream(post)
        if self.body:
            vel, om = self.v, self.w
            if mode != "paper":
                vel = self.v + 0.5 * (ge + (2 * F0 - F1) / self.m)
                om = self.d.T @ Ji @ self.d @ (self.L + 0.5 * (2 * T0 - T1)) / self.m
            self._couple(vel, om, warm=mode == "linear_warm")

    def state(self):
        return {"r": self.r, "d": self.d, "v": self.v, "w": self.w, "F": self.F, "T": self.T, "L": self.L, "Fp": self.Fp,
                "origin": self.origin.copy()}

    def macro(self):
        drho = self.q.sum(0)
        return torch.cat([(1 + drho)[None], torch.stack([sum(XI[i][a] * self.q[i] for i in range(27) if XI[i][a]) for a in range(3)])
                          / (1 + drho)])
