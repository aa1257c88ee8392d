"""Work that users of this framework have it do, as cases that can be timed.

A case is a dict of plain values.  Its "kind" is one of
  run    one lattice with its membranes, advanced by ``Simulation.step``; the
         markers and the fields phi, psi and u are then read back
         ("init": the plain start, given fields, or given fields uploaded
         again at the beginning of every pass);
  batch  a parameter sweep of lattices advanced by ``Batch.step``; the
         markers and the field psi of every lattice are then read back;
  net    the warm-start network: its forward pass, or one training step.
Fields are read as doubles into pinned host buffers that the program keeps
(as ``bench.py`` does) and kept in the run's own storage type; the markers
are kept in the run's arithmetic type.

``exact`` computes the same results in 64 bits with plain torch: the method of
the paper (ternary free-energy lattice Boltzmann fluid, elastic membranes,
immersed boundary coupling), and the network's definition in ``tlb.h``.
"""
import functools
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1906_03065_gb300 import Batch, Simulation, WarmStartNet, workloads as W

DEV = "cuda:0"
OUT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


# ------------------------------------------------------------------ the cases
def _run(name, storage, nx, ny, nz, radius, steps, alpha=2.0, caps=1, tau=1.0, forcing="edm",
         state="populations", init="plain"):
    return {"name": name, "kind": "run", "storage": storage, "nx": nx, "ny": ny, "nz": nz, "radius": radius,
            "steps": steps, "alpha": alpha, "caps": caps, "tau": tau, "forcing": forcing, "state": state,
            "init": init}


def _batch(name, dim, storage, n, lo, hi, steps, membrane=True):
    return {"name": name, "kind": "batch", "dim": dim, "storage": storage, "n": n, "lo": lo, "hi": hi,
            "steps": steps, "membrane": membrane}


def _net(name, edge, channels, levels, batch, train):
    return {"name": name, "kind": "net", "edge": edge, "channels": channels, "levels": levels, "batch": batch,
            "train": train}


def listed():
    return [
        # the smallest run there is: a 2D capsule in double precision, where
        # launches and latency are all the time
        _run("ring_64_f64", "f64", 64, 64, 1, 12.0, 60, alpha=1.0),
        # one drifting capsule of the paper's Sec. 4.1 (the Galilean runs)
        _run("paper_240x120_f32", "f32", 240, 120, 1, 20.0, 100),
        # a small ragged 3D lattice: odd sizes, a coarse mesh
        _run("ragged_41x37x35_f32", "f32", 41, 37, 35, 7.0, 60, alpha=1.0),
        # a relaxation from given fields: upload, equilibrium start, steps
        _run("restart_64_f32", "f32", 64, 64, 64, 13.0, 60, init="restart"),
        # the framework's headline workload
        _run("capsule_128_f32", "f32", 128, 128, 128, 20.0, 100),
        # the two-capsule bridge with 16-bit storage, the largest lattice
        _run("bridge_192x128x128_f16", "f16", 192, 128, 128, 20.0, 60, caps=2),
        # other relaxation times with Guo forcing: the general collision
        _run("guo_96_f32", "f32", 96, 96, 96, 16.0, 60, tau=0.8, forcing="guo"),
        # a liquid lens with no membrane (the pure-liquid reference of Sec.
        # 4.1), odd sizes, bfloat16 storage
        _run("lens_97x111x90_bf16", "bf16", 97, 111, 90, 20.0, 60, caps=0, init="fields"),
        # the 3D parameter sweep, 16 lattices of 48^3 to 96^3
        _batch("sweep_16x_f16", 3, "f16", 16, 48, 96, 40),
        # the paper's 2D sweep over stiffness and tension, 24 lattices
        _batch("paper_sweep_24x_f32", 2, "f32", 24, 240, 240, 100),
        # the warm start's network: inference on eight instances
        _net("net_forward_48x8", 48, 16, 4, 8, False),
        # and one training step of it
        _net("net_train_48x8", 48, 16, 4, 8, True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run2d", "run3d", "run3d", "run3d", "batch2d", "batch3d", "net"])
    if kind == "run2d":
        R = rng.uniform(9.0, 20.0)
        ny = rng.randint(int(4 * R) + 12, 140)
        return _drawn(_run("", rng.choice(["f64", "f32"]), rng.randint(int(4 * R) + 12, 300), ny, 1, R,
                           rng.randint(40, 100), alpha=rng.choice([1.0, 2.0])))
    if kind == "run3d":
        storage = rng.choice(["f32", "f32", "f16", "bf16"])
        general = rng.random() < 0.2
        t = rng.uniform(0.75, 1.2) if general else 1.0
        n = [_log_int(rng, 40, 132) for _ in range(3)]
        alpha = 2.0 if min(n) >= 64 else 1.0
        R = rng.uniform(0.15, 0.22) * min(n)
        moments = storage == "f32" and not general and rng.random() < 0.15
        caps = rng.choice([0, 1, 1, 1])
        init = "fields" if caps == 0 else ("restart" if rng.random() < 0.2 else "plain")
        return _drawn(_run("", storage, n[0], n[1], n[2], R, rng.randint(30, 60), alpha=alpha,
                           caps=caps, tau=t, forcing=rng.choice(["edm", "guo"]) if general else "edm",
                           state="moments" if moments else "populations", init=init))
    if kind == "batch2d":
        lo = rng.randint(130, 200)
        return _drawn(_batch("", 2, rng.choice(["f32", "f64"]), rng.randint(4, 32), lo, lo + rng.randint(8, 40),
                             rng.randint(30, 60), membrane=rng.random() < 0.8))
    if kind == "batch3d":
        lo = rng.randint(48, 64)
        return _drawn(_batch("", 3, rng.choice(["f16", "f32"]), rng.randint(2, 14), lo, lo + rng.randint(4, 32),
                             rng.randint(15, 30)))
    levels = rng.choice([3, 4])
    edge = 8 * rng.randint(2, 6)
    return _drawn(_net("", edge, rng.choice([16, 32]), levels, rng.randint(1, 6), rng.random() < 0.5))


def _drawn(c):
    del c["name"]
    return c


# ----------------------------------------------------------------- the inputs
@functools.lru_cache(maxsize=None)
def _unit_sphere(level):
    m = W.icosphere(level, 1.0, (0.0, 0.0, 0.0))
    return m.X, m.elems


def _capsule(dim, nominal, centre, rng, paper=False):
    """A membrane whose mesh is that of the nominal radius (markers about one
    lattice unit apart in 2D, an icosphere of the level the sweeps use in 3D),
    its radius within 2% of that, its moduli drawn over the sweeps' ranges."""
    R = nominal * float(rng.uniform(0.98, 1.0))
    if dim == 2:
        m = W.ring(int(round(2 * math.pi * nominal)), R, centre, phase=float(rng.uniform(0, 0.1)))
        m.ks = float(10 ** rng.uniform(-3, -1)) if paper else float(rng.uniform(0.03, 0.07))
        m.kb = float(10 ** rng.uniform(-4, -2)) if paper else float(rng.uniform(5e-4, 2e-3))
        return m
    X, T = _unit_sphere(2 if nominal < 9 else (3 if nominal < 15 else 4))
    m = W.Membrane(W.MEM_TRI3D, np.asarray(centre)[None, :] + R * X, T.copy())
    m.G, m.C, m.kb = float(rng.uniform(0.005, 0.02)), 1.0, float(rng.uniform(0.003, 0.007))
    return m


def _workload(case, seed):
    """The lattice and its membranes: sizes from the case; centres, tensions,
    stiffnesses and the initial drift from the seed."""
    rng = np.random.default_rng([seed, 1])
    dim = 2 if case["nz"] == 1 else 3
    R = case["radius"]
    last = case["ny"] if dim == 2 else case["nz"]
    u = float(10 ** rng.uniform(-2.5, -2))
    ang = float(rng.uniform(0, 2 * math.pi))
    gam = 0.2 if (dim == 2 and case["alpha"] < 2) else 1.0
    p = W.Params(dim=dim, nx=case["nx"], ny=case["ny"], nz=case["nz"], wall_last=int(dim == 3),
                 storage=case["storage"], tau=case["tau"], tau_phi=1.0, tau_psi=1.0, gamma_phi=gam,
                 gamma_psi=gam, alpha=case["alpha"], kappa1=float(rng.uniform(0.006, 0.012)),
                 kappa2=float(rng.uniform(0.008, 0.018)), kappa3=float(rng.uniform(0.008, 0.015)), kappa_c=0.01,
                 dc=8.0 * case["alpha"], interface_pos=-1.0 if case["caps"] == 2 else last / 2.0,
                 u0=(u, 0.0, 0.0) if dim == 2 else (u * math.cos(ang), u * math.sin(ang), 0.0),
                 forcing=case["forcing"], state=case["state"])
    n = [case["nx"], case["ny"], case["nz"]][:dim]
    mems = []
    for k in range(case["caps"]):
        c = [v / 2.0 + float(rng.uniform(-0.5, 0.5)) for v in n] + [0.0] * (3 - dim)
        if case["caps"] == 2:
            c[0] += (k - 0.5) * 2.4 * R
        mems.append(_capsule(dim, R, c, rng, paper=case["alpha"] >= 2))
    return W.Workload("", p, mems)


def _sweep(case, seed):
    """A sweep's lattices: sizes spread over the case's range, the rest drawn."""
    rng = np.random.default_rng([seed, 2])
    out = []
    for i in range(case["n"]):
        at = ((i * 7 + 3) % 16) / 15
        if case["dim"] == 2:  # 12R x 6R lattices of Sec. 4.1
            nx = case["lo"] + round((case["hi"] - case["lo"]) * at)
            ny, R = nx // 2, nx / 12.0
            p = W.Params(dim=2, nx=nx, ny=ny, nz=1, storage=case["storage"], alpha=2.0,
                         kappa1=8e-3, kappa2=float(rng.choice([8e-3, 2e-3])), kappa3=float(rng.uniform(5e-4, 1e-2)),
                         kappa_c=0.01, dc=16.0, interface_pos=ny / 2.0, u0=(float(10 ** rng.uniform(-4, -2)), 0.0, 0.0))
            c = (nx / 2.0 + float(rng.uniform(-0.5, 0.5)), ny / 2.0 + float(rng.uniform(-0.5, 0.5)), 0.0)
        else:
            n = case["lo"] + round((case["hi"] - case["lo"]) * at)
            R = n * (0.15 + 0.1 * ((i * 5 + 2) % 11) / 10)
            k1, k2, k3 = (float(v) for v in rng.uniform(0.005, 0.03, 3))
            p = W.Params(dim=3, nx=n, ny=n, nz=n, wall_last=1, storage=case["storage"], alpha=2.0, gamma_phi=0.5,
                         gamma_psi=0.5, kappa1=k1, kappa2=k2, kappa3=k3, kappa_c=0.01, dc=16.0, interface_pos=n / 2.0)
            c = tuple(n / 2.0 + float(v) for v in rng.uniform(-0.5, 0.5, 3))
        out.append(W.Workload("", p, [_capsule(case["dim"], R, c, rng, paper=True)] if case["membrane"] else []))
    return out


def _fields(case, wl, seed):
    """Concentrations and velocity that a 3D program starts from: the C3
    profile of a capsule (or of a lens, without one) in two fluids with a
    tilted, wavy interface, and a shear flow."""
    rng = np.random.default_rng([seed, 3])
    p = wl.params
    a, amp, tilt = p.alpha, float(rng.uniform(0.5, 1.5)), float(rng.uniform(-0.05, 0.05))
    z, y, x = (v.ravel() for v in np.meshgrid(np.arange(p.nz, dtype=float), np.arange(p.ny, dtype=float),
                                              np.arange(p.nx, dtype=float), indexing="ij"))
    C3 = np.zeros(p.ncells)
    drops = [(m.X.mean(axis=0), float(np.linalg.norm(m.X - m.X.mean(axis=0), axis=1).mean())) for m in wl.membranes]
    for c, R in drops or [((p.nx / 2.0, p.ny / 2.0, p.nz / 2.0), case["radius"] * float(rng.uniform(0.95, 1.05)))]:
        C3 = np.maximum(C3, 0.5 * (1 + np.tanh((R - np.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2)) / (2 * a))))
    h = p.nz / 2.0 + amp * np.cos(2 * math.pi * x / p.nx) + tilt * np.sin(2 * math.pi * y / p.ny) * p.ny
    s = 0.5 * (1 + np.tanh((z - h) / (2 * a)))
    u = np.zeros((3, p.ncells))
    u[0] = 4e-3 * np.sin(math.pi * (z + 0.5) / p.nz)
    u[1] = 2e-3 * np.sin(math.pi * (z + 0.5) / p.nz) * np.cos(2 * math.pi * x / p.nx)
    return np.stack([(1 - C3) * s, (1 - C3) * (1 - s), C3]), u


def _net_inputs(case, seed):
    """Network inputs as the warm start makes them (a diffuse capsule on a flat
    interface and normalised parameters), He-normal weights, and targets of
    the size of its corrections."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    E, B = case["edge"], case["batch"]
    V = E ** 3
    x = torch.zeros(B, V, 16, dtype=torch.float32, device=DEV)
    q = torch.arange(E, device=DEV, dtype=torch.float32)
    zz, yy, xx = (t.reshape(-1) for t in torch.meshgrid(q, q, q, indexing="ij"))
    R = E * (0.15 + 0.1 * torch.rand(B, 1, device=DEV, generator=gen))
    c = E / 2 + torch.rand(B, 3, device=DEV, generator=gen) - 0.5
    r = ((xx - c[:, :1]) ** 2 + (yy - c[:, 1:2]) ** 2 + (zz - c[:, 2:]) ** 2).sqrt()
    psi = torch.sigmoid((R - r) / 2)
    x[..., 0] = (1 - psi) * torch.tanh((zz - E / 2) / 4)
    x[..., 1] = psi
    x[..., 2:7] = 2 * torch.rand(B, 1, 5, device=DEV, generator=gen) - 1
    theta = []
    for t, ci, co in _layers(case):
        last = t == 1
        theta += [torch.randn(t * ci * co, device=DEV, generator=gen) * (0.1 if last else math.sqrt(2.0 / (t * ci))),
                  torch.randn(co, device=DEV, generator=gen) * 0.02]
    t0 = 0.1 * torch.randn(B, V, device=DEV, generator=gen)
    t1 = torch.zeros(B, V, device=DEV)
    sphere = torch.from_numpy(_unit_sphere(3)[0]).to(DEV, torch.float32)
    X0 = (c[:, None, :] + R[:, None] * sphere).contiguous()
    off = 0.3 * torch.randn(X0.shape, device=DEV, generator=gen)
    return x.to(torch.bfloat16), torch.cat(theta), t0, t1, X0, off


def _layers(case):
    """(taps, input channels, output channels) of the network's convolutions."""
    c = [case["channels"] * 2 ** k for k in range(case["levels"])]
    out = [(27, 16, c[0]), (27, c[0], c[0])]
    for k in range(1, len(c)):
        out += [(27, c[k - 1], c[k]), (27, c[k], c[k])]
    for k in range(len(c) - 2, -1, -1):
        out += [(27, c[k + 1] + c[k], c[k]), (27, c[k], c[k])]
    return out + [(1, c[0], 16)]


def prepare(case, seed):
    if case["kind"] == "run":
        wl = _workload(case, seed)
        start = _fields(case, wl, seed) if case["init"] != "plain" else None
        sim = Simulation(wl, device=DEV).init(*start or ())
        pin = {n: torch.empty(sim.N * (3 if n == "u" else 1), dtype=torch.float64, pin_memory=True)
               for n in ("phi", "psi", "u")}
        return {"case": case, "sim": sim, "pin": pin, "start": start if case["init"] == "restart" else None, "X0": [m.X for m in wl.membranes]}
    if case["kind"] == "batch":
        batch = Batch(_sweep(case, seed), device=DEV).init()
        pin = [torch.empty(wl.params.ncells, dtype=torch.float64, pin_memory=True) for wl in batch.wls]
        return {"case": case, "batch": batch, "pin": pin}
    x, theta, t0, t1, X0, off = _net_inputs(case, seed)
    net = WarmStartNet(case["edge"], case["channels"], case["levels"], max_batch=case["batch"],
                       max_nodes=X0.shape[1] if case["train"] else 0, device=DEV)
    net.set_params(theta.cpu().numpy())
    return {"case": case, "net": net, "x": x, "t0": t0, "t1": t1, "X0": X0, "off": off,
            "nn": [X0.shape[1]] * case["batch"]}


def run(state):
    case = state["case"]
    if case["kind"] == "run":
        sim, pin = state["sim"], state["pin"]
        if state["start"] is not None:
            for k, X in enumerate(state["X0"]):
                sim.set_nodes(k, X)
            sim.init(*state["start"])
        sim.step(case["steps"])
        out = {}
        for n in ("phi", "psi", "u"):
            sim.field(n, out=pin[n].numpy())
            out[n] = pin[n].to(OUT[case["storage"]])
        out["X"] = [_markers(sim, k, case) for k in range(case["caps"])]
        return out
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        psi, X = [], []
        for i in range(case["n"]):
            sim = batch[i]
            sim.field("psi", out=state["pin"][i].numpy())
            psi.append(state["pin"][i].to(OUT[case["storage"]]))
            X += [_markers(sim, k, case) for k in range(sim.n_mem)]
        return {"psi": psi, "X": torch.cat(X) if X else []}
    net = state["net"]
    if not case["train"]:
        return net.forward(state["x"])
    loss = net.train_step(state["x"], state["t0"], state["t1"], state["X0"], state["off"], state["nn"],
                          lam=1.0, lr=1e-4, update=True)
    return {"loss": torch.tensor(loss, dtype=torch.float32), "grads": net.grads()}


def _markers(sim, k, case):
    return torch.from_numpy(sim.nodes(k)).to(torch.float64 if case["storage"] == "f64" else torch.float32)


# --------------------------------------------------------------- work counted
def _cell_work(dim, storage, general, steps):
    """Per cell of a run: the state read once and written once in every step.
    At tau = 1 with the paper's forcing the state is 11 numbers a cell; any
    other run needs its 3Q populations.  Operations: both radius-1 stencils,
    the potentials and the equilibria of three sets, about 40 per velocity."""
    Q = 9 if dim == 2 else 19
    real = 8 if storage == "f64" else 4
    size = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[storage]
    state = (3 * Q - 2) * size + 2 * real if general else 11 * real
    return 2 * state * steps, 40 * Q * steps


def work(case):
    if case["kind"] == "net":
        E, B = case["edge"], case["batch"]
        edges = [E, E]
        for k in range(1, case["levels"]):
            edges += [E >> k, E >> k]
        for k in range(case["levels"] - 2, -1, -1):
            edges += [E >> k, E >> k]
        flops = sum(2 * B * e ** 3 * t * ci * co for e, (t, ci, co) in zip(edges + [E], _layers(case)))
        n = sum(t * ci * co + co for t, ci, co in _layers(case))
        first = 2 * B * E ** 3 * 27 * 16 * case["channels"]
        if case["train"]:
            return {"bytes": B * E ** 3 * (32 + 8) + 4 * n * 7, "flops": 3 * flops - first}
        return {"bytes": B * E ** 3 * (32 + 64) + 4 * n, "flops": flops}
    if case["kind"] == "run":
        cells = case["nx"] * case["ny"] * case["nz"]
        general = case["tau"] != 1.0 or case["forcing"] != "edm"
        b, f = _cell_work(2 if case["nz"] == 1 else 3, case["storage"], general, case["steps"])
        return {"bytes": cells * (b + 40), "flops": cells * f}
    cells = sum(wl.params.ncells for wl in _sweep(case, 0))
    b, f = _cell_work(case["dim"], case["storage"], False, case["steps"])
    return {"bytes": cells * (b + 8), "flops": cells * f}


# ------------------------------------------------------- the method in 64 bits
class _Exact:
    """The method in plain double precision: fields are arrays [z, y, x] (2D:
    [y, x]), velocities and marker axes are (x, y, z)."""

    def __init__(self, wl, start=None):
        p = self.p = wl.params
        self.dim = d = p.dim
        n3 = [(i, j, k) for k in (-1, 0, 1) for j in (-1, 0, 1) for i in (-1, 0, 1)]
        self.c = [c[:d] for c in n3 if (d == 3 or c[2] == 0) and sum(map(abs, c)) <= 2]
        w = {2: (4 / 9, 1 / 9, 1 / 36), 3: (1 / 3, 1 / 18, 1 / 36)}[d]
        self.w = [w[sum(map(abs, c))] for c in self.c]
        self.n = [p.nx, p.ny, p.nz][:d]
        self.shape = tuple(reversed(self.n))
        self.mem = wl.membranes
        self.X = [torch.from_numpy(m.X[:, :d].copy()).to(DEV) for m in self.mem]
        self.ref = [self._reference(m, X) for m, X in zip(self.mem, self.X)]
        self._profile()
        if start is None:
            z = torch.arange(self.shape[0], device=DEV, dtype=torch.float64).reshape(-1, *[1] * (d - 1))
            s = 0.5 * (1 + torch.tanh((z - p.interface_pos) / (2 * p.alpha)))
            s = s * (p.interface_pos >= 0)
            rho, psi = torch.ones(self.shape, device=DEV, dtype=torch.float64), self.I.clone()
            phi = (1 - psi) * (2 * s - 1)
            u = [torch.full_like(rho, p.u0[k]) for k in range(d)]
        else:
            C = [torch.from_numpy(v).to(DEV).reshape(self.shape) for v in start[0]]
            rho, phi, psi = C[0] + C[1] + C[2], C[0] - C[1], C[2]
            u = [torch.from_numpy(start[1][k]).to(DEV).reshape(self.shape) for k in range(d)]
        mu = self._potentials(rho, phi, psi)
        self.f = [self._feq(i, rho, u) for i in range(len(self.c))]
        self.g = self._oeq(phi, p.gamma_phi, mu[1], u)
        self.h = self._oeq(psi, p.gamma_psi, mu[2], u)

    # stencils: periodic, a mirror ghost at walls along the last axis
    def _at(self, a, c):
        if self.p.wall_last and c[-1]:
            a = torch.cat([a[1:], a[-1:]]) if c[-1] > 0 else torch.cat([a[:1], a[:-1]])
            c = (*c[:-1], 0)
        sh = [-v for v in reversed(c)]
        return torch.roll(a, sh, tuple(range(self.dim))) if any(sh) else a

    def _lap(self, a):
        return 6 * sum(w * (self._at(a, c) - a) for c, w in zip(self.c, self.w) if any(c))

    def _grad(self, a):
        out = [torch.zeros_like(a) for _ in range(self.dim)]
        for c, w in zip(self.c, self.w):
            if any(c):
                v = self._at(a, c)
                for k in range(self.dim):
                    if c[k]:
                        out[k] += 3 * w * c[k] * v
        return out

    def _potentials(self, rho, phi, psi):
        p = self.p
        A, B = rho + phi - psi, rho - phi - psi
        tA, tB = p.kappa1 / 8 * A * (A - 1) * (A - 2), p.kappa2 / 8 * B * (B - 1) * (B - 2)
        kp, km, q = p.kappa1 + p.kappa2, p.kappa2 - p.kappa1, p.alpha ** 2 / 4
        Lr, Lp, Ls = self._lap(rho), self._lap(phi), self._lap(psi)
        return (tA + tB + q * (kp * (Ls - Lr) + km * Lp), tA - tB + q * (km * (Lr - Ls) - kp * Lp),
                -tA - tB + q * (kp * Lr - km * Lp - (kp + 4 * p.kappa3) * Ls)
                + p.kappa3 * psi * (psi - 1) * (2 * psi - 1) + p.kappa_c * (psi - self.I))

    def _poly(self, i, v):
        cv = sum(ci * vi for ci, vi in zip(self.c[i], v) if ci) if any(self.c[i]) else 0.0
        return 3 * cv + 4.5 * cv * cv - 1.5 * sum(vi * vi for vi in v)

    def _feq(self, i, rho, v):
        return self.w[i] * rho * (1 + self._poly(i, v))

    def _oeq(self, a, gam, mu, v):
        out = [self.w[i] * (3 * gam * mu + a * self._poly(i, v)) for i in range(len(self.c))]
        rest = next(i for i, c in enumerate(self.c) if not any(c))
        out[rest] = a - sum(o for i, o in enumerate(out) if i != rest)
        return out

    def _stream(self, f):
        out = []
        for i, c in enumerate(self.c):
            a = torch.roll(f[i], tuple(reversed(c)), tuple(range(self.dim))) if any(c) else f[i]
            if self.p.wall_last and c[-1]:  # halfway bounce-back
                o = self.c.index(tuple(-v for v in c))
                a[0 if c[-1] > 0 else -1] = f[o][0 if c[-1] > 0 else -1]
            out.append(a)
        return out

    def _momentum(self):
        return [sum(c[k] * f for c, f in zip(self.c, self.f) if c[k]) for k in range(self.dim)]

    # membranes
    def _reference(self, m, X):
        if self.dim == 2:
            return (X.roll(-1, 0) - X).norm(dim=1)
        T = torch.from_numpy(m.elems.astype(np.int64)).to(DEV)
        a, b, c = X[T[:, 0]], X[T[:, 1]], X[T[:, 2]]
        e, f = b - a, c - a
        G = torch.stack([(e * e).sum(1), (e * f).sum(1), (f * f).sum(1)], 1)
        return T, G, G[:, 0] * G[:, 2] - G[:, 1] ** 2

    def _energy(self, m, ref, X):
        if self.dim == 2:
            a, b = X.roll(-1, 0) - X, X - X.roll(1, 0)
            la, lb = a.norm(dim=1), b.norm(dim=1)
            th = torch.atan2(a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0], (a * b).sum(1))
            return (0.5 * m.ks * (la / ref - 1) ** 2 * ref + m.kb * th * th / (la + lb)).sum()
        T, G, det0 = ref
        x = [X[T[:, k]] for k in range(3)]
        e, f = x[1] - x[0], x[2] - x[0]
        g11, g12, g22 = (e * e).sum(1), (e * f).sum(1), (f * f).sum(1)
        I1 = (G[:, 2] * g11 - 2 * G[:, 1] * g12 + G[:, 0] * g22) / det0 - 2
        I2 = (g11 * g22 - g12 * g12) / det0 - 1
        E = (0.5 * det0.sqrt() * m.G / 4 * (I1 ** 2 + 2 * I1 - 2 * I2 + m.C * I2 ** 2)).sum()
        area = 0.5 * torch.linalg.cross(e, f).norm(dim=1)
        dot = [((x[(k + 1) % 3] - x[k]) * (x[(k + 2) % 3] - x[k])).sum(1) for k in range(3)]
        cot = [v / (2 * area) for v in dot]
        obtuse = (dot[0] < 0) | (dot[1] < 0) | (dot[2] < 0)
        K, A = torch.zeros_like(X), torch.zeros_like(X[:, 0])
        for k in range(3):
            j, l = (k + 1) % 3, (k + 2) % 3
            vj, vl = x[k] - x[j], x[k] - x[l]
            K = K.index_add(0, T[:, k], cot[l][:, None] * vj + cot[j][:, None] * vl)
            vor = 0.125 * ((vj * vj).sum(1) * cot[l] + (vl * vl).sum(1) * cot[j])
            A = A.index_add(0, T[:, k], torch.where(obtuse, torch.where(dot[k] < 0, 0.5, 0.25) * area, vor))
        return E + (m.kb / 8 * (K * K).sum(1) / A).sum()

    @staticmethod
    def _segment(q, a, b):
        e = b - a
        t = (((q - a) * e).sum(-1) / (e * e).sum(-1)).clamp(0, 1)
        return t, (q - a - t[..., None] * e)

    def _closest(self, m, ref, X, q):
        """Per point of q: the nearest element's nodes, the weights of its
        closest point, and the vector from that point."""
        out = []
        for part in q.split(20000):
            if self.dim == 2:
                a, b = X[None], X.roll(-1, 0)[None]
                t, r = self._segment(part[:, None], a, b)
                e = (r * r).sum(-1).argmin(1)
                i = torch.arange(len(part), device=DEV)
                t, r = t[i, e], r[i, e]
                nodes, beta = torch.stack([e, (e + 1) % len(X)], 1), torch.stack([1 - t, t], 1)
            else:
                T = ref[0]
                mid = (X[T[:, 0]] + X[T[:, 1]] + X[T[:, 2]]) / 3
                near = torch.cdist(part, mid).topk(min(32, len(T)), dim=1, largest=False).indices
                x = [X[T[near, k]] for k in range(3)]
                e1, e2, qa = x[1] - x[0], x[2] - x[0], part[:, None] - x[0]
                d11, d12, d22 = (e1 * e1).sum(-1), (e1 * e2).sum(-1), (e2 * e2).sum(-1)
                q1, q2 = (qa * e1).sum(-1), (qa * e2).sum(-1)
                den = d11 * d22 - d12 * d12
                v, w = (d22 * q1 - d12 * q2) / den, (d11 * q2 - d12 * q1) / den
                inside = (v >= 0) & (w >= 0) & (v + w <= 1)
                beta = torch.stack([1 - v - w, v, w], -1)
                dist = torch.where(inside, (qa - v[..., None] * e1 - w[..., None] * e2).norm(dim=-1), torch.inf)
                for k in range(3):
                    l = (k + 1) % 3
                    t, r = self._segment(part[:, None], x[k], x[l])
                    be = torch.zeros_like(beta)
                    be[..., k], be[..., l] = 1 - t, t
                    better = (r.norm(dim=-1) < dist) & ~inside
                    beta = torch.where(better[..., None], be, beta)
                    dist = torch.where(better, r.norm(dim=-1), dist)
                e = dist.argmin(1)
                i = torch.arange(len(part), device=DEV)
                nodes, beta = T[near[i, e]], beta[i, e]
                r = part - (beta[..., None] * X[nodes]).sum(1)
            out.append((nodes, beta, r))
        return [torch.cat(v) for v in zip(*out)]

    def _normals(self, ref, X):
        if self.dim == 2:
            t = X.roll(-1, 0) - X
            n = torch.stack([t[:, 1], -t[:, 0]], 1) / t.norm(dim=1, keepdim=True)
            return n + n.roll(1, 0)
        T = ref[0]
        n = torch.linalg.cross(X[T[:, 1]] - X[T[:, 0]], X[T[:, 2]] - X[T[:, 0]])
        out = torch.zeros_like(X)
        for k in range(3):
            out.index_add_(0, T[:, k], n)
        return out / out.norm(dim=1, keepdim=True)

    def _profile(self):
        """I(x) from the signed distance to the nearest membrane (positive
        inside, clamped to dc), and the band |d| < dc with its owners."""
        p, dc = self.p, self.p.dc
        d = torch.full(self.shape, -dc, device=DEV, dtype=torch.float64).reshape(-1)
        cell = torch.stack([t.reshape(-1) for t in reversed(torch.meshgrid(
            *[torch.arange(v, device=DEV, dtype=torch.float64) for v in self.shape], indexing="ij"))], 1)
        n = torch.tensor([float(v) for v in self.n], device=DEV)
        if p.wall_last:
            n[-1] = torch.inf
        owner = torch.full_like(d, -1, dtype=torch.long)
        band = []
        for k, (m, ref, X) in enumerate(zip(self.mem, self.ref, self.X)):
            mid, far = X.mean(0), (X - X.mean(0)).norm(dim=1)
            q = cell - mid
            q = torch.where(torch.isfinite(n), q - n * torch.round(q / n), q)
            r = q.norm(dim=1)
            near = torch.nonzero((r < far.max() + dc) & (r > far.min() - dc - 2)).reshape(-1)
            nodes, beta, rel = self._closest(m, ref, X, q[near] + mid)
            dist = rel.norm(dim=1)
            out = (rel * (beta[..., None] * self._normals(ref, X)[nodes]).sum(1)).sum(1)
            dk = torch.full_like(d, -dc)
            dk[r <= far.min() - dc - 2] = dc
            dk[near] = torch.where(out > 0, -dist, dist).clamp(-dc, dc)
            better = dk > d
            d = torch.where(better, dk, d)
            owner[better] = k
            band.append((near, nodes, beta, rel, dist))
        self.I = (0.5 * (1 + torch.tanh(d / (2 * p.alpha)))).reshape(self.shape)
        self.d, self.owner, self.band = d, owner, band

    def _coupling(self, k, psi):
        p = self.p
        near, nodes, beta, rel, dist = self.band[k]
        d = self.d[near]
        use = (self.owner[near] == k) & (d.abs() < p.dc)
        near, nodes, beta, rel, dist, d = (t[use] for t in (near, nodes, beta, rel, dist, d))
        coef = p.kappa_c * (psi.reshape(-1)[near] - self.I.reshape(-1)[near]) / torch.cosh(d / (2 * p.alpha)) ** 2 / (4 * p.alpha)
        vec = -(coef * torch.sign(d) / dist)[:, None] * rel
        out = torch.zeros_like(self.X[k])
        for j in range(nodes.shape[1]):
            out.index_add_(0, nodes[:, j], beta[:, j:j + 1] * vec)
        return out

    def _support(self, X):
        """Cells and weights of the immersed boundary kernel at markers X."""
        base = torch.floor(X).long() - 1
        cell, wt = torch.zeros(len(X), 1, device=DEV, dtype=torch.long), torch.ones(len(X), 1, device=DEV, dtype=torch.float64)
        for k in reversed(range(self.dim)):
            q = base[:, k:k + 1] + torch.arange(4, device=DEV)
            a = (q - X[:, k:k + 1]).abs()
            near = (3 - 2 * a + (1 + 4 * a - 4 * a * a).clamp(min=0).sqrt()) / 8
            far = (5 - 2 * a - (-7 + 12 * a - 4 * a * a).clamp(min=0).sqrt()) / 8
            w = torch.where(a <= 1, near, torch.where(a <= 2, far, 0.0))
            if self.p.wall_last and k == self.dim - 1:
                w = torch.where((q >= 0) & (q < self.n[k]), w, 0.0)
                q = q.clamp(0, self.n[k] - 1)
            q = q % self.n[k]
            cell = (cell[:, :, None] * self.n[k] + q[:, None, :]).reshape(len(X), -1)
            wt = (wt[:, :, None] * w[:, None, :]).reshape(len(X), -1)
        return cell, wt

    def step(self):
        p, d = self.p, self.dim
        rho, phi, psi, j = sum(self.f), sum(self.g), sum(self.h), self._momentum()
        mu = self._potentials(rho, phi, psi)
        gr = [self._grad(m) for m in mu]
        Ft = [-rho * gr[0][k] - phi * gr[1][k] - psi * gr[2][k] for k in range(d)]
        support = []
        for k, m in enumerate(self.mem):
            X = self.X[k].clone().requires_grad_(True)
            Fm = self._coupling(k, psi) - torch.autograd.grad(self._energy(m, self.ref[k], X), X)[0]
            cell, wt = self._support(self.X[k])
            support.append((cell, wt))
            for a in range(d):
                Ft[a].view(-1).index_add_(0, cell.reshape(-1), (wt * Fm[:, a:a + 1]).reshape(-1))
        u = [v / rho for v in j]
        v = [(jk + 0.5 * Fk) / rho for jk, Fk in zip(j, Ft)]
        ud = [(jk + Fk) / rho for jk, Fk in zip(j, Ft)]
        vF = sum(a * b for a, b in zip(v, Ft))
        ge, he = self._oeq(phi, p.gamma_phi, mu[1], v), self._oeq(psi, p.gamma_psi, mu[2], v)
        for i, c in enumerate(self.c):
            if p.forcing == "guo":
                cF = sum(ck * Fk for ck, Fk in zip(c, Ft) if ck) if any(c) else 0.0
                cv = sum(ck * vk for ck, vk in zip(c, v) if ck) if any(c) else 0.0
                self.f[i] = (self.f[i] - (self.f[i] - self._feq(i, rho, v)) / p.tau
                             + (1 - 0.5 / p.tau) * self.w[i] * (3 * (cF - vF) + 9 * cv * cF))
            else:
                fe = self._feq(i, rho, u)
                self.f[i] = self.f[i] - (self.f[i] - fe) / p.tau + self._feq(i, rho, ud) - fe
            self.g[i] = self.g[i] - (self.g[i] - ge[i]) / p.tau_phi
            self.h[i] = self.h[i] - (self.h[i] - he[i]) / p.tau_psi
        self.f, self.g, self.h = self._stream(self.f), self._stream(self.g), self._stream(self.h)
        if self.mem:
            rho, j = sum(self.f), self._momentum()
            v = [((j[k] + 0.5 * Ft[k]) / rho).reshape(-1) for k in range(d)]
            for k in range(len(self.mem)):
                cell, wt = support[k]
                self.X[k] = self.X[k] + torch.stack([(wt * v[a][cell]).sum(1) for a in range(d)], 1)
            self._profile()

    def markers(self, k):
        return F.pad(self.X[k], (0, 3 - self.dim))

    def velocity(self):
        rho, j = sum(self.f), self._momentum()
        out = torch.zeros(3, rho.numel(), device=DEV, dtype=torch.float64)
        for k in range(self.dim):
            out[k] = (j[k] / rho).reshape(-1)
        return out.reshape(-1)


def _exact_net(case, seed):
    x, theta, t0, t1, X0, off = _net_inputs(case, seed)
    E, B = case["edge"], case["batch"]
    theta = theta.double().requires_grad_(case["train"])
    par, o = [], 0
    for t, ci, co in _layers(case):
        k = 3 if t == 27 else 1
        par.append((theta[o:o + t * ci * co].reshape(k, k, k, ci, co).permute(4, 3, 0, 1, 2), theta[o + t * ci * co:o + t * ci * co + co]))
        o += t * ci * co + co
    it = iter(par)

    def conv(h):
        w, b = next(it)
        return F.conv3d(h, w, b, padding=w.shape[-1] // 2)

    h, enc = x.double().reshape(B, E, E, E, 16).permute(0, 4, 1, 2, 3), []
    for k in range(case["levels"]):
        h = F.avg_pool3d(h, 2) if k else h
        h = torch.relu(conv(torch.relu(conv(h))))
        enc.append(h)
    for k in range(case["levels"] - 2, -1, -1):
        h = torch.cat([F.interpolate(h, scale_factor=2, mode="nearest"), enc[k]], 1)
        h = torch.relu(conv(torch.relu(conv(h))))
    y = conv(h).permute(0, 2, 3, 4, 1).reshape(B, E ** 3, 16)
    if not case["train"]:
        return y
    loss = ((y[..., 0] - t0.double()) ** 2 + (y[..., 1] - t1.double()) ** 2).mean()
    X = X0.double().clamp(0, E - 1)
    i0 = X.floor().clamp(0, E - 2).long()
    fr = X - i0
    disp = 0.0
    for c in ((i, j, k) for i in (0, 1) for j in (0, 1) for k in (0, 1)):
        wt = math.prod(fr[..., a] if c[a] else 1 - fr[..., a] for a in range(3))
        n = ((i0[..., 2] + c[2]) * E + i0[..., 1] + c[1]) * E + i0[..., 0] + c[0]
        disp = disp + wt[..., None] * torch.gather(y[..., 2:5], 1, n[..., None].expand(-1, -1, 3))
    loss = loss + ((disp - off.double()) ** 2).mean()
    return {"loss": loss.detach(), "grads": torch.autograd.grad(loss, theta)[0]}


def exact(case, seed):
    if case["kind"] == "net":
        return _exact_net(case, seed)
    if case["kind"] == "run":
        wl = _workload(case, seed)
        if wl.params.ncells * case["steps"] > 2.2e8:  # tens of seconds
            return None
        e = _Exact(wl, _fields(case, wl, seed) if case["init"] != "plain" else None)
        for _ in range(case["steps"]):
            e.step()
        return {"phi": sum(e.g).reshape(-1), "psi": sum(e.h).reshape(-1), "u": e.velocity(),
                "X": [e.markers(k) for k in range(case["caps"])]}
    wls = _sweep(case, seed)
    if sum(wl.params.ncells for wl in wls) * case["steps"] > 2.2e8:
        return None
    psi, X = [], []
    for wl in wls:
        e = _Exact(wl)
        for _ in range(case["steps"]):
            e.step()
        psi.append(sum(e.h).reshape(-1))
        X += [e.markers(k) for k in range(len(wl.membranes))]
    return {"psi": psi, "X": torch.cat(X) if X else []}
