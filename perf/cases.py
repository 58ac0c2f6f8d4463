"""The work a user has the solver do, as measurable cases.

listed() names the cases, draw() gives more of the same ranges, prepare()
makes a case's inputs and solver on the GPU, run() is one pass through the
public entry points, work() its necessary traffic and arithmetic, and exact()
the same pass in plain FP64 torch, without this repository's code.

Three kinds of pass:
  flow      Simulation: initial fields in, `steps` steps, macroscopic fields out
  batch     Batch: the same for many independent runs stepped together
  gradient  cbc_loss_adjoint: the pressure loss and its gradient with respect
            to the five relaxation parameters (forward and backward)
Fields are returned in the storage's own precision.
"""
import math
import random

import numpy as np
import torch

import paper_2307_16766_gb300 as lbm

CS2 = {"D2Q9": 1.0 / 3.0, "D2Q17": 0.3702518670183398497189151, "D2Q37": 0.6979533220196830882384091}
LAYERS = {"D2Q9": 1, "D2Q17": 3, "D2Q37": 3}
SIZE = {"f64": 8, "f32": 4, "f16": 2}
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}


def _flow(name, lattice, nx, ny, storage, shape, sides, steps, tau, **more):
    c = {"kind": "flow", "lattice": lattice, "nx": nx, "ny": ny, "storage": storage, "shape": shape, "sides": sides,
         "steps": steps, "tau": tau, "scheme": "cbc_relax", "viscous": "meso", "dirichlet": "eq", "alpha_T": 0.0,
         "mach": 0.0, "ref": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest workload: isothermal pulse between four characteristic sides, the first parity configuration
        _flow("pulse_d2q9_64_f64", "D2Q9", 64, 64, "f64", "pulse", "cbc cbc cbc cbc", 200, 0.6, scheme="cbc", viscous="fd"),
        # temperature step carried through two artificial sides (the paper's Sec. 4.1), with the NEEP write
        _flow("step_d2q17_200x20_f64", "D2Q17", 200, 20, "f64", "step", "cbc cbc periodic periodic", 100, 0.9,
              scheme="cbc", dirichlet="neep", mach=0.1),
        # thermal vortex on an odd-sized third-order grid, relaxed outlet (Sec. 4.2)
        _flow("vortex_d2q17_150_f64", "D2Q17", 150, 150, "f64", "vortex", "cbc cbc cbc cbc", 100, 0.77, alpha_T=0.1,
              mach=0.1, scheme="lodi cbc_relax lodi lodi"),
        # the 256^2 pulse between four characteristic sides in single precision
        _flow("pulse_d2q37_256_f32", "D2Q37", 256, 256, "f32", "pulse", "cbc cbc cbc cbc", 100, 0.8, alpha_T=0.5),
        # the benchmark workload: a vortex carried by a stream, inflow and characteristic outlet
        _flow("vortex_d2q37_1024x512_f32", "D2Q37", 1024, 512, "f32", "vortex", "inflow cbc periodic periodic", 100, 0.8,
              alpha_T=0.1, mach=0.1),
        # the same with the populations held relative to the stream's equilibrium (long runs)
        _flow("vortex_d2q37_1024x512_f32_ref", "D2Q37", 1024, 512, "f32", "vortex", "inflow cbc periodic periodic", 100,
              0.8, alpha_T=0.1, mach=0.1, ref=True),
        # the same in double precision
        _flow("vortex_d2q37_1024x512_f64", "D2Q37", 1024, 512, "f64", "vortex", "inflow cbc periodic periodic", 20, 0.8,
              alpha_T=0.1, mach=0.1),
        # the largest pulse grid
        _flow("pulse_d2q37_4096_f32", "D2Q37", 4096, 4096, "f32", "pulse", "cbc cbc cbc cbc", 20, 0.8, alpha_T=0.5),
        # the largest vortex grid in half-precision storage
        _flow("vortex_d2q37_4096_f16", "D2Q37", 4096, 4096, "f16", "vortex", "inflow cbc periodic periodic", 20, 0.8,
              alpha_T=0.1, mach=0.1),
        # a periodic reference run, several times larger than the domain it is cropped to
        _flow("periodic_d2q37_2048x1024_f32", "D2Q37", 2048, 1024, "f32", "pulse", "periodic periodic periodic periodic",
              40, 0.8),
        # the coefficient sweep: 96 runs of uneven sizes on two lattices
        {"name": "sweep_96_f32", "kind": "batch", "runs": 96, "lo": 128, "hi": 512, "storage": "f32", "steps": 40},
        # gradient of the reflection energy with respect to the relaxation parameters
        {"name": "gradient_d2q37_512x256_f32", "kind": "gradient", "lattice": "D2Q37", "nx": 512, "ny": 256,
         "storage": "f32", "steps": 60, "every": 20, "tau": 0.8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small", "medium", "medium", "large", "periodic", "batch", "gradient"])
    if kind == "small":
        lattice = rng.choice(["D2Q9", "D2Q17", "D2Q37"])
        sides = rng.choice(["cbc cbc cbc cbc", "cbc cbc periodic periodic", "inflow cbc periodic periodic",
                            "zg zg periodic periodic"])
        # a viscous vector needs a flow through the side; its -FD form a small viscosity
        viscous = "off" if sides == "cbc cbc cbc cbc" else rng.choice(["meso", "off" if lattice == "D2Q37" else "fd"])
        return _flow("", lattice, _log(rng, 40, 400), _log(rng, 40, 400), rng.choice(["f64", "f32"]),
                     "pulse" if sides == "cbc cbc cbc cbc" else rng.choice(["pulse", "vortex"]), sides,
                     rng.randint(50, 200), round(rng.uniform(0.6, 0.95), 3),
                     scheme=rng.choice(["lodi", "lodi_relax", "cbc_relax"]), viscous=viscous,
                     dirichlet=rng.choice(["eq", "neep"]), alpha_T=round(rng.uniform(0.2, 0.8), 3), mach=0.1)
    if kind in ("medium", "large"):
        storage = rng.choice(["f32", "f16", "f64"] if kind == "medium" else ["f32", "f16"])
        nx, ny = (_log(rng, 400, 1600), _log(rng, 300, 1200)) if kind == "medium" else (_log(rng, 1600, 4096), _log(rng, 1200, 4096))
        still = rng.random() < 0.5
        return _flow("", "D2Q37", nx, ny, storage, "pulse" if still else "vortex",
                     "cbc cbc cbc cbc" if still else "inflow cbc periodic periodic",
                     rng.randint(10, 20) if kind == "large" or storage == "f64" else rng.randint(40, 100), 0.8, alpha_T=0.5 if still else 0.1,
                     mach=0.0 if still else 0.1, ref=not still and storage != "f64" and rng.random() < 0.5)
    if kind == "periodic":
        return _flow("", rng.choice(["D2Q37", "D2Q17"]), _log(rng, 200, 3000), _log(rng, 200, 1500),
                     rng.choice(["f32", "f64"]), "pulse", "periodic periodic periodic periodic", rng.randint(10, 20), 0.8)
    if kind == "batch":
        return {"kind": "batch", "runs": rng.randint(12, 96), "lo": 64, "hi": rng.randint(200, 512), "storage": "f32",
                "steps": rng.randint(20, 40)}
    return {"kind": "gradient", "lattice": rng.choice(["D2Q37", "D2Q17"]), "nx": _log(rng, 100, 512), "ny": _log(rng, 80, 256),
            "storage": "f32", "steps": rng.randint(24, 60), "every": rng.randint(8, 30), "tau": 0.8}


# ------------------------------------------------------------------ inputs ---

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fields(shape, lattice, nx, ny, mach, rnd):
    """(rho, ux, uy, T): a pulse, a vortex in a stream or a temperature step, placed and sized by the seed."""
    dev = _device()
    x = torch.arange(nx, dtype=torch.float64, device=dev)[None, :]
    y = torch.arange(ny, dtype=torch.float64, device=dev)[:, None]
    one = torch.ones(ny, nx, dtype=torch.float64, device=dev)
    u0 = mach * math.sqrt(CS2[lattice])
    cx = (nx - 1) * rnd.uniform(0.3, 0.7)
    cy = (ny - 1) * rnd.uniform(0.3, 0.7)
    thermal = lattice != "D2Q9"
    if shape == "step":
        s, T1 = 0.5, 1.0 + rnd.uniform(3e-4, 7e-4)
        T = 1.0 + 0.5 * (T1 - 1.0) * (torch.tanh(s * (x - 0.25 * nx)) - torch.tanh(s * (x - rnd.uniform(0.7, 0.8) * nx)))
        # a slight shear along the step, so that the transversal velocity carries a signal
        return one.clone(), one * u0, one * (0.02 * u0 * torch.sin(2.0 * math.pi * y / ny)), one * T
    if shape == "pulse":
        w, a = rnd.uniform(5.0, 10.0), rnd.uniform(0.5e-3, 1.5e-3)
        G = torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2.0 * w * w))
        return 1.0 + a * G, one * u0, one * (0.6 * u0), 1.0 + (a * G if thermal else 0.0 * G)
    R, eps = rnd.uniform(0.04, 0.12) * min(nx, ny, 400), rnd.uniform(0.03, 0.07) * max(u0, 0.05)
    dx, dy = (x - cx) / R, (y - cy) / R
    e = torch.exp(0.5 * (1.0 - dx * dx - dy * dy))
    T = 1.0 - 0.25 * eps * eps * e * e / CS2[lattice]
    return T.clone(), u0 - eps * dy * e, eps * dx * e, (T if thermal else one)


def _config(case):
    lat = case["lattice"]
    u0 = case["mach"] * math.sqrt(CS2[lat])
    return {"lattice": lat, "nx": case["nx"], "ny": case["ny"], "tau": case["tau"], "rho0": 1.0,
            "sides": case["sides"].split(), "schemes": (case["scheme"].split() * 4)[:4], "viscous": case["viscous"],
            "dirichlet": case["dirichlet"], "alpha_T": case["alpha_T"], "beta_P": 0.0, "t_inf": 0.0, "alpha_V": 0.0,
            "p_inf": [CS2[lat]] * 4, "inflow": [1.0, u0, 0.0, 1.0], "storage": case["storage"],
            "u_ref": [u0 if case["ref"] else 0.0, 0.0]}


def _flow_inputs(case, seed):
    rnd = random.Random(seed)
    return _config(case), _fields(case["shape"], case["lattice"], case["nx"], case["ny"], case["mach"], rnd)


def _batch_inputs(case, seed):
    """Run descriptions (fixed by the case: a program keeps its batch) and fields (by the seed)."""
    lay, rnd = random.Random(case["runs"] * 1000 + case["hi"]), random.Random(seed)
    cfgs, fields = [], []
    for _ in range(case["runs"]):
        lat = "D2Q37" if lay.random() < 0.5 else "D2Q9"
        nx, ny = lay.randint(case["lo"], case["hi"]), lay.randint(case["lo"], case["hi"])
        cfgs.append(_config({"lattice": lat, "nx": nx, "ny": ny, "tau": lay.uniform(0.55, 1.0), "sides": "cbc cbc cbc cbc",
                             "scheme": "cbc_relax", "viscous": "meso", "dirichlet": "eq", "alpha_T": lay.random(),
                             "mach": 0.0, "storage": case["storage"], "ref": False}))
        cfgs[-1]["beta_P"] = lay.random()
        fields.append(_fields("pulse", lat, nx, ny, 0.0, rnd))
    return cfgs, fields


def _gradient_inputs(case, seed):
    """A pulse next to two sides in a stream oblique to them, and the pressure an open domain would show (an outgoing ring)."""
    rnd = random.Random(seed)
    lat, nx, ny = case["lattice"], case["nx"], case["ny"]
    cfg = _config({"lattice": lat, "nx": nx, "ny": ny, "tau": case["tau"], "sides": "cbc cbc cbc cbc", "scheme": "cbc_relax",
                   "viscous": "meso", "dirichlet": "eq", "alpha_T": 0.0, "mach": 0.0, "storage": case["storage"],
                   "ref": False})
    dev, cs = _device(), math.sqrt(CS2[lat])
    x = torch.arange(nx, dtype=torch.float64, device=dev)[None, :]
    y = torch.arange(ny, dtype=torch.float64, device=dev)[:, None]
    cx, cy, w, a = nx - rnd.uniform(20.0, 28.0), ny - rnd.uniform(20.0, 28.0), 8.0, rnd.uniform(0.8e-3, 1.2e-3)
    r2 = (x - cx) ** 2 + (y - cy) ** 2
    G = torch.exp(-r2 / (2.0 * w * w))
    one = torch.ones_like(G)
    fields = (1.0 + a * G, one * (0.05 * cs), one * (0.03 * cs), 1.0 + a * G)
    t = torch.arange(1, case["steps"] + 1, dtype=torch.float64, device=dev)[:, None, None]
    r = torch.sqrt(r2)[None]
    ref = a * CS2[lat] * torch.exp(-(r - math.sqrt(2.0) * cs * t) ** 2 / (2.0 * w * w)) / torch.sqrt(1.0 + r / w)
    theta = [rnd.uniform(0.3, 0.6), rnd.uniform(0.3, 0.6), CS2[lat] * (1.0 + rnd.uniform(-2e-4, 2e-4)), rnd.uniform(0.2, 0.4),
             rnd.uniform(-1e-5, 1e-5)]
    return cfg, fields, ref, torch.tensor(theta, dtype=torch.float32, device=dev)


def prepare(case, seed):
    if case["kind"] == "flow":
        cfg, fields = _flow_inputs(case, seed)
        return {"case": case, "sim": lbm.Simulation(cfg), "fields": fields}
    if case["kind"] == "batch":
        cfgs, fields = _batch_inputs(case, seed)
        return {"case": case, "batch": lbm.Batch(cfgs), "fields": fields}
    cfg, fields, ref, theta = _gradient_inputs(case, seed)
    return {"case": case, "cfg": cfg, "fields": fields, "ref": ref, "theta": theta}


def run(state):
    case = state["case"]
    if case["kind"] == "flow":
        sim = state["sim"]
        sim.init_fields(*state["fields"])
        sim.step(case["steps"])
        return [a.to(DTYPE[case["storage"]]) for a in sim.macros(device=True)]
    if case["kind"] == "batch":
        batch = state["batch"]
        for r, f in enumerate(state["fields"]):
            batch[r].init_fields(*f)
        batch.step(case["steps"])
        out = [batch[r].macros(device=True) for r in range(len(batch))]
        return [torch.cat([o[k].reshape(-1) for o in out]).to(DTYPE[case["storage"]]) for k in range(4)]
    theta = state["theta"].detach().clone().requires_grad_(True)
    J = lbm.cbc_loss_adjoint(theta, state["cfg"], state["fields"], case["steps"], state["ref"],
                             checkpoint_every=case["every"])
    J.backward()
    return [J.detach(), theta.grad]


# -------------------------------------------------------------- necessities ---

# arithmetic of one node's moments, equilibrium and collision
FLOPS = {"D2Q9": 130, "D2Q17": 330, "D2Q37": 735}


def work(case):
    """Every step reads and writes each population once; the initial and final fields are FP64 in, FP64 out."""
    if case["kind"] == "batch":
        runs = [(c["lattice"], c["nx"] * c["ny"]) for c in _batch_shapes(case)]
    else:
        runs = [(case["lattice"], case["nx"] * case["ny"])]
    b = f = 0.0
    for lat, n in runs:
        Q = int(lat[3:])
        b += case["steps"] * 2.0 * Q * SIZE[case["storage"]] * n + 64.0 * n
        f += case["steps"] * float(FLOPS[lat]) * n
    if case["kind"] == "gradient":
        # forward, forward again from the checkpoints, and the reverse step's own populations; the reference twice
        n = runs[0][1]
        b = 3.0 * b + case["steps"] * 16.0 * n
        f = 4.0 * f
    return {"bytes": b, "flops": f}


def _batch_shapes(case):
    lay, out = random.Random(case["runs"] * 1000 + case["hi"]), []
    for _ in range(case["runs"]):
        lat = "D2Q37" if lay.random() < 0.5 else "D2Q9"
        out.append({"lattice": lat, "nx": lay.randint(case["lo"], case["hi"]), "ny": lay.randint(case["lo"], case["hi"])})
        lay.uniform(0.55, 1.0), lay.random(), lay.random()
    return out


# ------------------------------------------------------------ the same in FP64 ---

W37 = [0.23315066913235250229, 0.10730609154221900241, 0.05766785988879488203, 0.014208216158450750265,
       0.0053530490005137752327, 0.0010119375926735754754, 0.00024530102775771734547, 0.0002834142529941982174]
W17 = [0.4020051469091126259416644, 0.1161548664977815438740355, 0.0330063536229869139497538,
       0.0000790786021659181312371, 0.0002584145497874675595575]
W9 = [4.0 / 9.0, 1.0 / 9.0, 1.0 / 36.0]
# velocity classes (|c_x|, |c_y|), in the order of the weights
CLASSES = {"D2Q9": [(0, 0), (1, 0), (1, 1)], "D2Q17": [(0, 0), (1, 0), (1, 1), (2, 2), (3, 0)],
           "D2Q37": [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 0), (3, 1)]}
WEIGHTS = {"D2Q9": W9, "D2Q17": W17, "D2Q37": W37}
NORMAL = [(-1, 0), (1, 0), (0, -1), (0, 1)]      # outward normals of W, E, S, N
TANGENT = [(0, 1), (0, 1), (1, 0), (1, 0)]


class _Plain:
    """The method in FP64 torch operations: pull, BGK, the layer-wise characteristic condition and its Dirichlet write."""

    def __init__(self, cfg):
        self.cfg, self.lat = cfg, cfg["lattice"]
        self.cs2, self.M = CS2[self.lat], LAYERS[self.lat]
        self.thermal, self.order = self.lat != "D2Q9", {"D2Q9": 2, "D2Q17": 3, "D2Q37": 4}[self.lat]
        self.nx, self.ny, self.tau = cfg["nx"], cfg["ny"], cfg["tau"]
        dev = self.dev = _device()
        c, w = [], []
        for (a, b), wk in zip(CLASSES[self.lat], WEIGHTS[self.lat]):
            for v in sorted({(p * x, q * y) for x, y in ((a, b), (b, a)) for p in (1, -1) for q in (1, -1)}):
                c.append(v)
                w.append(wk)
        self.c = torch.tensor(c, dtype=torch.float64, device=dev)
        self.w = torch.tensor(w, dtype=torch.float64, device=dev)[:, None]
        self.shifts, self.c2 = c, (self.c ** 2).sum(1)[:, None]
        self._boundary()

    # -- populations: g = f - w (rho0 = 1), [Q, n]
    def moments(self, g):
        s0 = g.sum(0)
        s = torch.matmul(self.c.T, g)
        rho = 1.0 + s0
        u = s / rho
        if not self.thermal:
            return s0, u[0], u[1], torch.zeros_like(s0)
        e = (self.c2 * g).sum(0)
        return s0, u[0], u[1], (e - rho * (u * u).sum(0) - 2.0 * self.cs2 * s0) / (2.0 * self.cs2 * rho)

    def equilibrium(self, U):
        s0, ux, uy, t = U
        u2 = (ux * ux + uy * uy) / self.cs2
        p = torch.matmul(self.c / self.cs2, torch.stack([ux, uy]))
        x = self.c2 / self.cs2
        if self.order == 2:
            poly = -0.5 * u2 + p * (1.0 + 0.5 * p)
        elif self.order == 3:
            poly = 0.5 * t * (x - 2.0) - 0.5 * u2 + p * (1.0 - 0.5 * u2 + 0.5 * t * (x - 4.0) + p * (0.5 + p / 6.0))
        else:
            a0 = -0.5 * u2 + 0.125 * u2 * u2 + 0.5 * t * (x - 2.0) - 0.25 * t * u2 * (x - 4.0) + 0.125 * t * t * ((x - 8.0) * x + 8.0)
            a1 = 1.0 - 0.5 * u2 + 0.5 * t * (x - 4.0)
            a2 = 0.5 - 0.25 * u2 + 0.25 * t * (x - 6.0)
            poly = a0 + p * (a1 + p * (a2 + p * (1.0 / 6.0 + p / 24.0)))
        return self.w * (s0 + (1.0 + s0) * poly)

    # -- which unknown or bulk node every boundary stencil reads
    def _boundary(self):
        nx, ny, M, cfg = self.nx, self.ny, self.M, self.cfg
        kinds = cfg["sides"]
        per = [kinds[0] == "periodic", kinds[2] == "periodic"]
        length, tper = [ny, ny, nx, nx], [per[1], per[1], per[0], per[0]]
        lo = [0 if p else M for p in tper]
        hi = [n - 1 - (0 if p else M) for n, p in zip(length, tper)]
        cbc = [s for s in range(4) if kinds[s] == "cbc"]
        corners = not per[0] and not per[1] and len(cbc) == 4
        base, n = {}, 0
        for s in cbc:
            base[s] = n
            n += (hi[s] - lo[s] + 1) * M
        self.n_side, self.n = n, n + (4 if corners else 0)
        first, last = [0, 1, 0, 2], [2, 3, 1, 3]

        def xy(s, j, p):        # the node at layer j (0: x_f, negative: further in)
            x0 = {0: M, 1: nx - 1 - M}.get(s)
            y0 = {2: M, 3: ny - 1 - M}.get(s)
            if s < 2:
                return np.full_like(p, x0 + j * NORMAL[s][0]), p
            return p, np.full_like(p, y0 + j * NORMAL[s][1])

        def node(s, j, p):
            x, y = xy(s, j, p)
            return y * nx + x

        def ref(s, j, p):       # unknown index, or self.n + grid node
            p = p % length[s] if tper[s] else p
            if j <= 0:
                return self.n + node(s, j, p)
            r = base[s] + (j - 1) * (hi[s] - lo[s] + 1) + (p - lo[s])
            if not tper[s]:
                r = np.where(p < lo[s], self.n_side + first[s], np.where(p > hi[s], self.n_side + last[s], r))
            return r

        rows = {k: [] for k in ("a", "b", "k0", "ka", "kb", "tp", "tm", "n0", "n1", "t0", "t1", "scheme", "side", "write", "xf",
                                "last", "fa", "fb", "fc", "v0", "v1", "v2", "v3", "v4", "vt", "pinf")}
        code = {"lodi": 0, "lodi_relax": 1, "cbc": 2, "cbc_relax": 3}
        for s in cbc:
            p = np.arange(lo[s], hi[s] + 1)
            z = np.zeros_like(p)
            for j in range(1, M + 1):
                out = j == M
                tmode = z if tper[s] else np.where(p == hi[s], 1, np.where(p == lo[s], -1, 0))
                step = np.where(tmode == 0, 1, -tmode)
                vals = {"a": ref(s, j - 1 if out else j + 1, p), "b": ref(s, j - 2 if out else j - 1, p),
                        "k0": z + (1.5 if out else 0.0), "ka": z + (-2.0 if out else 0.5), "kb": z + (0.5 if out else -0.5),
                        "tp": ref(s, j, p + 1), "tm": ref(s, j, p - 1), "n0": z + NORMAL[s][0], "n1": z + NORMAL[s][1],
                        "t0": z + TANGENT[s][0], "t1": z + TANGENT[s][1], "scheme": z + code[cfg["schemes"][s]],
                        "side": z + 1, "write": node(s, j, p), "xf": node(s, 0, p), "last": z + int(out),
                        "fa": ref(s, j - 2 if out else j + 1, p), "fb": ref(s, j - 1, p),
                        "fc": ref(s, j - 3 if out else j - 1, p), "vt": tmode, "pinf": z + cfg["p_inf"][s]}
                if cfg["viscous"] == "meso":
                    w = (lambda q: q % length[s]) if tper[s] else (lambda q: q)  # noqa: E731
                    vals.update(v0=node(s, -M, p), v1=node(s, -M - 1, p), v2=node(s, -M - 2, p),
                                v3=node(s, -M, w(p + step)), v4=node(s, -M, w(np.where(tmode == 0, p - 1, p + 2 * step))))
                else:
                    vals.update(v0=z, v1=z, v2=z, v3=z, v4=z)
                for k, v in vals.items():
                    rows[k].append(v)
        h = math.sqrt(0.5)
        self.blocks = []
        for k in range(4 if corners else 0):
            sx, sy = (1 if k & 1 else -1), (1 if k & 2 else -1)
            xc, yc = (M - 1 if sx < 0 else nx - M), (M - 1 if sy < 0 else ny - M)
            me = self.n_side + k
            vals = {"a": self.n + (yc - sy) * nx + xc - sx, "b": self.n + (yc - 2 * sy) * nx + xc - 2 * sx,
                    "k0": 1.5 * h, "ka": -2.0 * h, "kb": 0.5 * h, "tp": me, "tm": me, "n0": sx * h, "n1": sy * h,
                    "t0": -sy * h, "t1": sx * h, "scheme": 0, "side": 0, "write": yc * nx + xc, "xf": (yc - sy) * nx + xc - sx,
                    "last": 0, "fa": me, "fb": me, "fc": me, "v0": 0, "v1": 0, "v2": 0, "v3": 0, "v4": 0, "vt": 0,
                    "pinf": 0.0}
            for key, v in vals.items():
                rows[key].append(np.array([v]))
            xs = range(0, M) if sx < 0 else range(nx - M, nx)
            ys = range(0, M) if sy < 0 else range(ny - M, ny)
            self.blocks += [(me, y * nx + x) for y in ys for x in xs]
        real = ("k0", "ka", "kb", "n0", "n1", "t0", "t1", "vt", "pinf")
        if self.n:
            self.row = {k: torch.tensor(np.concatenate(v), dtype=torch.float64 if k in real else torch.int64, device=self.dev)
                        for k, v in rows.items()}
            unk = list(range(self.n_side)) + [u for u, _ in self.blocks]
            wr = self.row["write"][:self.n_side].tolist() + [q for _, q in self.blocks]
            self.w_unk = torch.tensor(unk, device=self.dev)
            self.w_node = torch.tensor(wr, device=self.dev)
        # inflow and zero-gradient nodes (two opposite sides with the other axis periodic)
        self.in_node, self.zg_node, self.zg_src = [], [], []
        for s in range(4):
            for j in range(1, M + 1):
                p = np.arange(lo[s], hi[s] + 1)
                if kinds[s] == "inflow":
                    self.in_node += node(s, j, p).tolist()
                elif kinds[s] == "zg":
                    self.zg_node += node(s, j, p).tolist()
                    self.zg_src += node(s, 0, p).tolist()
        bx = (0, nx) if per[0] else (M, nx - M)
        by = (0, ny) if per[1] else (M, ny - M)
        self.bulk = (slice(*by), slice(*bx))

    def local(self, U):         # (drho, u_n, u_t, dT) of [n, 4] lab values
        r = self.row
        return U[:, 0], U[:, 1] * r["n0"] + U[:, 2] * r["n1"], U[:, 1] * r["t0"] + U[:, 2] * r["t1"], U[:, 3]

    def project(self, U, v):    # S v
        s0, un, ut, t = U
        if self.thermal:
            r = (1.0 + t) / (1.0 + s0)
            a = torch.sqrt((1.0 + t) / (8.0 * self.cs2))
            e = 0.25 * (r * v[0] + v[3])
            return [0.5 * (v[3] - r * v[0]), v[2], e - a * v[1], e + a * v[1]]
        h = (1.0 + s0) / (2.0 * math.sqrt(self.cs2)) * v[1]
        return [0.5 * v[0] - h, v[2], 0.5 * v[0] + h]

    def speeds(self, U):
        if self.thermal:
            c = torch.sqrt(2.0 * self.cs2 * (1.0 + U[3]))
            return [U[1], U[1], U[1] - c, U[1] + c]
        c = math.sqrt(self.cs2)
        return [U[1] - c, U[1], U[1] + c]

    def rhs(self, Y, grid, V, incoming, P):
        r, cs2 = self.row, self.cs2
        every = torch.cat([Y, grid])
        U = self.local(Y)
        A, B = self.local(every[r["a"]]), self.local(every[r["b"]])
        Up, Um = self.local(every[r["tp"]]), self.local(every[r["tm"]])
        dn = [r["k0"] * U[m] + r["ka"] * A[m] + r["kb"] * B[m] for m in range(4)]
        rho, on = 1.0 + U[0], r["side"].double()

        def d(f):
            return 0.5 * on * (f(Up) - f(Um))

        TT = [-d(lambda u: (1.0 + u[0]) * u[2]), -U[2] * d(lambda u: u[1]),
              -cs2 / rho * d(lambda u: u[0] + u[3] + u[0] * u[3]) - U[2] * d(lambda u: u[2]),
              -d(lambda u: (1.0 + u[3]) * u[2]) if self.thermal else torch.zeros_like(rho)]
        dP = cs2 * (U[0] + U[3] + U[0] * U[3]) - (r["pinf"] + P["p_inf"] - cs2)
        sd, st, sv = self.project(U, dn), self.project(U, TT), self.project(U, V)
        lam, wave = self.speeds(U), []
        for i in range(len(lam)):
            acoustic = i >= 2 if self.thermal else i != 1
            relax = P["beta_P"] * dP if acoustic else 0.0
            full = st[i] + sv[i]
            inc = torch.where(r["scheme"] == 1, P["alpha_T"] * (P["t_inf"] - st[i]) + relax, torch.zeros_like(full))
            inc = torch.where(r["scheme"] == 2, full, inc)
            inc = torch.where(r["scheme"] == 3, full + P["alpha_T"] * (P["t_inf"] - st[i]) - P["alpha_V"] * sv[i] + relax, inc)
            wave.append(torch.where(incoming[i], inc, lam[i] * sd[i]))
        if self.thermal:
            th = 1.0 + U[3]
            o = [(wave[2] + wave[3] - wave[0]) * rho / th, torch.sqrt(2.0 * cs2 / th) * (wave[3] - wave[2]), wave[1],
                 wave[0] + wave[2] + wave[3]]
        else:
            o = [wave[0] + wave[2], math.sqrt(cs2) / rho * (wave[2] - wave[0]), wave[1], torch.zeros_like(rho)]
        full = (r["scheme"] >= 2).double()
        k = [full * (TT[m] + V[m]) - o[m] for m in range(4)]
        return torch.stack([k[0], k[1] * r["n0"] + k[2] * r["t0"], k[1] * r["n1"] + k[2] * r["t1"], k[3]], 1)

    def viscous(self, Y, grid, neq):
        r, cs2 = self.row, self.cs2
        nu = (self.tau - 0.5) * cs2
        zero = torch.zeros_like(Y[:, 0])
        on = r["side"].double()
        mode = self.cfg["viscous"]
        if mode == "off":
            return [zero] * 4
        if mode == "fd":
            every = torch.cat([Y, grid])
            U, A, B, C = (self.local(every[r[k]]) if k else self.local(Y) for k in ("", "fa", "fb", "fc"))
            Up, Um = self.local(every[r["tp"]]), self.local(every[r["tm"]])
            last = r["last"].bool()
            dnn = [torch.where(last, 2.0 * U[m] - 5.0 * B[m] + 4.0 * A[m] - C[m], A[m] - 2.0 * U[m] + B[m]) for m in range(4)]
            d1 = [torch.where(last, 0.5 * (3.0 * U[m] - 4.0 * B[m] + A[m]), 0.5 * (A[m] - B[m])) for m in range(4)]
            lap = [dnn[m] + Up[m] - 2.0 * U[m] + Um[m] for m in range(4)]
            e1, e2 = d1[1] - 0.5 * (Up[2] - Um[2]), d1[2] + 0.5 * (Up[1] - Um[1])
            heat = 2.0 * nu * lap[3] + nu / cs2 * (e1 * e1 + e2 * e2) if self.thermal else zero
            return [zero, on * nu * lap[1], on * nu * lap[2], on * heat]
        # mesoscopic: stress and heat flux of the stencil's nodes, in the local frame
        H = []
        for k in ("v0", "v1", "v2", "v3", "v4"):
            N, U = neq(r[k]), grid[r[k]]
            n0, n1, t0, t1 = r["n0"], r["n1"], r["t0"], r["t1"]
            H.append([n0 * n0 * N[0] + 2.0 * n0 * n1 * N[1] + n1 * n1 * N[2],
                      n0 * t0 * N[0] + (n0 * t1 + n1 * t0) * N[1] + n1 * t1 * N[2],
                      t0 * t0 * N[0] + 2.0 * t0 * t1 * N[1] + t1 * t1 * N[2], n0 * N[3] + n1 * N[4], t0 * N[3] + t1 * N[4],
                      n0 * U[:, 1] + n1 * U[:, 2], t0 * U[:, 1] + t1 * U[:, 2]])
        tm = r["vt"]
        dn = [0.5 * (3.0 * H[0][m] - 4.0 * H[1][m] + H[2][m]) for m in range(7)]
        dt = [torch.where(tm == 0, 0.5 * (H[3][m] - H[4][m]), 0.5 * tm * (3.0 * H[0][m] - 4.0 * H[3][m] + H[4][m]))
              for m in range(7)]
        rho = 1.0 + grid[r["v0"]][:, 0]
        e1, e2 = dn[5] - dt[6], dn[6] + dt[5]
        heat = -(dn[3] + dt[4]) / rho / cs2 + nu / cs2 * (e1 * e1 + e2 * e2) if self.thermal else zero
        return [zero, on * (dn[0] + dt[1]) / rho, on * (dn[1] + dt[2]) / rho, on * heat]

    def neq_of(self, g, U):     # (sigma', q) at grid nodes from their pulled populations
        fac = 1.0 - 0.5 / self.tau

        def at(nodes):
            gi = g[:, nodes]
            u = [v[nodes] for v in U]
            d = gi - self.equilibrium(u)
            cx, cy = self.c[:, :1], self.c[:, 1:]
            ex, ey = cx - u[1], cy - u[2]
            q = 0.5 * d * (ex * ex + ey * ey) if self.thermal else 0.0 * d
            return [-fac * (cx * cx * d).sum(0), -fac * (cx * cy * d).sum(0), -fac * (cy * cy * d).sum(0),
                    fac * (q * ex).sum(0), fac * (q * ey).sum(0)]
        return at

    def start(self, fields):
        U = [fields[0].reshape(-1) - 1.0, fields[1].reshape(-1), fields[2].reshape(-1),
             fields[3].reshape(-1) - 1.0 if self.thermal else torch.zeros_like(fields[3]).reshape(-1)]
        Ub = torch.stack(U, 1)[self.row["write"]] if self.n else None
        zeros = lambda nodes: [torch.zeros(len(nodes), dtype=torch.float64, device=self.dev)] * 5  # noqa: E731
        return self.equilibrium(U), Ub, U, zeros

    def step(self, f, Ub, U, neq, P):
        """f* and U_b of the next time, its macros and the moments of its pulled populations."""
        ny, nx = self.ny, self.nx
        g = torch.stack([torch.roll(f[i].reshape(ny, nx), (c[1], c[0]), (0, 1)).reshape(-1) for i, c in enumerate(self.shifts)])
        U1 = self.moments(g)
        f1 = g + (self.equilibrium(U1) - g) / self.tau
        if self.n:
            G0, G1 = torch.stack(list(U), 1), torch.stack(list(U1), 1)
            V = self.viscous(Ub, G0, neq)
            inc = [x < 0.0 for x in self.speeds(self.local(Ub))]
            Gh = 0.5 * (G0 + G1)
            k1 = self.rhs(Ub, G0, V, inc, P)
            k2 = self.rhs(Ub + 0.5 * k1, Gh, V, inc, P)
            k3 = self.rhs(Ub + 0.5 * k2, Gh, V, inc, P)
            k4 = self.rhs(Ub + k3, G1, V, inc, P)
            Ub = Ub + (k1 + 2.0 * k2 + 2.0 * k3 + k4) / 6.0
            fb = self.equilibrium(list(Ub.T))
            if self.cfg["dirichlet"] == "neep":
                xf = self.row["xf"]
                fb = fb + f1[:, xf] - self.equilibrium([v[xf] for v in U1])
            f1 = f1.index_copy(1, self.w_node, fb[:, self.w_unk])
        if self.in_node:
            i = self.cfg["inflow"]
            one = torch.ones(1, dtype=torch.float64, device=self.dev)
            fin = self.equilibrium([one * (i[0] - 1.0), one * i[1], one * i[2], one * (i[3] - 1.0 if self.thermal else 0.0)])
            f1[:, self.in_node] = fin
        if self.zg_node:
            f1[:, self.zg_node] = f1[:, self.zg_src]
        return f1, Ub, U1, self.neq_of(g, U1)

    def params(self):
        c = self.cfg
        return {"alpha_T": c["alpha_T"], "beta_P": c["beta_P"], "t_inf": c["t_inf"], "alpha_V": c["alpha_V"], "p_inf": 0.0}

    @torch.no_grad()
    def fields_after(self, fields, steps):
        s, P = self.start(fields), self.params()
        for _ in range(steps):
            s = self.step(*s, P)
        U = self.moments(s[0])
        shape = (self.ny, self.nx)
        return [(1.0 + U[0]).reshape(shape), U[1].reshape(shape), U[2].reshape(shape), (1.0 + U[3]).reshape(shape)]


def exact(case, seed):
    if case["kind"] == "flow":
        cfg, fields = _flow_inputs(case, seed)
        return _Plain(cfg).fields_after(fields, case["steps"])
    if case["kind"] == "batch":
        cfgs, fields = _batch_inputs(case, seed)
        out = [_Plain(c).fields_after(f, case["steps"]) for c, f in zip(cfgs, fields)]
        return [torch.cat([o[k].reshape(-1) for o in out]) for k in range(4)]
    cfg, fields, ref, theta = _gradient_inputs(case, seed)
    plain = _Plain(cfg)
    th = theta.double().requires_grad_(True)
    P = {"alpha_T": th[0], "beta_P": th[1], "p_inf": th[2] - CS2[case["lattice"]], "alpha_V": th[3], "t_inf": th[4]}

    J, s = torch.zeros((), dtype=torch.float64, device=plain.dev), plain.start(fields)
    for n in range(case["steps"]):
        s = plain.step(*s, P)
        m = [v.reshape(case["ny"], case["nx"])[plain.bulk] for v in s[2]]
        J = J + ((plain.cs2 * (m[0] + m[3] + m[0] * m[3]) - ref[n][plain.bulk]) ** 2).sum()
    J.backward()
    return [J.detach(), th.grad]
