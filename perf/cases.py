"""The workloads whose speed is followed: droplet boxes, ensembles, observables, the learned surrogate and the
Maffettone-Minale model, each called as a user's program calls it.

``listed`` names the cases, ``draw`` gives others of the same ranges, ``prepare`` makes what a program has in hand
before the call, ``run`` is one pass, ``work`` what a pass cannot do without and ``exact`` the same outputs from plain
torch in 64 bits.

Kinds of case:

* ``box``          one droplet box: ``steps`` time steps, then D, the inertia tensor and the droplet's position, as a
                   run samples them; boxes up to ``FIELD_NODES`` nodes also read their density and velocity fields;
* ``ensemble``     many boxes of uneven size advanced together, then every box's moments (how the surrogate's training
                   data and ensemble statistics are collected);
* ``observables``  the shape measures of one stored state: inertia tensor, connected components, surface area;
* ``mlp_predict``  conformation tensor and D of a batch of gradient windows on the GPU;
* ``mlp_train``    a run of Adam steps on minibatches, then the updated parameters;
* ``mm``           Maffettone-Minale trajectories.

What comes from a state kept in float32 or 16 bits is returned in float32, what comes from float64 in float64.
"""

import numpy as np
import torch

from paper_2112_09972_gb300 import inputs, workloads
from paper_2112_09972_gb300.lbm import MLP, BatchLBM, DropletLBM, mm_integrate

FIELD_NODES = 1 << 18
KNOT_STEPS = 200  # time steps between two samples of the gradient history
VISC = (1.0 / 6.0, 1.0 / 6.0)  # tau = 1 in both phases
NODE_BYTES = {"fp64": 608, "fp32": 304, "fp16dev": 176, "bf16dev": 176}  # one read and one write of a node's state
READ_BYTES = {"fp64": 304, "fp32": 152, "fp16dev": 16, "bf16dev": 16}  # what a node's densities are summed from
STEP_FLOPS = {"bgk": 550, "mrt": 1600}  # of one node's update


def listed():
    return [
        # the FP64 parity box, the smallest call: launches and latency count
        _box("shear32_fp64", 32, 32, 32, 6.0, "fp64", "bgk", 50),
        # a box of no row width, as a user's own geometry gives
        _box("ragged_fp32", 60, 50, 44, 8.0, "fp32", "bgk", 100),
        # the 64^3 downscale of the precision case
        _box("droplet64_bf16", 64, 64, 64, 8.0, "bf16dev", "bgk", 200),
        # the throughput case: one sampling interval of 200 steps
        _box("droplet128_fp32", 128, 128, 128, 16.0, "fp32", "bgk", 200),
        # the same box with the multi-relaxation-time collision
        _box("droplet128_mrt", 128, 128, 128, 16.0, "fp32", "mrt", 50),
        # the precision case in 16-bit deviation storage
        _box("droplet256_fp16", 256, 256, 256, 32.0, "fp16dev", "bgk", 50),
        # a sampling interval of the ensemble of edges 40 to 64
        {"name": "ensemble128", "kind": "ensemble", "boxes": 128, "low": 40, "high": 64, "multiple": 8, "steps": 8,
         "mix": 1},
        # shape measures of the throughput case's state
        {"name": "observables128", "kind": "observables", "x": 128, "y": 128, "z": 128, "radius": 16.0,
         "precision": "fp32"},
        # the surrogate's inference batch
        {"name": "mlp_predict_65536", "kind": "mlp_predict", "batch": 65536, "window": 64, "hidden": 256, "layers": 3},
        # the surrogate's training: minibatches of 512
        {"name": "mlp_train_512", "kind": "mlp_train", "batch": 512, "steps": 10, "window": 64, "hidden": 256,
         "layers": 3},
        # the model in float32, as for ensembles of trajectories
        {"name": "mm_fp32", "kind": "mm", "trajectories": 16384, "times": 251, "substeps": 10, "every": 8,
         "precision": "fp32"},
        # the model in float64, as for comparisons
        {"name": "mm_fp64", "kind": "mm", "trajectories": 16384, "times": 51, "substeps": 4, "every": 10,
         "precision": "fp64"},
    ]


def _box(name, x, y, z, radius, precision, collision, steps):
    return {"name": name, "kind": "box", "x": x, "y": y, "z": z, "radius": radius, "precision": precision,
            "collision": collision, "steps": steps}


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _extents(rng, limit):
    """A box: a row width of the fast path with y a multiple of 8, or any extents."""
    while True:
        if rng.random() < 0.5:
            x, y, z = rng.choice((32, 64, 128, 256)), 8 * _log(rng, 2, 32), _log(rng, 16, 256)
        else:
            x, y, z = (_log(rng, 16, 200) for _ in range(3))
        if x * y * z <= limit:
            return x, y, z


def draw(rng):
    kind = rng.choice(("box", "box", "box", "box", "ensemble", "observables", "mlp_predict", "mlp_train", "mm", "mm"))
    if kind in ("box", "observables"):
        precision = rng.choice(("fp32", "fp32", "fp64", "fp16dev", "bf16dev"))
        x, y, z = _extents(rng, 1 << (20 if precision == "fp64" else 23))
        radius = round(min(x, y, z) * rng.uniform(0.17, 0.22), 1)
        if kind == "observables":
            return {"kind": kind, "x": x, "y": y, "z": z, "radius": radius, "precision": precision}
        n = x * y * z
        steps = max(4, min(200, _log(rng, 10, 200), (1 << (24 if precision == "fp64" else 27)) // n))
        case = _box("", x, y, z, radius, precision, rng.choice(("bgk", "bgk", "bgk", "mrt")), steps)
        del case["name"]
        return case
    if kind == "ensemble":
        multiple = rng.choice((8, 8, 1))
        low = 8 * rng.randint(3, 6) - (0 if multiple == 8 else rng.randint(0, 3))
        return {"kind": kind, "boxes": _log(rng, 4, 96), "low": low, "high": min(64, low + 8 * rng.randint(0, 3)),
                "multiple": multiple, "steps": rng.randint(2, 12), "mix": rng.randint(1, 1 << 20)}
    if kind == "mlp_predict":
        return {"kind": kind, "batch": _log(rng, 1, 65536), "window": rng.choice((32, 64)),
                "hidden": rng.choice((128, 256, 256, 320)), "layers": rng.randint(1, 4)}
    if kind == "mlp_train":
        return {"kind": kind, "batch": 32 * _log(rng, 1, 256), "steps": rng.randint(2, 10),
                "window": rng.choice((32, 64)), "hidden": rng.choice((128, 256, 256, 320)), "layers": rng.randint(1, 3)}
    precision = rng.choice(("fp32", "fp64"))
    return {"kind": "mm", "trajectories": _log(rng, 1, 16384), "times": _log(rng, 12, 50 if precision == "fp64" else 250),
            "substeps": rng.randint(1, 4 if precision == "fp64" else 10), "every": rng.randint(1, 12),
            "precision": precision}


def prepare(case, seed):
    return {"box": _prepare_box, "observables": _prepare_box, "ensemble": _prepare_ensemble,
            "mlp_predict": _prepare_mlp, "mlp_train": _prepare_mlp, "mm": _prepare_mm}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


# ---- droplet boxes ----------------------------------------------------------------------------------------------------

WARM = {"box": 2, "observables": 24}  # steps taken before the call


def _history(edge, seed, n=400):
    """Samples of the boundary's velocity gradient, every KNOT_STEPS steps, at the boundary speed of the throughput case."""
    h = inputs.ou_gradient_history(n, 10.0, 1.0, 20000 + int(seed))
    return inputs.rescale_to_lattice(h, 0.1, edge)


def _prepare_box(case, seed):
    box = (case["x"], case["y"], case["z"])
    g = DropletLBM(box, case["radius"], VISC, workloads.G_COUPLING, precision=case["precision"],
                   rho_hi=workloads.RHO_HI, rho_lo=workloads.RHO_LO, xi=1.0,
                   mrt=True if case.get("collision") == "mrt" else None)
    hist = _history(max(box), seed)
    g.set_gradient_table(KNOT_STEPS * np.arange(len(hist)), hist)
    g.step(WARM[case["kind"]])
    g.sync()
    return {"run": _run_box if case["kind"] == "box" else _run_observables, "g": g, "steps": case.get("steps", 0),
            "kind": np.float64 if case["precision"] == "fp64" else np.float32,
            "fields": case["kind"] == "box" and box[0] * box[1] * box[2] <= FIELD_NODES}


def _shape(g, kind):
    """D, the droplet's inertia tensor and its position in the box."""
    D, axes, lam, centre = g.deformation()
    return {"D": kind(D), "tensor": ((axes * lam) @ axes.T).astype(kind),
            "position": (centre + 0.5 * (np.array(g.box) - 1)).astype(kind)}


def _run_box(s):
    g, kind = s["g"], s["kind"]
    g.step(s["steps"])
    out = _shape(g, kind)
    if s["fields"]:
        out["rho_a"], out["rho_b"], out["u"] = (a.astype(kind, copy=False) for a in g.fields())
    return out


def _run_observables(s):
    g, kind = s["g"], s["kind"]
    out = _shape(g, kind)
    out["count"], out["sizes"] = g.components(0.0, 10)
    out["surface"] = np.array(g.surface_deformation()).astype(kind)
    return out


# ---- ensembles --------------------------------------------------------------------------------------------------------

def _edges(case):
    rng = np.random.Generator(np.random.Philox(key=[int(case["mix"]), 3]))
    m = case["multiple"]
    lo, hi = -(-case["low"] // m), case["high"] // m
    return [tuple(int(v) * m for v in e) if m == 1 else (int(e[0]) * m,) * 3
            for e in rng.integers(lo, max(lo, hi) + 1, size=(case["boxes"], 3))]


def _ensemble_history(case, seed, n=64):
    boxes = _edges(case)
    out = np.empty((n, len(boxes), 9))
    for k, b in enumerate(boxes):
        h = inputs.ou_gradient_history(n, 200.0, 1.0, 30000 + int(seed), box_id=k)
        out[:, k] = inputs.rescale_to_lattice(h, 0.1, max(b))
    return out


def _prepare_ensemble(case, seed):
    boxes = _edges(case)
    b = BatchLBM(boxes, [min(e) / 5.0 for e in boxes], VISC, workloads.G_COUPLING, rho_lo=workloads.RHO_LO,
                 rho_hi=workloads.RHO_HI)
    b.set_gradients(_ensemble_history(case, seed))
    b.step(2)
    b.sync()
    return {"run": _run_ensemble, "b": b, "steps": case["steps"]}


def _run_ensemble(s):
    s["b"].step(s["steps"])
    return s["b"].moments().astype(np.float32)


# ---- surrogate --------------------------------------------------------------------------------------------------------

RATE = 1e-3


def _sizes(case):
    return (9 * case["window"],) + (case["hidden"],) * case["layers"] + (6,)


def _mlp_inputs(case, seed):
    """Normalisation, parameters, gradient windows and targets near the identity tensor."""
    sizes = _sizes(case)
    rng = np.random.default_rng(40000 + int(seed))
    n = case["batch"] * case.get("steps", 1)
    gen = torch.Generator(device="cuda").manual_seed(50000 + int(seed))
    x = torch.empty((n, sizes[0]), device="cuda").normal_(0.0, 1e-3, generator=gen)
    mean = np.array([1, 0, 0, 1, 0, 1], dtype=np.float32)
    t = torch.empty((n, 6), device="cuda").normal_(0.0, 0.02, generator=gen) + torch.from_numpy(mean).cuda()
    norm = (rng.normal(0.0, 1e-4, sizes[0]).astype(np.float32), np.full(sizes[0], 1e3, dtype=np.float32), mean,
            np.full(6, 50.0, dtype=np.float32))
    p = []
    for a, b in zip(sizes[:-1], sizes[1:]):
        p += [rng.normal(0.0, (2.0 / a) ** 0.5, a * b), rng.normal(0.0, 0.02, b)]
    return x, t, norm, np.concatenate(p).astype(np.float32)


def _prepare_mlp(case, seed):
    x, t, norm, p = _mlp_inputs(case, seed)
    stream = torch.cuda.Stream()
    train = case["kind"] == "mlp_train"
    net = MLP(_sizes(case), max_batch=case["batch"] if train else 16384, seed=0, stream=stream.cuda_stream)
    net.set_normalisation(*norm)
    net.set_params(p)
    s = {"net": net, "stream": stream, "x": x, "t": t, "batch": case["batch"],
         "run": _run_train if train else _run_predict}
    if not train:
        s["m6"] = torch.empty((case["batch"], 6), device="cuda")
        s["D"] = torch.empty(case["batch"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


def _run_predict(s):
    s["net"].deformation(s["x"], s["m6"], s["D"])
    return s["m6"], s["D"]


def _run_train(s):
    n = s["batch"]
    for k in range(0, s["x"].shape[0], n):
        s["net"].train_step(s["x"][k:k + n], s["t"][k:k + n], RATE)
    return s["net"].get_params()


# ---- Maffettone-Minale model ------------------------------------------------------------------------------------------

TAU_D, CHI = 30.0, 1.0


def _gradients(case, seed):
    """A [times, trajectories, 9]: the exact-update Ornstein-Uhlenbeck components on the traceless basis."""
    n, T = case["trajectories"], case["times"]
    gen = torch.Generator(device="cuda").manual_seed(60000 + int(seed))
    decay = float(np.exp(-1.0 / 200.0))
    kick = float(np.sqrt(1.0 - decay * decay))
    scale = np.array([1.0 / np.sqrt(10.0)] * 5 + [1.0 / np.sqrt(6.0)] * 3) / 300.0
    basis = torch.from_numpy((inputs.traceless_basis() * scale[:, None, None]).reshape(8, 9)).cuda()
    A = torch.empty((T, n, 9), dtype=torch.float64, device="cuda")
    a = torch.randn((n, 8), dtype=torch.float64, device="cuda", generator=gen)
    for t in range(T):
        if t:
            a = decay * a + kick * torch.randn((n, 8), dtype=torch.float64, device="cuda", generator=gen)
        torch.matmul(a, basis, out=A[t])
    return A


def _prepare_mm(case, seed):
    return {"run": _run_mm, "A": _gradients(case, seed), "case": case}


def _run_mm(s):
    c = s["case"]
    D, M = mm_integrate(s["A"], TAU_D, CHI, substeps=c["substeps"], record_every=c["every"], precision=c["precision"],
                        want_M=True)
    return (D, M) if c["precision"] == "fp64" else (D.float(), M.float())


# ---- what a pass cannot do without ------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("box", "observables"):
        n = case["x"] * case["y"] * case["z"]
        p = case["precision"]
        if kind == "observables":
            return {"bytes": n * READ_BYTES[p], "flops": n * 60}
        out = 8 * 5 * n if n <= FIELD_NODES else 0
        return {"bytes": case["steps"] * n * NODE_BYTES[p] + out,
                "flops": case["steps"] * n * STEP_FLOPS[case["collision"]]}
    if kind == "ensemble":
        n = sum(x * y * z for x, y, z in _edges(case))
        return {"bytes": n * (case["steps"] * NODE_BYTES["fp32"] + READ_BYTES["fp32"]),
                "flops": n * case["steps"] * STEP_FLOPS["bgk"]}
    if kind == "mm":
        n, steps = case["trajectories"], case["times"] - 1
        return {"bytes": 8 * n * (9 * case["times"] + steps // case["every"] + 1 + 6),
                "flops": n * steps * case["substeps"] * 4 * 150}
    sizes = _sizes(case)
    weights = sum(a * b for a, b in zip(sizes[:-1], sizes[1:]))
    n = case["batch"]
    if kind == "mlp_predict":
        return {"bytes": n * (4 * sizes[0] + 24 + 8) + 2 * weights, "flops": 2 * n * weights}
    first = sizes[0] * sizes[1]
    return {"bytes": case["steps"] * (n * 4 * (sizes[0] + 6) + 28 * weights),
            "flops": case["steps"] * 2 * n * (3 * weights - first)}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------------

def exact(case, seed):
    return {"box": _exact_box, "observables": _exact_box, "ensemble": _exact_ensemble, "mlp_predict": _exact_predict,
            "mlp_train": _exact_train, "mm": _exact_mm}[case["kind"]](case, seed)


C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)])
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _equilibrium(i, rho, u):
    cu = sum(float(C[i][a]) * u[a] for a in range(3) if C[i][a])
    u2 = 1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
    return W[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - u2)


def _relaxation(tau):
    """M^-1 S M of the multi-relaxation-time collision, the moment basis of d'Humieres et al. (2002)."""
    x, y, z = C.T.astype(float)
    r = x * x + y * y + z * z
    rows = [r ** 0, 19 * r - 30, (21 * r * r - 53 * r + 24) / 2, x, (5 * r - 9) * x, y, (5 * r - 9) * y, z,
            (5 * r - 9) * z, 3 * x * x - r, (3 * r - 5) * (3 * x * x - r), y * y - z * z, (3 * r - 5) * (y * y - z * z),
            x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z]
    s = 1.0 / tau
    rates = [s, 1.19, 1.4, s, 1.2, s, 1.2, s, 1.2, s, 1.4, s, 1.4, s, s, s, 1.98, 1.98, 1.98]
    M = np.array(rows)
    return np.linalg.inv(M) @ np.diag(rates) @ M


class _Exact:
    """One droplet box in float64 torch: ghost nodes, pull streaming, Shan-Chen force, BGK or MRT collision."""

    def __init__(self, box, radius, A0, collision="bgk"):
        self.n, self.tau = box, 3.0 * VISC[0] + 0.5
        self.rho_b = (workloads.RHO_LO, workloads.RHO_HI)
        self.K = _relaxation(self.tau) if collision == "mrt" else None
        ax = [torch.arange(-1, m + 1, dtype=torch.float64, device="cuda") - 0.5 * (m - 1) for m in box]
        self.X = (ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None])
        Z, Y, X = box[2], box[1], box[0]
        self.P = torch.zeros((2, 19, Z + 2, Y + 2, X + 2), dtype=torch.float64, device="cuda")
        p = [v[tuple(slice(1, -1) if d > 1 else slice(None) for d in v.shape)] for v in self.X]
        self.x = p
        th = torch.tanh(torch.sqrt(p[0] ** 2 + p[1] ** 2 + p[2] ** 2) - radius)
        lo, hi = self.rho_b
        rho = (lo + (hi - lo) * 0.5 * (1 - th), lo + (hi - lo) * 0.5 * (1 + th))
        u = self._flow(A0, p)
        self.f = self.P[:, :, 1:-1, 1:-1, 1:-1]
        for s in range(2):
            for i in range(19):
                self.f[s, i] = _equilibrium(i, rho[s], u)

    @staticmethod
    def _flow(A, p):
        A = np.asarray(A).reshape(3, 3)
        return [A[a, 0] * p[0] + A[a, 1] * p[1] + A[a, 2] * p[2] for a in range(3)]

    def moments(self):
        r = [self.f[s].sum(0) for s in range(2)]
        w = ((r[0] - r[1]) / (r[0] + r[1])).clamp_min_(0.0)
        x, y, z = self.x
        return np.array([float(v.sum()) for v in (w, w * x, w * y, w * z, w * x * x, w * x * y, w * x * z, w * y * y,
                                                  w * y * z, w * z * z)])

    def step(self, A):
        m = self.moments()
        xc = m[1:4] / m[0] if m[0] > 0 else np.zeros(3)
        full = slice(None)
        for d in range(3):
            for end in (slice(0, 1), slice(-1, None)):
                cut = [full] * 3
                cut[2 - d] = end
                p = [v[tuple(c if v.shape[k] > 1 else full for k, c in enumerate(cut))] - xc[a]
                     for a, v in enumerate(self.X)]
                u = self._flow(A, p)
                for s in range(2):
                    for i in range(1, 19):
                        self.P[s, i][tuple(cut)] = _equilibrium(i, self.rho_b[s], u)
        Z, Y, X = self.n[2], self.n[1], self.n[0]

        def at(t, c):  # t[x + c] at the fluid nodes
            return t[1 + c[2]:1 + c[2] + Z, 1 + c[1]:1 + c[1] + Y, 1 + c[0]:1 + c[0] + X]

        g = torch.empty((2, 19, Z, Y, X), dtype=torch.float64, device="cuda")
        for s in range(2):
            for i in range(19):
                g[s, i] = at(self.P[s, i], -C[i])
        rho = g.sum(1)
        pad = torch.empty((2, Z + 2, Y + 2, X + 2), dtype=torch.float64, device="cuda")
        for s in range(2):
            pad[s] = self.rho_b[s]
            pad[s, 1:-1, 1:-1, 1:-1] = rho[s]
        force = [[0.0, 0.0, 0.0], [0.0, 0.0, 0.0]]
        for s in range(2):
            for i in range(1, 19):
                v = W[i] * at(pad[s], C[i])
                for a in range(3):
                    if C[i][a]:
                        force[s][a] = force[s][a] + float(C[i][a]) * v
        common = []
        for a in range(3):
            j = 0.0
            for i in range(1, 19):
                if C[i][a]:
                    j = j + float(C[i][a]) * (g[0, i] + g[1, i])
            common.append(j / (rho[0] + rho[1]))
        for s in range(2):
            u = [common[a] - workloads.G_COUPLING * self.tau * force[1 - s][a] for a in range(3)]
            if self.K is None:
                for i in range(19):
                    self.f[s, i] = g[s, i] - (g[s, i] - _equilibrium(i, rho[s], u)) / self.tau
            else:
                dev = torch.stack([g[s, i] - _equilibrium(i, rho[s], u) for i in range(19)])
                K = torch.from_numpy(self.K).cuda()
                self.f[s] = g[s] - (K @ dev.reshape(19, -1)).reshape(dev.shape)

    def fields(self):
        r = [self.f[s].sum(0) for s in range(2)]
        u = []
        for a in range(3):
            j = 0.0
            for i in range(1, 19):
                if C[i][a]:
                    j = j + float(C[i][a]) * (self.f[0, i] + self.f[1, i])
            u.append(j / (r[0] + r[1]))
        return r[0], r[1], torch.stack(u, dim=-1)


def _shape_of(m, box):
    c = m[1:4] / m[0]
    I = np.array([[m[4], m[5], m[6]], [m[5], m[7], m[8]], [m[6], m[8], m[9]]]) / m[0] - np.outer(c, c)
    lam = np.sqrt(np.linalg.eigvalsh(I))
    return {"D": (lam[2] - lam[0]) / (lam[2] + lam[0]), "tensor": I, "position": c + 0.5 * (np.array(box) - 1)}


def _exact_box(case, seed):
    box = (case["x"], case["y"], case["z"])
    steps = WARM[case["kind"]] + case.get("steps", 0)
    if box[0] * box[1] * box[2] * steps > 1 << 30:
        return None
    hist = _history(max(box), seed)
    b = _Exact(box, case["radius"], hist[0], case.get("collision", "bgk"))
    for t in range(steps):
        k, w = divmod(t, KNOT_STEPS)
        b.step(hist[k] + w / KNOT_STEPS * (hist[k + 1] - hist[k]))
    out = _shape_of(b.moments(), box)
    if case["kind"] == "observables":
        r = [b.f[s].sum(0) for s in range(2)]
        phi = (r[0] - r[1]) / (r[0] + r[1])
        span = float(phi.max() - phi.min())
        d = [0.5 * (phi.narrow(a, 2, phi.shape[a] - 2) - phi.narrow(a, 0, phi.shape[a] - 2)) for a in range(3)]
        d = [v[tuple(slice(None) if k == a else slice(1, -1) for k in range(3))] for a, v in enumerate(d)]
        area = float(torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2).sum()) / span
        volume = float((phi - phi.min()).sum()) / span
        sphere = float(np.cbrt(36.0 * np.pi * volume * volume))
        return {**out, "count": None, "sizes": None,
                "surface": np.array([np.sqrt(max(0.0, 1.0 - sphere / area)), area, volume])}
    if box[0] * box[1] * box[2] <= FIELD_NODES:
        out["rho_a"], out["rho_b"], out["u"] = b.fields()
    return out


def _exact_ensemble(case, seed):
    boxes, hist = _edges(case), _ensemble_history(case, seed)
    out = []
    for k, box in enumerate(boxes):
        b = _Exact(box, min(box) / 5.0, hist[0, k])
        for t in range(2 + case["steps"]):
            b.step(hist[min(t, len(hist) - 1), k])
        out.append(b.moments())
    return np.array(out)


def _layers(case, p):
    at, out = 0, []
    for a, b in zip(_sizes(case)[:-1], _sizes(case)[1:]):
        Wl = p[at:at + a * b].reshape(b, a)
        out += [Wl, p[at + a * b:at + a * b + b]]
        at += a * b + b
    return out


def _forward(x, layers):
    h = [x]
    for l in range(0, len(layers), 2):
        z = h[-1] @ layers[l].T + layers[l + 1]
        h.append(z.clamp_min(0.0) if l + 2 < len(layers) else z)
    return h


def _mlp64(case, seed):
    x, t, norm, p = _mlp_inputs(case, seed)
    xm, xs, ym, ys = (torch.from_numpy(v).cuda().double() for v in norm)
    return (x.double() - xm) * xs, (t.double() - ym) * ys, ym, ys, torch.from_numpy(p).cuda().double()


def _exact_predict(case, seed):
    x, _, ym, ys, p = _mlp64(case, seed)
    m = _forward(x, _layers(case, p))[-1] / ys + ym
    q = m[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3)
    lam = torch.linalg.eigvalsh(q.cpu()).clamp_min(0.0).sqrt()
    return m, (lam[:, 2] - lam[:, 0]) / (lam[:, 2] + lam[:, 0])


def _exact_train(case, seed):
    x, t, _, _, p = _mlp64(case, seed)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    n = case["batch"]
    for step in range(1, case["steps"] + 1):
        rows = slice((step - 1) * n, step * n)
        layers = _layers(case, p)
        h = _forward(x[rows], layers)
        d = 2.0 / (6 * n) * (h[-1] - t[rows])
        grads = []
        for l in range(len(layers) - 2, -1, -2):
            grads = [(d.T @ h[l // 2]).reshape(-1), d.sum(0)] + grads
            if l:
                d = (d @ layers[l]) * (h[l // 2] > 0)
        g = torch.cat(grads)
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        p = p - RATE * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return p


def _exact_mm(case, seed):
    A = _gradients(case, seed).reshape(case["times"], -1, 3, 3)
    n = A.shape[1]
    eye = torch.eye(3, dtype=torch.float64, device="cuda")
    f1 = 40.0 * (CHI + 1.0) / ((3.0 + 2.0 * CHI) * (16.0 + 19.0 * CHI))

    def rate(M, G):
        S, R = 0.5 * (G + G.transpose(1, 2)), 0.5 * (G - G.transpose(1, 2))
        ca = TAU_D * G.abs().amax(dim=(1, 2))[:, None, None]
        f2 = 5.0 / (3.0 + 2.0 * CHI) + 3.0 * ca * ca / (2.0 + 6.0 * ca * ca)
        tr = M.diagonal(dim1=1, dim2=2).sum(1)
        two = 0.5 * (tr * tr - (M * M).sum((1, 2)))
        a, b, c = M.unbind(1)
        three = (a * torch.linalg.cross(b, c)).sum(1)
        iso = (3.0 * three / two)[:, None, None] * eye
        return f2 * (S @ M + M @ S) + (R @ M - M @ R) - f1 / TAU_D * (M - iso)

    def deformation(M):
        lam = torch.linalg.eigvalsh(M.cpu()).clamp_min(0.0).sqrt()
        return (lam[:, 2] - lam[:, 0]) / (lam[:, 2] + lam[:, 0])

    M = eye.expand(n, 3, 3).clone()
    D, k, h = [deformation(M)], case["substeps"], 1.0 / case["substeps"]
    for t in range(case["times"] - 1):
        d = A[t + 1] - A[t]
        for q in range(k):
            a, b, c = (A[t] + (q + e) * h * d for e in (0.0, 0.5, 1.0))
            k1 = rate(M, a)
            k2 = rate(M + 0.5 * h * k1, b)
            k3 = rate(M + 0.5 * h * k2, b)
            k4 = rate(M + h * k3, c)
            M = M + (h / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
        if (t + 1) % case["every"] == 0:
            D.append(deformation(M))
    i, j = torch.triu_indices(3, 3)
    return torch.stack(D), M[:, i, j]
