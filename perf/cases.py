"""The workloads whose speed this library is measured by.

A case is one pass a user's program makes through the public entry points:

* ``cavity``: a block of time steps between two samples of a run, then the
  fields of the new state (the loop of every cavity run);
* ``sample``: what a monitored run does at a sample: the Nu / Re reductions,
  the steady-state change, the time average and the fields;
* ``batch``: a block of steps of a Rayleigh-number sweep advanced together,
  then the fields of every cavity;
* ``predict``: the warm-start network's prediction of steady fields;
* ``train``: one training step of that network.

Fields are kept in the storage's own type (an FP32 run has no more than FP32 to
keep), the way a program stores its snapshots.  The flow that every cavity
starts from is a developed one: thermal layers on the isothermal walls, a
stratified core and a convection roll with seeded disturbances.
"""
import math
import os

import numpy as np
import torch

import paper_2509_01099_gb300 as pkg
from paper_2509_01099_gb300 import warmstart
from paper_2509_01099_gb300.cnn import features

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WEIGHTS = os.path.join(ROOT, "paper_2509_01099_gb300", "weights", "warmstart_tanh256.npz")

MA, T_HOT, T_COLD, PR = 0.1, 0.5, -0.5, 0.71
U_F = MA / math.sqrt(3.0)
KEPT = {"fp64": torch.float64, "fp32": torch.float32, "fp16neq": torch.float32,
        "fp16dev": torch.float16, "bf16dev": torch.bfloat16}
REDUCED = ("Nu", "Nu_hot", "Nu_cold", "Re", "Re_uv", "Re_mean", "mass", "max_speed")
BATCH_SIZES = (128, 256, 384, 512)     # mesh sizes of the Rayleigh-number sweep
LR, ADAM_STEP = 1e-4, 1000             # late in the training's learning-rate schedule


def listed():
    c = dict(kind="cavity", dim=2, mesh="tanh", a=1.5)
    return [
        # the parity workload, in the paper's precision: the smallest mesh in
        # use, where a step is a few microseconds and launches count; 1000
        # steps is the sampling interval of the steady-state searches
        dict(c, name="cavity2d_n64_fp64", n=64, Ra=1e6, precision="fp64", steps=1000),
        # the validation case of the paper's tables: an odd mesh, error-function
        # stretching, sampled every 200 steps
        dict(c, name="cavity2d_n257_fp32", n=257, mesh="erf", Ra=1e6, precision="fp32", steps=200),
        # the headline workload, read back every 100 steps
        dict(c, name="cavity2d_n1024_fp32", n=1024, Ra=1e8, precision="fp32", steps=100),
        # the same cavity with 16-bit deviations (half the memory)
        dict(c, name="cavity2d_n1024_fp16dev", n=1024, Ra=1e8, precision="fp16dev", steps=100),
        # the accurate 16-bit storage on the paper's finest Ra = 1e8 mesh
        dict(c, name="cavity2d_n2049_fp16neq", n=2049, mesh="erf", Ra=1e8, precision="fp16neq",
             steps=40),
        # a large mesh, far beyond L2: the memory-bandwidth regime
        dict(c, name="cavity2d_n4096_fp32", n=4096, Ra=1e8, precision="fp32", steps=40),
        # the 3-D workload in FP32 and with 16-bit deviations
        dict(c, name="cavity3d_n256_fp32", dim=3, n=256, Ra=1e7, precision="fp32", steps=25),
        dict(c, name="cavity3d_n256_bf16dev", dim=3, n=256, Ra=1e7, precision="bf16dev", steps=25),
        # one sample of a monitored run: an odd mesh of the grid studies
        dict(c, name="sample2d_n1025_fp32", kind="sample", n=1025, mesh="erf", Ra=1e7,
             precision="fp32", steps=64),
        # the 64-cavity sweep over Ra and mesh size, one block of steps
        dict(name="batch64_fp32", kind="batch", count=64, precision="fp32", steps=64),
        # the warm start of one cavity: the network's smallest call
        dict(name="predict_1", kind="predict", batch=1),
        # one training step at the training's batch size
        dict(name="train_16", kind="train", batch=16),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rayleigh(rng, n, dim):
    """A Rayleigh number that a mesh of n nodes a side resolves."""
    lo, hi = (5.5, 6.5) if n <= 160 else (6.0, 7.0) if n <= 300 else (6.7, 8.0) if n <= 1000 \
        else (7.3, 8.0)
    return float("%.3g" % 10.0 ** rng.uniform(lo, min(hi, 7.0) if dim == 3 else hi))


def draw(rng):
    kind = rng.choices(("cavity2", "cavity3", "sample", "batch", "predict", "train"),
                       (9, 4, 3, 2, 2, 2))[0]
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 48),
                    precision=rng.choice(("fp32", "fp32", "bf16dev", "fp16neq")),
                    steps=rng.choice((16, 64, 100)))
    if kind == "predict":
        return dict(kind="predict", batch=_spread(rng, 1, 32))
    if kind == "train":
        return dict(kind="train", batch=_spread(rng, 1, 16))
    dim = 3 if kind == "cavity3" else 2
    mesh = rng.choices(("tanh", "erf", "uniform"), (4, 3, 1))[0]
    precision = rng.choices(("fp32", "fp64", "fp16dev", "bf16dev", "fp16neq"), (5, 2, 1, 1, 1))[0]
    if precision == "fp16neq" and dim == 3:
        precision = "bf16dev"
    top = {2: 2049, 3: 192} if precision != "fp64" else {2: 1025, 3: 96}
    n = _spread(rng, {2: 40, 3: 24}[dim], top[dim])
    nodes = float(n) ** dim
    most = 2e8 if precision != "fp64" else 1.5e7     # node updates of a pass
    steps = max(4, min(rng.choice((16, 64, 100, 200, 333)), int(most / nodes / dim)))
    return dict(kind="sample" if kind == "sample" else "cavity", dim=dim, n=n, mesh=mesh,
                a=rng.choice((1.0, 1.5, 2.1)), Ra=_rayleigh(rng, n, dim), precision=precision,
                steps=steps)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _mesh(kind, n, a):
    """Ghost and fluid nodes xi_0 .. xi_(n+1) of one axis."""
    if kind == "uniform":
        xi = np.array([(j - 0.5) / n for j in range(n + 2)])
    else:
        fn = math.erf if kind == "erf" else math.tanh
        xi = np.array([0.5 * (fn(a * (j / (n + 1) - 0.5)) / fn(0.5 * a) + 1.0)
                       for j in range(n + 2)])
    for j in range((n + 2) // 2, n + 2):
        xi[j] = 1.0 - xi[n + 1 - j]
    return xi


def _flow(dim, xi, seed):
    """T, u, v[, w] of a developed side-heated flow, [z,] y, x, FP64 on the GPU."""
    rng = np.random.default_rng(seed)
    s = torch.from_numpy(xi[1:-1].copy()).cuda().clamp(0.0, 1.0)
    x = s.view((1,) * (dim - 1) + (-1,))
    y = s.view((1,) * (dim - 2) + (-1, 1))
    pi = math.pi
    delta = 0.05 + 0.02 * rng.random()
    core = 0.35 + 0.1 * rng.random()
    T = (0.5 * (torch.exp(-x / delta) - torch.exp(-(1 - x) / delta))
         + core * (y - 0.5) * torch.sin(pi * x))
    u = torch.zeros_like(T)
    v = torch.zeros_like(T)
    # stream function: the roll and a few disturbances, all at rest on the walls
    for k, m, amp in [(1, 1, -0.1)] + [(int(rng.integers(1, 5)), int(rng.integers(1, 5)),
                                        0.01 * rng.standard_normal()) for _ in range(4)]:
        u = u + amp * U_F * pi * m * torch.sin(pi * k * x) ** 2 * torch.sin(2 * pi * m * y)
        v = v - amp * U_F * pi * k * torch.sin(2 * pi * k * x) * torch.sin(pi * m * y) ** 2
        T = T + 0.05 * amp * torch.sin(pi * (k + 1) * x) * torch.cos(pi * m * y)
    out = [T, u, v]
    if dim == 3:
        z = s.view(-1, 1, 1)
        wave = 1.0 + (0.1 + 0.1 * rng.random()) * torch.cos(2 * pi * z)
        out = [T + 0.01 * torch.sin(pi * x) * torch.cos(pi * z), u * wave, v * wave]
        out.append(0.05 * U_F * torch.sin(pi * x) * torch.sin(pi * y) * torch.sin(2 * pi * z))
    shape = (len(xi) - 2,) * dim
    return [f.expand(shape).contiguous() for f in out]


def _sweep(case, seed):
    """The cavities of a batch: Ra log-uniform in [1e6, 1e8], sizes of the sweep.
    The sizes belong to the case, the Rayleigh numbers to the seed."""
    n = np.random.default_rng(case["count"]).choice(BATCH_SIZES, size=case["count"])
    ra = 10.0 ** np.random.default_rng(seed).uniform(6.0, 8.0, size=case["count"])
    return [dict(n=int(k), mesh="tanh", a=1.5, Ra=float(r), Pr=PR) for k, r in zip(n, ra)]


def _training_data(case, seed):
    """(features, snapshots [B, 256, 256, 3]) of a minibatch."""
    rng = np.random.default_rng(seed)
    z = features(rng.uniform(6.0, 8.0, case["batch"]), [PR] * case["batch"],
                 [1.5] * case["batch"])
    xi = _mesh("tanh", 256, 1.5)
    snaps = []
    for k in range(case["batch"]):
        T, u, v = _flow(2, xi, int(rng.integers(1 << 30)))
        snaps.append(torch.stack([T, 4.0 * u / U_F, 4.0 * v / U_F], dim=-1).float())
    return z, torch.stack(snaps)


def _adam_state(net, seed):
    """Adam's moments in the middle of a training."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    for name in net.names:
        m, v = net.m[name], net.v[name]
        m.copy_(1e-4 * torch.randn(m.shape, generator=g, device="cuda"))
        v.copy_(1e-8 * (0.5 + torch.rand(v.shape, generator=g, device="cuda")))
        if name.startswith("Wc"):       # rows that pad K have never had a gradient
            rows = 9 * net.channels[int(name[2:])]
            m[rows:] = 0.0
            v[rows:] = 0.0
    net.t = ADAM_STEP


def prepare(case, seed):
    st = dict(case=case)
    kind = case["kind"]
    if kind in ("cavity", "sample"):
        dim, n = case["dim"], case["n"]
        xi = _mesh(case["mesh"], n, case["a"])
        s = pkg.Solver(*([xi] * dim), Ra=case["Ra"], Pr=PR, precision=case["precision"])
        s.set_fields_device(*_flow(dim, xi, seed))
        names = ("rho", "T", "u", "v") + (("w",) if dim == 3 else ())
        st.update(solver=s, kept=KEPT[case["precision"]],
                  out={k: torch.empty(s.shape, dtype=torch.float64, device="cuda") for k in names})
        if kind == "sample":            # the sample before this one
            s.average_reset()
            s.steady_change()
            s.step(case["steps"])
            s.synchronize()
    elif kind == "batch":
        b = pkg.Batch(_sweep(case, seed), case["precision"])
        nodes = sum(m.info.n[0] * m.info.n[1] for m in b.members)
        out = {k: torch.empty(nodes, dtype=torch.float64, device="cuda") for k in ("T", "u", "v")}
        views, at = [], 0
        for k, m in enumerate(b.members):
            size = m.info.n[0] * m.info.n[1]
            T, u, v = _flow(2, _mesh("tanh", m.info.n[0], 1.5), seed + 1000 * k)
            m.set_fields_device(T, u, v)
            views.append({f: out[f][at:at + size] for f in out})
            at += size
        st.update(batch=b, kept=KEPT[case["precision"]], out=out, views=views)
    elif kind == "predict":
        rng = np.random.default_rng(seed)
        z = features(rng.uniform(6.0, 8.0, case["batch"]), [PR] * case["batch"],
                     [1.5] * case["batch"])
        st.update(net=warmstart.load(WEIGHTS), z=z)
    else:
        net = warmstart.load(WEIGHTS)
        _adam_state(net, seed)
        st["z"], st["target"] = _training_data(case, seed)
        st["net"] = net
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "cavity":
        s = st["solver"]
        s.step(case["steps"])
        s.fields_device(**st["out"])
        return {k: f.to(st["kept"]) for k, f in st["out"].items()}
    if kind == "sample":
        s = st["solver"]
        red = s.reduce()
        du, dT = s.steady_change()
        s.average_add()
        s.fields_device(**st["out"])
        got = {k: f.to(st["kept"]) for k, f in st["out"].items()}
        got["reduced"] = [float(red[k]) for k in REDUCED]
        got["change"] = [float(du), float(dT)]
        return got
    if kind == "batch":
        b = st["batch"]
        b.step(case["steps"])
        for m, view in zip(b.members, st["views"]):
            m.fields_device(**view)
        return {k: f.to(st["kept"]) for k, f in st["out"].items()}
    net = st["net"]
    if kind == "predict":
        return net.forward(st["z"], keep=False)
    y = net.forward(st["z"])
    part, dy = net.mse(y, st["target"])
    grads = net.backward(dy)
    net.adam(lr=LR)
    return {"y": y, "loss": (part.sum() / y.numel()).float(), "grads": dict(grads),
            "params": dict(net.params)}


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------

def _net_layers(batch):
    """(M, N, K) of the network's products: 16 -> 256 -> 8x8x64, then 3x3
    convolutions 64 -> 64 -> 48 -> 32 -> 16 -> 16 -> 3 on 16^2 .. 256^2, 256^2."""
    ch, out = (64, 64, 48, 32, 16, 16), []
    out += [(batch, 256, 16), (batch, 4096, 256)]
    size = 8
    for cin, cout in zip(ch, ch[1:] + (3,)):
        size = size * 2 if cout != 3 else size
        out.append((batch * size * size, cout, 9 * cin))
    return out


def work(case):
    kind = case["kind"]
    if kind in ("cavity", "sample"):
        dim, nodes = case["dim"], float(case["n"]) ** case["dim"]
        q = 14 if dim == 2 else 26
        size = {"fp64": 8, "fp32": 4}.get(case["precision"], 2)
        state = 44.0 if case["precision"] == "fp16neq" else float(q * size)
        fields = (dim + 2) * torch.finfo(KEPT[case["precision"]]).bits / 8.0
        if kind == "sample":
            # the state once, the snapshot and the average in and out, the fields
            return {"bytes": nodes * (state + 4 * 8.0 * (dim + 1) + fields),
                    "flops": nodes * (4.0 * q + 60)}
        # moments, relaxation and interpolation of a node: about 450 operations
        # in 2-D and 1100 in 3-D
        return {"bytes": nodes * (2 * state * case["steps"] + fields),
                "flops": nodes * case["steps"] * (450.0 if dim == 2 else 1100.0)}
    if kind == "batch":
        nodes = float(sum(c["n"] ** 2 for c in _sweep(case, 0)))
        state = {"fp32": 56.0, "fp16neq": 44.0}.get(case["precision"], 28.0)
        fields = 3 * torch.finfo(KEPT[case["precision"]]).bits / 8.0
        return {"bytes": nodes * (2 * state * case["steps"] + fields),
                "flops": nodes * case["steps"] * 450.0}
    layers = _net_layers(case["batch"])
    macs = float(sum(m * n * k for m, n, k in layers))
    weights = float(sum(n * (k + 1) for _, n, k in layers))
    pixels = case["batch"] * 256.0 * 256.0
    if kind == "predict":
        return {"bytes": 2 * weights + 12 * pixels, "flops": 2 * macs}
    # the targets and the prediction, every layer's activations out and back in
    # (BF16, the products' type), the weights and Adam's moments in and out
    acts = float(sum(m * n for m, n, _ in layers[:-1]))
    return {"bytes": 24 * pixels + 4 * acts + 32 * weights, "flops": 6 * macs}


# ---------------------------------------------------------------------------
# the same in 64 bits (plain torch)
# ---------------------------------------------------------------------------

_E = {2: [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)],
      3: [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
          (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
          (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]}


class _Exact:
    """The interpolation-supplemented lattice Boltzmann cavity in FP64: MRT
    collision as matrices, then streaming by quadratic interpolation."""

    def __init__(self, dim, xi, Ra):
        self.dim, self.n = dim, len(xi) - 2
        X = (xi - xi[0]) / (xi[1] - xi[0])
        self.uniform = np.abs(X - np.round(X)).max() < 1e-9
        X = np.round(X) if self.uniform else X
        self.X, self.L = X, X[self.n] - X[1] + 1.0
        self.Ra = Ra
        nu = U_F * self.L * math.sqrt(PR / Ra)
        alpha = U_F * self.L / math.sqrt(PR * Ra)
        self.gbeta = U_F ** 2 / self.L
        self.T0, self.Ts, self.dT = T_COLD, 0.5 * (T_HOT + T_COLD), T_HOT - T_COLD
        s_nu = 1.0 / (3.0 * nu + 0.5)
        s_q = 8.0 * (2.0 - s_nu) / (8.0 - s_nu)
        e = np.array(_E[dim], dtype=np.float64)
        c2 = (e ** 2).sum(1)
        one = np.ones(len(e))
        x, y = e[:, 0], e[:, 1]
        if dim == 2:
            M = [one, 3 * c2 - 4, (9 * c2 ** 2 - 21 * c2 + 8) / 2, x, (3 * c2 - 5) * x, y,
                 (3 * c2 - 5) * y, x * x - y * y, x * y]
            S = [1, s_nu, s_nu, 1, s_q, 1, s_q, s_nu, s_nu]
            self.w = np.where(c2 == 0, 4 / 9, np.where(c2 == 1, 1 / 9, 1 / 36))
            a_T = 20 * math.sqrt(3.0) * alpha - 4
            self.omega, self.t0, self.ti = (4 + a_T) / 10, (1 - a_T) / 5, (4 + a_T) / 20
        else:
            z = e[:, 2]
            p, q = 3 * x * x - c2, y * y - z * z
            M = [one, 19 * c2 - 30, (21 * c2 ** 2 - 53 * c2 + 24) / 2, x, (5 * c2 - 9) * x, y,
                 (5 * c2 - 9) * y, z, (5 * c2 - 9) * z, p, (3 * c2 - 5) * p, q, (3 * c2 - 5) * q,
                 x * y, y * z, x * z, q * x, (z * z - x * x) * y, (x * x - y * y) * z]
            S = [1, s_nu, s_nu, 1, s_q, 1, s_q, 1, s_q, s_nu, s_nu, s_nu, s_nu, s_nu, s_nu, s_nu,
                 s_q, s_q, s_q]
            self.w = np.where(c2 == 0, 1 / 3, np.where(c2 == 1, 1 / 18, 1 / 36))
            a_T = 42 * math.sqrt(3.0) * alpha - 6
            self.omega, self.t0, self.ti = (6 + a_T) / 21, (1 - a_T) / 7, (6 + a_T) / 42
        M = np.array(M)
        self.relax = torch.from_numpy(np.linalg.inv(M) @ np.diag(S) @ M).cuda()
        q = 2 * dim + 1
        eg, cg = e[:q], c2[:q]
        if dim == 2:
            N = [one[:q], eg[:, 0], eg[:, 1], 5 * cg - 4, eg[:, 0] ** 2 - eg[:, 1] ** 2]
            Q = [1, 3 - math.sqrt(3.0), 3 - math.sqrt(3.0), 1, 1]
        else:
            N = [one[:q], eg[:, 0], eg[:, 1], eg[:, 2], 7 * cg - 6, 3 * eg[:, 0] ** 2 - cg,
                 eg[:, 1] ** 2 - eg[:, 2] ** 2]
            Q = [1] + [3 - math.sqrt(3.0)] * 3 + [1, 1, 1]
        N = np.array(N)
        self.relax_g = torch.from_numpy(np.linalg.inv(N) @ np.diag(Q) @ N).cuda()
        self.e, self.qg = _E[dim], q
        self.opp = [self.e.index(tuple(-k for k in v)) for v in self.e]
        col = (-1,) + (1,) * dim
        self.ev = torch.from_numpy(e).cuda()
        self.wv = torch.from_numpy(self.w).cuda().view(col)
        self.tv = torch.tensor([self.t0] + [self.ti] * (q - 1), dtype=torch.float64,
                               device="cuda").view(col)
        # interpolation tables of one axis: departure point X_j -/+ 1
        n = self.n
        self.tab = {}
        for c in (1, -1):
            b = np.clip(np.arange(1, n + 1) - 1, 1, n - 2)
            d, x0, x1, x2 = X[1:n + 1] - c, X[b], X[b + 1], X[b + 2]
            w = np.stack([(d - x1) * (d - x2) / ((x0 - x1) * (x0 - x2)),
                          (d - x0) * (d - x2) / ((x1 - x0) * (x1 - x2)),
                          (d - x0) * (d - x1) / ((x2 - x0) * (x2 - x1))])
            self.tab[c] = (torch.from_numpy(b - 1).cuda(), torch.from_numpy(w).cuda())

    def equilibrium(self, rho, T, u):
        """Deviations f^eq - w, g^eq, and e.u of every velocity."""
        eu = torch.tensordot(self.ev, torch.stack(u), 1)
        usq = sum(k * k for k in u)
        f = self.wv * (rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * usq) - 1)
        g = self.tv * T + 0.5 * eu[:self.qg] * T
        return f, g, eu

    def macro(self, f, g):
        """rho, T - Ts, u of pre-collision deviations and the force F_y."""
        rho = 1 + f.sum(0)
        T = g.sum(0)
        j = [sum(v[a] * f[i] for i, v in enumerate(self.e) if v[a]) for a in range(self.dim)]
        F = rho * self.gbeta * (T + self.Ts - self.T0)
        j[1] = j[1] + 0.5 * F
        return rho, T, [k / rho for k in j], F

    def start(self, T, u):
        T = T - self.Ts
        self.f, self.g, _ = self.equilibrium(torch.ones_like(T), T, u)

    def step(self):
        """Collide, stream."""
        f, g = self.f, self.g
        rho, T, u, F = self.macro(f, g)
        feq, geq, eu = self.equilibrium(rho, T, u)
        ey = self.ev[:, 1].view(self.wv.shape)
        force = self.wv * (3 * (ey * F - u[1] * F) + 9 * eu * ey * F)
        del eu
        flat = lambda t: t.reshape(t.shape[0], -1)     # noqa: E731
        post = f + force - (self.relax @ flat(f - feq + 0.5 * force)).view_as(f)
        del feq, force
        postg = g - (self.relax_g @ flat(g - geq)).view_as(g)
        del geq
        self.f = torch.stack([self._pull(post, i) for i in range(len(self.e))])
        gg = []
        for i in range(self.qg):
            t = self._pull(postg, i)
            if self.e[i][0]:                # anti-bounce-back on the isothermal x-walls
                at = 0 if self.e[i][0] > 0 else self.n - 1
                wall = (T_HOT if at == 0 else T_COLD) - self.Ts
                t[..., at] = self.omega * wall - postg[self.opp[i]][..., at]
            gg.append(t)
        self.g = torch.stack(gg)

    def _pull(self, post, i):
        t = post[i]
        for a, c in enumerate(self.e[i]):
            if not c:
                continue
            d = self.dim - 1 - a            # tensor axis of direction a
            if self.uniform:
                t = torch.roll(t, c, d)
                continue
            b, w = self.tab[c]
            shape = [1] * self.dim
            shape[d] = -1
            t = sum(w[k].view(shape) * t.index_select(d, b + k) for k in range(3))
        t = t.clone() if t.data_ptr() == post[i].data_ptr() else t
        for a, c in enumerate(self.e[i]):   # half-way bounce-back behind a wall
            if c:
                d = self.dim - 1 - a
                at = 0 if c > 0 else self.n - 1
                t.select(d, at).copy_(post[self.opp[i]].select(d, at))
        return t

    def fields(self):
        rho, T, u, _ = self.macro(self.f, self.g)
        return dict(zip(("rho", "T", "u", "v", "w"), [rho, T + self.Ts] + u))

    def reduced(self):
        """The volume and wall averages named in REDUCED."""
        X, n, L = self.X, self.n, self.L
        W1 = torch.from_numpy(0.5 * (X[2:] - X[:-2])).cuda()
        W = wp = torch.ones((), dtype=torch.float64, device="cuda")
        for a in range(self.dim):
            shape = [1] * self.dim
            shape[self.dim - 1 - a] = -1
            W = W * W1.view(shape)
            if a:
                wp = wp * W1.view(shape)
        fl = self.fields()
        rho, T = fl["rho"], fl["T"]
        u = [fl[k] for k in "uvw"[:self.dim]]
        u2, uv2 = sum(k * k for k in u), u[0] ** 2 + u[1] ** 2
        vol, area, sp = L ** self.dim, L ** (self.dim - 1), u2.sqrt()
        q = (X[2] - X[1]) / (X[1] - X[0])
        cw, c1, c2 = -4 * q * (q + 1), (2 * q + 1) ** 2, -1.0

        def wall(Tw, a, b):
            t = cw * Tw * area + c1 * (wp * T[..., a:a + 1]).sum() \
                + c2 * (wp * T[..., b:b + 1]).sum()
            return float(t) / (q * (2 * q + 1))

        sra = math.sqrt(self.Ra / PR)
        return {"Nu": math.sqrt(self.Ra * PR) * float((W * u[0] * (T - self.T0)).sum())
                / (U_F * self.dT * vol) + 1.0,
                "Nu_hot": -wall(T_HOT, 0, 1) * L / (self.dT * area),
                "Nu_cold": wall(T_COLD, n - 1, n - 2) * L / (self.dT * area),
                "Re": sra * math.sqrt(float((W * u2).sum()) / vol) / U_F,
                "Re_uv": sra * math.sqrt(float((W * uv2).sum()) / vol) / U_F,
                "Re_mean": sra * float((W * sp).sum()) / (U_F * vol),
                "mass": float((W * rho).sum()), "max_speed": float(sp.max()) / U_F}


def _exact_cavity(dim, n, mesh, a, Ra, steps, seed):
    xi = _mesh(mesh, n, a)
    x = _Exact(dim, xi, Ra)
    T, *u = _flow(dim, xi, seed)
    x.start(T, u)
    before = x.fields()
    for _ in range(steps):
        x.step()
    return x, before


def _exact_net(case, seed):
    """Outputs, loss, gradients and updated weights of the network in FP64."""
    net = warmstart.load(WEIGHTS)
    P = {k: v.double() for k, v in net.params.items()}
    if case["kind"] == "predict":
        rng = np.random.default_rng(seed)
        z = features(rng.uniform(6.0, 8.0, case["batch"]), [PR] * case["batch"],
                     [1.5] * case["batch"])
    else:
        z, target = _training_data(case, seed)
        target = target.double()
    for t in P.values():
        t.requires_grad_(True)
    size, ch = 8, (64, 64, 48, 32, 16, 16, 3)
    h = torch.tanh(torch.from_numpy(z).cuda().double() @ P["W1"] + P["b1"])
    x = torch.tanh(h @ P["W2"] + P["b2"]).view(-1, size, size, ch[0]).permute(0, 3, 1, 2)
    for k in range(6):
        last = k == 5
        if not last:
            x = x.repeat_interleave(2, 2).repeat_interleave(2, 3)
        H = x.shape[2]
        cols = torch.nn.functional.pad(x, (1, 1, 1, 1))
        taps = P[f"Wc{k}"][:9 * ch[k]].view(9, ch[k], ch[k + 1])
        y = P[f"bc{k}"].view(1, -1, 1, 1)
        for t in range(9):
            y = y + torch.einsum("bchw,co->bohw",
                                 cols[:, :, t // 3:t // 3 + H, t % 3:t % 3 + H], taps[t])
        x = y if last else torch.tanh(y)
    y = x.permute(0, 2, 3, 1)
    if case["kind"] == "predict":
        return y.detach().contiguous()
    loss = ((y - target) ** 2).mean()
    loss.backward()
    _adam_state(net, seed)
    t, b1, b2 = ADAM_STEP + 1, 0.9, 0.999
    grads, params = {}, {}
    for name, w in P.items():
        g = w.grad
        m = b1 * net.m[name].double() + (1 - b1) * g
        v = b2 * net.v[name].double() + (1 - b2) * g * g
        grads[name] = g
        params[name] = w.detach() - LR * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + 1e-8)
    return {"y": y.detach().contiguous(), "loss": loss.detach(), "grads": grads, "params": params}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("predict", "train"):
        return _exact_net(case, seed)
    with torch.no_grad():
        if kind == "batch":
            got = {"T": [], "u": [], "v": []}
            for k, c in enumerate(_sweep(case, seed)):
                x, _ = _exact_cavity(2, c["n"], "tanh", 1.5, c["Ra"], case["steps"],
                                     seed + 1000 * k)
                fl = x.fields()
                for f in got:
                    got[f].append(fl[f].reshape(-1))
            return {f: torch.cat(v) for f, v in got.items()}
        x, before = _exact_cavity(case["dim"], case["n"], case["mesh"], case["a"], case["Ra"],
                                  case["steps"], seed)
        got = x.fields()
        if kind == "sample":
            names = "uvw"[:case["dim"]]
            du = sum((got[k] - before[k]) ** 2 for k in names).sqrt().sum()
            u0 = sum(before[k] ** 2 for k in names).sqrt().sum()
            dT = (got["T"] - before["T"]).abs().sum()
            red = x.reduced()
            got["change"] = [float(du / u0), float(dT / (before["T"] - T_COLD).abs().sum())]
            got["reduced"] = [red[k] for k in REDUCED]
        return got
