"""The work whose speed is measured: whole jobs through the package's public calls.

A lattice job is what a user's program does with a solver: hand over the initial
fields, advance, read the fields back.  The fields are FP64 device tensors (the
form in which a GPU program holds them), so a pass is ``Solver.init``,
``Solver.step`` (or ``step_diagnostics`` at intervals) and ``Solver.moments``; the
solver and its memory are kept from job to job.  A sweep does the same for the
members of a ``Batch``; a training job runs Adam steps of the surrogate network
from given weights.

``exact`` restates the method (pull, moments, equilibrium by the moment rule,
BGK relaxation; and the network with its gradients and Adam) in plain FP64 torch.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

from paper_1402_5487_gb300 import batch as B
from paper_1402_5487_gb300 import inputs as I
from paper_1402_5487_gb300 import plbm
from paper_1402_5487_gb300 import surrogate as SG

SETS = {"013": I.SET_013, "012": I.SET_012}
#: node updates of the largest listed lattice job (2048 x 2048, 100 steps)
MOST_UPDATES = 2048 * 2048 * 100
#: the same for FP64 jobs, whose updates cost more
MOST_UPDATES_F64 = 1024 * 1024 * 40
#: populations updated by the largest 3D job
MOST_3D = 256 * 256 * 128 * 10


def _lattice(name, nx, ny, steps, prec, **kw):
    c = {"name": name, "kind": "kh", "dim": 2, "nx": nx, "ny": ny, "nz": 1, "set": "013", "omega": 1.3, "theta0": 1.0,
         "prec": prec, "steps": steps, "every": 0}
    c.update(kw)
    return c


def listed():
    return [
        # The 1000-node thermal shock tube run to the time at which it is compared with the exact
        # Riemann solution: the smallest lattice a user runs, hundreds of very short steps.
        _lattice("tube_1000_f64", 1000, 1, 361, "f64", kind="tube", dim=1, omega=1.5, theta0=0.5),
        # The paper's own shear layer, in the precision in which it stays stable.
        _lattice("paper_128_f64", 128, 128, 200, "f64", kind="paper", set="012", omega=1.9, theta0=1.0 / 2.56),
        # The double shear layer at a size that stays in the second-level cache.
        _lattice("kh_512_f32", 512, 512, 200, "f32"),
        # The benchmark's workload.
        _lattice("kh_2048_f32", 2048, 2048, 100, "f32"),
        # An odd side: the lattice cannot be stored as row pairs.
        _lattice("kh_2047_f32", 2047, 2047, 60, "f32"),
        # 16-bit storage at the benchmark's size.
        _lattice("kh_2048_f16", 2048, 2048, 100, "f16dev"),
        # 16-bit storage on a rectangle, with the global sums read every ten steps, as a monitored run does.
        _lattice("kh_1500x900_bf16_diag", 1500, 900, 100, "bf16dev", every=10),
        # An FP64 reference run.
        _lattice("kh_1024_f64", 1024, 1024, 40, "f64"),
        # Three dimensions, 32-bit storage.
        _lattice("kh3_128_f32", 128, 128, 20, "f32", kind="kh3", dim=3, nz=128),
        # Three dimensions, 16-bit storage.
        _lattice("kh3_256x256x128_f16", 256, 256, 10, "f16dev", kind="kh3", dim=3, nz=128),
        # A parameter sweep: lattices of every size, both parities, advanced together.
        {"name": "sweep_16_f32", "kind": "sweep", "instances": 16, "size_lo": 64, "size_hi": 1024, "sizes_seed": 1000,
         "prec": "f32", "steps": 40},
        # Training of the surrogate on minibatches of 16 snapshots of 256 x 256 nodes.
        {"name": "train_16", "kind": "train", "batch": 16, "H": 256, "W": 256, "steps": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "paper", "kh", "kh", "kh", "kh3", "sweep", "train"])
    if kind == "tube":
        c = _lattice("", _log_int(rng, 200, 20000), 1, rng.randint(100, 400), rng.choice(["f64", "f64", "f32"]), kind="tube",
                     dim=1, omega=1.5, theta0=0.5)
    elif kind == "paper":
        n = rng.randint(64, 256)
        c = _lattice("", n, n, rng.randint(50, 200), rng.choice(["f64", "f64", "f32"]), kind="paper", set="012", omega=1.9,
                     theta0=1.0 / 2.56)
    elif kind == "kh":
        prec = rng.choice(["f32", "f32", "f16dev", "bf16dev", "f64"])
        hi = 1024 if prec == "f64" else 2048
        nx, ny = _log_int(rng, 64, hi), _log_int(rng, 64, hi)
        most = MOST_UPDATES_F64 if prec == "f64" else MOST_UPDATES
        steps = max(1, min(rng.randint(20, 200), most // (nx * ny)))
        c = _lattice("", nx, ny, steps, prec, every=rng.choice([0, 0, 10]))
    elif kind == "kh3":
        prec = rng.choice(["f32", "f16dev", "bf16dev"])
        nx, ny, nz = (_log_int(rng, 16, 192) for _ in range(3))
        steps = max(1, min(rng.randint(5, 40), MOST_3D // (nx * ny * nz)))
        c = _lattice("", nx, ny, steps, prec, kind="kh3", dim=3, nz=nz)
    elif kind == "sweep":
        return {"kind": "sweep", "instances": rng.randint(4, 16), "size_lo": 64, "size_hi": rng.randint(200, 1024),
                "sizes_seed": rng.randrange(1 << 20), "prec": rng.choice(["f32", "f16dev", "bf16dev"]), "steps": rng.randint(10, 40)}
    else:
        return {"kind": "train", "batch": rng.randint(1, 16), "H": rng.randint(64, 256), "W": 128 * rng.randint(1, 2),
                "steps": rng.randint(2, 4)}
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _noise(g, *shape):
    return 1e-4 * (2.0 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 1.0)


def _fields(c, seed):
    """Initial fields of a lattice job (rho, u_x[, u_y[, u_z]], theta), FP64 on the device."""
    g = _gen(seed)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    ax = dict(device="cuda", dtype=torch.float64)
    pick = torch.rand(4, generator=g, **ax).tolist()
    if c["kind"] == "tube":
        left = torch.arange(nx, device="cuda")[None, :] < nx // 2
        rho = torch.where(left, 1.08 + 0.04 * pick[0], 1.0)
        u = 1e-3 * pick[1] * torch.sin(2 * math.pi * torch.arange(nx, **ax) / nx)[None, :]
        return [rho.double(), u, torch.zeros_like(u), torch.full((1, nx), 0.5, **ax)]
    x = torch.arange(nx, **ax)
    if c["kind"] == "kh3":
        y, z = torch.arange(ny, **ax)[None, :, None], torch.arange(nz, **ax)[:, None, None]
        x = x[None, None, :]
        one = torch.ones((nz, ny, nx), **ax)
        u0 = 0.08 + 0.02 * pick[0]
        ux = u0 * torch.tanh(((z - nz / 2).abs() - nz / 4) / (nz / 16)) * one + _noise(g, nz, ny, nx)
        uy = 0.003 * torch.sin(2 * math.pi * (x / nx + pick[1])) * one + _noise(g, nz, ny, nx)
        uz = 0.005 * torch.sin(2 * math.pi * (x / nx + y / ny + pick[2])) * one + _noise(g, nz, ny, nx)
        return [one, ux.contiguous(), uy.contiguous(), uz.contiguous(), c["theta0"] * one]
    y = torch.arange(ny, **ax)[:, None]
    x = x[None, :]
    one = torch.ones((ny, nx), **ax)
    if c["kind"] == "paper":
        s = math.sqrt(c["theta0"])
        u0 = (0.06 + 0.01 * pick[0]) * s
        yy = y / ny
        ux = u0 * torch.where(yy <= 0.5, torch.tanh(80.0 * (yy - 0.25)), torch.tanh(80.0 * (0.75 - yy))) * one
        uy = u0 * 0.05 * torch.sin(2 * math.pi * (x / nx + 0.25 + pick[1])) * one
    else:
        u0 = 0.08 + 0.02 * pick[0]
        ux = u0 * torch.tanh(((y - ny / 2).abs() - ny / 4) / (ny / 80.0)) * one + _noise(g, ny, nx)
        uy = 0.005 * torch.sin(2 * math.pi * (x / nx + pick[1])) * one + _noise(g, ny, nx)
    return [one, ux.contiguous(), uy.contiguous(), c["theta0"] * one]


def _sweep_instances(c):
    """Members of a sweep: sides uniform over the integers of the range; velocity set, omega and theta0 drawn from
    the part of the sweep's parameter range in which both sets are linearly stable and non-negative."""
    out = []
    for k in range(c["instances"]):
        rng = np.random.default_rng(c["sizes_seed"] + k)
        L = int(rng.integers(c["size_lo"], c["size_hi"] + 1))
        v = "013" if k % 2 else "012"
        th = float(rng.uniform(0.6, 1.2 if v == "013" else 0.9))
        out.append(I.Instance(index=k, L=L, v=SETS[v], omega=float(rng.uniform(1.0, 1.3)), theta0=th, kind="kh", seed=k))
    return out


def _sweep_fields(c, seed):
    return [_fields({"kind": "kh", "nx": i.L, "ny": i.L, "nz": 1, "theta0": i.theta0}, 1000 * int(seed) + i.index)
            for i in _sweep_instances(c)]


def _snapshots(c, seed):
    """FP32 snapshot stack [2 n][H W][4] (rho, u_x, u_y, theta) of n shear layers, each at two times: the layer
    widens and its cross flow grows, as over 32 lattice steps; and the pairs' indices."""
    n, H, W = 2 * c["batch"], c["H"], c["W"]
    g = _gen(seed)
    ax = dict(device="cuda", dtype=torch.float64)
    y, x = torch.arange(H, **ax)[:, None], torch.arange(W, **ax)[None, :]
    stack = torch.empty((2 * n, H * W, 4), device="cuda", dtype=torch.float32)
    for k in range(n):
        a, b, d, e = torch.rand(4, generator=g, **ax).tolist()
        for t in range(2):
            u0, width = 0.06 + 0.04 * a, H / (80.0 - 40.0 * b) * (1.0 + 0.1 * t)
            grow = 1.0 + 0.2 * t
            ux = u0 * torch.tanh(((y - H / 2).abs() - H / 4) / width) * (1.0 + 0.02 * grow * torch.cos(2 * math.pi * (x / W + d)))
            uy = 0.005 * grow * torch.sin(2 * math.pi * (x / W + e)) * torch.cos(2 * math.pi * y / H)
            p = 2e-4 * grow * torch.cos(2 * math.pi * (x / W + d)) * torch.sin(4 * math.pi * y / H)
            f = torch.stack([1.0 + p, ux + 0 * p, uy + 0 * p, 1.0 + 0.5 * p], dim=-1)
            f = f + 0.1 * torch.cat([0.1 * _noise(g, H, W, 1), _noise(g, H, W, 2), 0.1 * _noise(g, H, W, 1)], dim=-1)
            stack[2 * k + t] = f.reshape(H * W, 4).float()
    return stack, np.array([(2 * k, 2 * k + 1) for k in range(n)], dtype=np.int32)


CIN, COUT = (4, 64, 64, 64, 64, 64), (64, 64, 64, 64, 64, 4)


def _weights(seed):
    """Weights to start training from, W[3][3][cin][cout] then b[cout] per layer: normal, variance 2 / (9 cin), the
    last layer scaled by 0.1, biases zero."""
    rng = np.random.default_rng(int(seed))
    out = []
    for i, o in zip(CIN, COUT):
        out += [rng.normal(0.0, (0.1 if o == 4 else 1.0) * math.sqrt(2.0 / (9 * i)), 9 * i * o), np.zeros(o)]
    return np.concatenate(out).astype(np.float32)


# ---------------------------------------------------------------------------
# Passes
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    if c["kind"] == "sweep":
        return {"c": c, "b": B.Batch(_sweep_instances(c), prec=c["prec"]), "fields": _sweep_fields(c, seed)}
    if c["kind"] == "train":
        stack, pairs = _snapshots(c, seed)
        net = SG.Surrogate(c["batch"], c["H"], c["W"], seed=int(seed))
        net.set_norm(*SG.fit_norm(stack, pairs))
        return {"c": c, "net": net, "stack": stack, "pairs": pairs, "p0": _weights(seed), "seed": int(seed)}
    fixed = {"bc": "fixed", "left_state": (1.1, 0.0, 0.5), "right_state": (1.0, 0.0, 0.5)} if c["kind"] == "tube" else {}
    s = plbm.Solver(c["dim"], SETS[c["set"]], c["omega"], c["nx"], c["ny"], theta0=c["theta0"], prec=c["prec"], nz=c["nz"],
                    **fixed)
    return {"c": c, "s": s, "fields": _fields(c, seed)}


def run(state):
    c = state["c"]
    if c["kind"] == "sweep":
        b = state["b"]
        with torch.cuda.stream(b.stream):
            for s, f in zip(b.solvers, state["fields"]):
                s.init(*f)
            b.step(c["steps"])
            return [s.moments(on_device=True) for s in b.solvers]
    if c["kind"] == "train":
        net = state["net"]
        net.set_params(state["p0"])
        net.train(state["stack"], state["pairs"], c["steps"], batch=c["batch"], lr=1e-3, seed=state["seed"])
        return net.params()
    s, f = state["s"], state["fields"]
    if c["dim"] == 3:
        s.init(f[0], f[1], f[2], theta=f[4], uz=f[3])
    else:
        s.init(*f)
    if not c["every"]:
        s.step(c["steps"])
        return s.moments(on_device=True)
    said, left = [], c["steps"]
    while left > 0:
        n = min(c["every"], left)
        d = s.step_diagnostics(n)
        said.append([d[k] for k in ("mass", "jx", "jy", "energy", "rho_min", "theta_min")])
        left -= n
    return s.moments(on_device=True), np.array(said)


def _updates(c):
    if c["kind"] == "sweep":
        return sum(i.L * i.L for i in _sweep_instances(c)) * c["steps"]
    return c["nx"] * c["ny"] * c["nz"] * c["steps"]


def work(case):
    """Bytes: the fields read and written once each (the populations are the job's own state).  Operations: a node
    update's sums (two per population: its row's and its column's or plane's), its relaxation (a product, a scaled
    difference and a sum: 4) and the moments and the rule per axis (45)."""
    c = case
    if c["kind"] == "train":
        pix, n = c["batch"] * c["H"] * c["W"], 2 * 4 * 64 * 9 * 2 + 4 * 2 * 64 * 64 * 9
        params = 9 * (2 * 4 * 64 + 4 * 64 * 64) + 5 * 64 + 4
        return {"bytes": c["steps"] * pix * 4 * 4 * 2 + 2 * 4 * params, "flops": c["steps"] * pix * n * 3}
    dim = c.get("dim", 2)
    nodes = _updates(c) // c["steps"]
    return {"bytes": nodes * 8 * 2 * (2 + max(dim, 2)), "flops": nodes * c["steps"] * (6 * 5 ** dim + 45 * dim)}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------
def _coefficients(v):
    """c_in: coefficient of v^n in the Lagrange polynomial of velocity i, correctly rounded."""
    out = []
    for i, vi in enumerate(v):
        poly, den = [Fraction(1)], Fraction(1)
        for j, vj in enumerate(v):
            if j != i:
                poly = [(poly[k - 1] if k else 0) - (vj * poly[k] if k < len(poly) else 0) for k in range(len(poly) + 1)]
                den *= vi - vj
        out.append([float(a / den) for a in poly])
    return out


def _rule(C, u, th):
    mu = [torch.ones_like(u), u]
    for n in range(1, len(C) - 1):
        mu.append(u * mu[n] + n * th * mu[n - 1])
    return [sum(row[n] * mu[n] for n in range(len(C))) for row in C]


class _Exact:
    def __init__(self, dim, v, omega, fixed=None):
        self.dim, self.v, self.omega, self.C = dim, v, omega, _coefficients(v)
        self.ends = None
        if fixed:
            t = lambda a: torch.tensor([a], device="cuda", dtype=torch.float64)
            self.ends = [[float(rho * r) for r in _rule(self.C, t(u), t(th))] for rho, u, th in fixed]

    def feq(self, rho, u, th):
        r = [_rule(self.C, a, th) for a in u]
        if self.dim == 1:
            return [rho * a for a in r[0]]
        if self.dim == 2:
            return [rho * a * b for a in r[0] for b in r[1]]
        return [rho * a * b * c for a in r[0] for b in r[1] for c in r[2]]

    def moments(self, f):
        q, d = len(self.v), self.dim
        sums = [[0] * q for _ in range(d)]
        for p, g in enumerate(f):
            for a in range(d):
                i = (p // q ** (d - 1 - a)) % q
                sums[a][i] = sums[a][i] + g
        rho = sum(sums[0])
        u = [sum(w * s for w, s in zip(self.v, sums[a])) / rho for a in range(d)]
        e = sum(w * w * s for a in range(d) for w, s in zip(self.v, sums[a]))
        th = (e / rho - sum(a * a for a in u)) / d
        return rho, u, th, e

    def pull(self, f):
        q, d = len(self.v), self.dim
        out = []
        for p, g in enumerate(f):
            vel = [self.v[(p // q ** (d - 1 - a)) % q] for a in range(d)]
            if d == 1 and self.ends:
                h = torch.roll(g, vel[0], -1)
                if vel[0] > 0:
                    h[..., :vel[0]] = self.ends[0][p]
                elif vel[0] < 0:
                    h[..., vel[0]:] = self.ends[1][p]
            else:   # velocity components (x, y, z) shift the axes (-1, -2, -3)
                h = torch.roll(g, vel, [-1 - a for a in range(d)])
            out.append(h)
        return out

    def step(self, f):
        f = self.pull(f)
        rho, u, th, _ = self.moments(f)
        fe = self.feq(rho, u, th)
        for p in range(len(f)):
            f[p].mul_(1.0 - self.omega).add_(fe[p], alpha=self.omega)
            fe[p] = None
        return f


def _exact_lattice(dim, v, omega, fields, steps, every=0, fixed=None):
    L = _Exact(dim, v, omega, fixed)
    rho, u, th = fields[0], list(fields[1:1 + dim]), fields[-1]
    f = L.feq(rho, u, th)
    said = []
    for s in range(steps):
        f = L.step(f)
        if every and ((s + 1) % every == 0 or s + 1 == steps):
            r, w, t, e = L.moments(f)
            said.append([float(r.sum()), float((r * w[0]).sum()), float((r * w[1]).sum()), float(e.sum()), float(r.min()),
                         float(t.min())])
    r, w, t, _ = L.moments(f)
    if dim == 1:
        w = [w[0], torch.zeros_like(r)]
    out = (r, *w, t)
    return (out, np.array(said)) if every else out


def _conv(X, W, b):
    """3 x 3 convolution with circular padding, NHWC, weights [3][3][cin][cout]."""
    out = b
    for ky in range(3):
        for kx in range(3):
            out = out + torch.roll(X, (1 - ky, 1 - kx), (1, 2)) @ W[ky, kx]
    return out


def _exact_train(c, seed):
    stack, pairs = _snapshots(c, seed)
    norm = [torch.tensor(np.asarray(a, dtype=np.float32), device="cuda").double() for a in SG.fit_norm(stack, pairs)]
    p = torch.tensor(_weights(seed), device="cuda").double().requires_grad_()
    m, v2 = torch.zeros_like(p), torch.zeros_like(p)
    rng = np.random.default_rng(int(seed))
    order, pos, n = rng.permutation(len(pairs)), 0, c["batch"]
    for t in range(1, c["steps"] + 1):
        if pos + n > len(order):
            order, pos = rng.permutation(len(pairs)), 0
        sel = pairs[order[pos:pos + n]]
        pos += n
        a, b = (stack[torch.from_numpy(sel[:, k].astype(np.int64)).cuda()].double() for k in (0, 1))
        x = ((a - norm[0]) / norm[1]).reshape(n, c["H"], c["W"], 4)
        y = ((b - a - norm[2]) / norm[3]).reshape(n, c["H"], c["W"], 4)
        h, off = x, 0
        for i in range(6):
            k = 9 * CIN[i] * COUT[i]
            h = _conv(h, p[off:off + k].reshape(3, 3, CIN[i], COUT[i]), p[off + k:off + k + COUT[i]])
            off += k + COUT[i]
            if i < 5:
                h = torch.relu(h)
        (g,) = torch.autograd.grad(((h - y) ** 2).mean(), p)
        with torch.no_grad():
            m = 0.9 * m + 0.1 * g
            v2 = 0.999 * v2 + 0.001 * g * g
            p -= 1e-3 * (m / (1 - 0.9 ** t)) / ((v2 / (1 - 0.999 ** t)).sqrt() + 1e-8)
    # the gradients of the last step are those of weights that already differ: no value
    return p.detach(), None


def exact(case, seed):
    c = case
    if c["kind"] == "train":
        return _exact_train(c, seed)
    if c["kind"] == "sweep":
        return [_exact_lattice(2, i.v, i.omega, f, c["steps"]) for i, f in zip(_sweep_instances(c), _sweep_fields(c, seed))]
    fixed = [(1.1, 0.0, 0.5), (1.0, 0.0, 0.5)] if c["kind"] == "tube" else None
    return _exact_lattice(c["dim"], SETS[c["set"]], c["omega"], _fields(c, seed), c["steps"], c["every"], fixed)
