"""Performance cases of the binary Shan-Chen capillary library and its surrogate.

Each case is one thing a user's program does through the public classes
(`Lattice`, `Slab`, `Network`, `Surrogate`): a capillary or a batch of them is
advanced and its fields, fronts or populations are read; the surrogate is
evaluated, differentiated or fitted.  Sizes are those of the workloads, the
calibration module, the tests and the benchmark.

Runs stay in the band where the model is finite for 10^5 steps (G = 1.0 to
1.1, tau >= 1, couplings -0.5 to 0.3; the density-ratio species at G = 1.2),
so a case can be stepped on for as long as it is timed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as W
from paper_0807_0602_gb300 import slab as S
from paper_0807_0602_gb300 import surrogate as M
from paper_0807_0602_gb300.lbm import Lattice

# 1:3 density ratio of the paper's species model (rest fractions, masses)
RATIO_ALPHA, RATIO_MASS = (4.0 / 9.0, 0.8), (1.0, 25.0 / 9.0)
# steps an autotuned program takes before it measures: the tuner runs in them
TUNE_STEPS = 2000
# floating-point operations of one node's step (two species; sums, products
# and the reciprocal of Eqs. 2-11, each shared term once)
FLOPS_NODE = 260
ELEM = {"f64": 8, "f32": 4, "f16s": 2}
# parameters of the network, products per row of its forward pass
MLP_MACS = 6 * 128 + 2 * 128 * 128 + 128 * 3


def listed():
    return [
        # the smallest capillary of the workloads, logged every 50 steps, fronts
        # read at the end: launches and latency
        dict(name="capillary_256x32_f32", kind="capillary", nx=256, ny=32, precision="f32", steps=300, log_every=50),
        # one capillary cut into two x-slabs held by one process, halo exchange
        # after every step: single steps and column copies
        dict(name="slabs_2x1024x66_f32", kind="slabs", nx=2048, ny=66, parts=2, precision="f32", steps=20),
        # the benchmark workload: 8192 x 160, autotuned as the benchmark does
        dict(name="capillary_8192x160_f32", kind="capillary", nx=8192, ny=160, precision="f32", steps=100,
             log_every=50, autotune=True),
        # FP16-shifted storage on the same grid, with the library's own choice of kernel
        dict(name="capillary_8192x160_f16s", kind="capillary", nx=8192, ny=160, precision="f16s", steps=100,
             log_every=0),
        # the density-ratio species on a verification capillary of ragged size,
        # whole-fluid velocity read at the end
        dict(name="ratio_4095x67_f32", kind="capillary", nx=4095, ny=67, precision="f32", steps=100, log_every=0,
             ratio=True, velocity=True),
        # the FP64 reference capillary, logged
        dict(name="capillary_2048x130_f64", kind="capillary", nx=2048, ny=130, precision="f64", steps=50,
             log_every=50),
        # FP64 droplets that judge the surrogate's proposals: nine couplings of
        # one calibration row, angles read from the host fields
        dict(name="droplets_judge_9x128x80_f64", kind="droplets", runs=9, nx=128, ny=80, radius=24.0,
             precision="f64", steps=100),
        # a quarter of the droplet calibration batch
        dict(name="droplets_256x256x128_f32", kind="droplets", runs=256, nx=256, ny=128, radius=40.0,
             precision="f32", steps=50),
        # an eighth of the uneven capillary ensemble
        dict(name="ensemble_64_uneven_f32", kind="ensemble", runs=64, sizes=3, precision="f32", steps=50),
        # proposals: the network on one grid of candidate couplings
        dict(name="mlp_forward_1201", kind="forward", rows=1201),
        # gradients of the loss over a full batch
        dict(name="mlp_gradients_4096", kind="gradients", rows=4096),
        # training on the calibration samples, minibatches of 512
        dict(name="surrogate_fit_960", kind="fit", samples=960, batch=512, steps=20),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["capillary", "capillary", "capillary", "slabs", "droplets", "ensemble", "forward", "gradients",
                       "fit"])
    if kind == "capillary":
        precision = rng.choice(["f32", "f32", "f16s", "f64"])
        nx = _logint(rng, 64, 8192 if precision != "f64" else 2048)
        ny = rng.randint(18, 160 if precision != "f64" else 130)
        ratio = precision != "f16s" and rng.random() < 0.25
        return dict(kind=kind, nx=nx, ny=ny, precision=precision,
                    steps=rng.randint(20, 100 if precision != "f64" else 50), log_every=rng.choice([0, 20, 50]),
                    ratio=ratio, velocity=rng.random() < 0.3)
    if kind == "slabs":
        return dict(kind=kind, nx=_logint(rng, 128, 4096), ny=rng.randint(18, 130), parts=rng.randint(2, 3),
                    precision=rng.choice(["f32", "f64"]), steps=rng.randint(5, 20))
    if kind == "droplets":
        precision = rng.choice(["f32", "f32", "f64"])
        nx = rng.choice([128, 192, 256])
        return dict(kind=kind, runs=_logint(rng, 1, 256 if precision == "f32" else 16), nx=nx, ny=rng.randint(64, 128),
                    radius=nx * 0.16, precision=precision, steps=rng.randint(20, 50))
    if kind == "ensemble":
        return dict(kind=kind, runs=_logint(rng, 2, 64), sizes=rng.randint(0, 10 ** 6), precision="f32",
                    steps=rng.randint(10, 40))
    if kind == "forward":
        return dict(kind=kind, rows=_logint(rng, 1, 65536))
    if kind == "gradients":
        return dict(kind=kind, rows=_logint(rng, 16, 4096))
    return dict(kind=kind, samples=_logint(rng, 64, 960), batch=_logint(rng, 32, 512), steps=rng.randint(5, 20))


# ---- inputs -----------------------------------------------------------------

def _rng(seed, tag):
    return np.random.Generator(np.random.PCG64([int(seed), tag]))


def _capillary(case, seed):
    """A capillary across the middle three quarters of the box, an outer slit
    above the top plate where the box is tall enough, liquid up to a front
    inside the capillary; densities carry a small random deviation."""
    r = _rng(seed, 1)
    nx, ny = case["nx"], case["ny"]
    y_top = ny - 1 if ny < 30 else int(ny * 0.81)
    geom = W.capillary_geometry(nx, ny, nx // 8, nx - nx // 8, 0, y_top)
    if case.get("ratio"):
        prm = W.params(1.2, 1.0, 1.0, r.uniform(-0.3, -0.1), 0.0)
        prm.update(alpha=RATIO_ALPHA, mass=RATIO_MASS)
    else:
        prm = W.params(r.uniform(1.0, 1.05), 1.0, 1.0 if case["precision"] != "f64" else r.uniform(1.0, 1.2),
                       r.uniform(-0.5, -0.1), 0.0)
    front = int(nx * r.uniform(0.25, 0.4))
    nA, nB = W.slab_fields(geom, 0, front)
    nA *= 1.0 + 1e-3 * r.standard_normal(nA.shape)
    nB *= 1.0 + 1e-3 * r.standard_normal(nB.shape)
    return dict(geom=geom, params=prm, init=("fields", nA, nB))


def _droplets(case, seed):
    """Sessile droplets on a wall at y = 0, couplings over the stable band."""
    r = _rng(seed, 2)
    out = []
    for _ in range(case["runs"]):
        geom = dict(nx=case["nx"], ny=case["ny"], cap_x0=0, cap_x1=case["nx"], y_bot=0, y_top=-1)
        prm = W.params(r.uniform(1.0, 1.1), 1.0, r.uniform(1.0, 1.5), r.uniform(-0.5, 0.3), 0.0)
        out.append(dict(geom=geom, params=prm, init=("droplet", case["nx"] / 2.0 + r.uniform(-4, 4), 0.5,
                                                     case["radius"] * r.uniform(0.9, 1.1))))
    return out


def _ensemble(case, seed):
    """Uneven capillaries: the sizes belong to the case, parameters and fronts to the seed."""
    sizes = W.batch_uneven_capillaries_stable(case["runs"], seed=case["sizes"])
    r = _rng(seed, 3)
    out = []
    for run in sizes:
        g = run["geom"]
        prm = W.params(r.uniform(1.0, 1.1), 1.0, r.uniform(1.0, 1.5), r.uniform(-0.5, 0.3), 0.0)
        L = g["nx"] // 2
        out.append(dict(geom=g, params=prm, init=("slab", int(L * r.uniform(0.4, 0.6)), int(L * r.uniform(1.2, 1.4)))))
    return out


def _lattice_runs(case, seed):
    if case["kind"] in ("capillary", "slabs"):
        return [_capillary(case, seed)]
    return _droplets(case, seed) if case["kind"] == "droplets" else _ensemble(case, seed)


def _samples(rows, seed):
    """Sample parameters of the stable band (G_Aw, G_Bw, G_AB, tau_A, tau_B, H)
    and smooth targets of them with scatter, as a calibration gives."""
    r = _rng(seed, 4)
    X = np.stack([r.uniform(-0.5, 0.3, rows), r.uniform(-0.3, 0.6, rows), r.uniform(1.0, 1.08, rows),
                  r.uniform(1.0, 1.1, rows), r.uniform(1.0, 1.5, rows), r.uniform(16, 64, rows)], axis=1)
    c = np.cos(2.0 * X[:, 0] + 1.0) - X[:, 1]
    T = np.stack([c, 0.1 * X[:, 5] * c / X[:, 4], 0.1 + 0.05 * X[:, 0] * X[:, 2]], axis=1)
    return X, T + 0.01 * r.standard_normal(T.shape)


def _normalised(rows, seed):
    X, T = _samples(max(rows, 64), seed)
    X = (X - X.mean(0)) / X.std(0)
    T = (T - T.mean(0)) / T.std(0)
    return X[:rows].astype(np.float32), T[:rows].astype(np.float32)


def _net_params(seed):
    """Initial weights with biases that are not zero, as after some training."""
    p = M.init_params(int(seed) % (1 << 31))
    r = _rng(seed, 5)
    o = 0
    for a, b in ((6, 128), (128, 128), (128, 128), (128, 3)):
        o += a * b
        p[o:o + b] = 0.1 * r.standard_normal(b)
        o += b
    return p


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        X, T = _normalised(case["rows"], seed)
        net = M.Network(max_batch=max(4096, case["rows"]), params=_net_params(seed))
        return dict(case=case, net=net, x=torch.as_tensor(X, device="cuda"), t=torch.as_tensor(T, device="cuda"))
    if kind == "fit":
        X, T = _samples(case["samples"], seed)
        return dict(case=case, seed=int(seed) % (1 << 31), X=X, T=T,
                    sur=M.Surrogate(X, T, seed=int(seed) % (1 << 31)))
    if kind == "slabs":
        run = _capillary(case, seed)
        _, nA, nB = run["init"]
        return dict(case=case, slabs=[S.Slab(run, x0, x1, nA, nB, precision=case["precision"])
                                      for x0, x1 in S.slab_bounds(case["nx"], case["parts"])])
    runs = _lattice_runs(case, seed)
    kw = dict(precision=case["precision"])
    if kind == "capillary":
        if case["log_every"]:
            kw.update(log_every=case["log_every"], log_capacity=4096)
        if case["precision"] == "f16s":
            kw.update(rho_ref=W.fp16_shift(runs[0]))
        if case.get("autotune"):
            kw.update(autotune=True)
    if kind == "droplets":
        kw.update(tile=(128, 16))   # the calibration module's tiling
    lat = Lattice(runs, **kw)
    if case.get("autotune"):
        lat.step(TUNE_STEPS)
    return dict(case=case, lat=lat)


# ---- one pass ---------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "forward":
        return state["net"].forward(state["x"])
    if kind == "gradients":
        g, loss = state["net"].gradients(state["x"], state["t"])
        return dict(grad=g, loss=loss)
    if kind == "fit":
        losses = state["sur"].fit(state["X"], state["T"], steps=case["steps"], batch=case["batch"], seed=state["seed"])
        return dict(losses=losses, params=state["sur"].net.params)
    if kind == "slabs":
        S.step_local(state["slabs"], case["steps"])
        return [s.lat.get_columns(S.HALO, s.w) for s in state["slabs"]]
    lat = state["lat"]
    lat.step(case["steps"])
    if kind == "droplets" and case["precision"] == "f64":   # the judge reads angles on the host
        return [lat.densities(r) for r in range(case["runs"])]
    if kind != "capillary":   # the fields of the whole batch in one tensor
        return torch.cat([n.flatten() for r in range(case["runs"]) for n in lat.densities(r, device=True)])
    out = dict(populations=lat.get_columns(0, case["nx"]), densities=lat.densities(device=True))
    if case.get("velocity"):
        out["velocity"] = lat.velocity(device=True)
    if case["log_every"]:
        out["log"] = lat.log()
    elif case["precision"] != "f16s":
        out["interface"] = lat.interface()
    return out


# ---- the work a pass cannot do without ---------------------------------------

def work(case):
    """Bytes: the state read once and written once, the outputs written once
    (a pass of several steps need not move the state between them)."""
    kind = case["kind"]
    if kind == "forward":
        return {"bytes": case["rows"] * 9 * 4 + M.N_PARAMS * 4, "flops": 2 * MLP_MACS * case["rows"]}
    if kind == "gradients":
        return {"bytes": case["rows"] * 9 * 4 + M.N_PARAMS * 8, "flops": 6 * MLP_MACS * case["rows"]}
    if kind == "fit":
        b = min(case["batch"], case["samples"])
        return {"bytes": case["steps"] * b * 9 * 4 + M.N_PARAMS * 24, "flops": case["steps"] * 6 * MLP_MACS * b}
    if kind == "ensemble":
        nodes = sum(r["geom"]["nx"] * r["geom"]["ny"]
                    for r in W.batch_uneven_capillaries_stable(case["runs"], seed=case["sizes"]))
    else:
        nodes = case.get("runs", 1) * case["nx"] * case["ny"]
    state = 18 * ELEM[case["precision"]]
    outputs = 16
    if kind == "slabs":
        outputs = state
    elif kind == "capillary":
        outputs = 16 + state + (16 if case.get("velocity") else 0)
    return {"bytes": nodes * (2 * state + outputs), "flops": nodes * FLOPS_NODE * case["steps"]}


# ---- the same in 64 bits, by plain torch ---------------------------------------

_C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
_WT = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


class _Model:
    """The step of Eqs. 2-11 in 64 bits on [runs, ny, nx] arrays (runs of one size)."""

    def __init__(self, runs, device):
        g = runs[0]["geom"]
        self.geom, self.dev = g, device
        new = lambda v: torch.tensor(v, dtype=torch.float64, device=device).view(-1, 1, 1)   # noqa: E731
        p = [r["params"] for r in runs]
        self.G = new([q["G"] for q in p])
        self.Gw = [new([q.get("G_Aw", 0.0) for q in p]), new([q.get("G_Bw", 0.0) for q in p])]
        self.tau = [new([q["tau_A"] for q in p]), new([q["tau_B"] for q in p])]
        self.alpha = p[0].get("alpha", (4 / 9, 4 / 9))
        self.m = p[0].get("mass", (1.0, 1.0))
        self.thr = p[0].get("rho_bulk", 2.0) / 3.0
        solid = torch.as_tensor(W.solid_mask(g).astype(bool), device=device)[None]
        self.solid, self.fluid = solid, ~solid
        # solid flag of the node at x + c_i, and the wall sum of Eq. 11
        self.sol = [self._at(solid, i) for i in range(9)]
        self.wall = [sum(_WT[i] * _C[i][d] * self.sol[i].double() for i in range(1, 9)) for d in (0, 1)]
        nA, nB = zip(*[W.initial_fields(r) for r in runs])
        self.F = []
        for k, n in enumerate((nA, nB)):
            n = torch.as_tensor(np.stack(n), dtype=torch.float64, device=device)
            n = torch.where(self.fluid, n, torch.zeros_like(n))
            self.F.append(torch.stack([self._aw(k, i) * n for i in range(9)]))
        self.u = [torch.zeros_like(self.F[0][0]) for _ in range(2)]

    def _aw(self, k, i):
        a = self.alpha[k]
        return a if i == 0 else ((1 - a) / 5 if i <= 4 else (1 - a) / 20)

    @staticmethod
    def _at(a, i):   # a(x + c_i)
        return torch.roll(a, (-_C[i][1], -_C[i][0]), (-2, -1))

    def step(self, velocity=False):
        f, n, j, a = [], [], [], []
        for k in range(2):
            F = self.F[k]
            f.append([F[0]] + [torch.where(self.sol[_OPP[i]], F[_OPP[i]], self._at(F[i], _OPP[i]))
                               for i in range(1, 9)])
            z = torch.zeros_like(F[0])
            n.append(torch.where(self.fluid, sum(f[k]), z))
            j.append([sum(_C[i][d] * f[k][i] for i in range(9) if _C[i][d]) for d in (0, 1)])
        for k in range(2):
            other = n[1 - k]
            s = [sum(_WT[i] * _C[i][d] * self._at(other, i) for i in range(1, 9) if _C[i][d]) for d in (0, 1)]
            a.append([-self.G * s[d] - self.Gw[k] * self.wall[d] for d in (0, 1)])
        one = torch.ones_like(n[0])
        if velocity:
            rho = torch.where(self.fluid, self.m[0] * n[0] + self.m[1] * n[1], one)
            self.u = [torch.where(self.fluid, sum(self.m[k] * j[k][d] + 0.5 * n[k] * a[k][d] for k in range(2)) / rho,
                                  torch.zeros_like(rho)) for d in (0, 1)]
        den = torch.where(self.fluid, sum(self.m[k] * n[k] / self.tau[k] for k in range(2)), one)
        U = [sum(self.m[k] * j[k][d] / self.tau[k] for k in range(2)) / den for d in (0, 1)]
        for k in range(2):
            ux, uy = (U[d] + self.tau[k] / self.m[k] * a[k][d] for d in (0, 1))
            usq = 1.5 * (ux * ux + uy * uy)
            out = []
            for i in range(9):
                cu = _C[i][0] * ux + _C[i][1] * uy
                feq = n[k] * (_WT[i] * (3 * cu + 4.5 * cu * cu - usq) + self._aw(k, i))
                new = f[k][i] - (f[k][i] - feq) / self.tau[k]
                out.append(torch.where(self.fluid, new, torch.zeros_like(new)))
            self.F[k] = torch.stack(out)

    def densities(self):
        return [F.sum(0) for F in self.F]

    def _front(self, v, ok, cap):
        """Crossing of v between the last passing and the first failing column."""
        bad = np.nonzero(~ok)[0]
        if len(bad) == 0:
            return float(cap)
        x = int(bad[0])
        return 0.0 if x == 0 else x - 1 + v[x - 1] / (v[x - 1] - v[x])

    def fronts(self):
        g = self.geom
        nA, nB = (n[0, :, g["cap_x0"]:g["cap_x1"]].cpu().numpy() for n in self.densities())
        cap, H = g["cap_x1"] - g["cap_x0"], g["y_top"] - g["y_bot"] - 1
        rows = [g["y_bot"] + H // 2, g["y_bot"] + H // 2 + 1] if H % 2 == 0 else [g["y_bot"] + (H + 1) // 2]
        phi = [(nA[y] - nB[y]) / (nA[y] + nB[y]) for y in rows]
        z = [np.mean([self._front(p, p >= 0, cap) for p in phi])]
        for y in (g["y_bot"] + 1, g["y_top"] - 1):
            v = nA[y] - self.thr
            z.append(self._front(v, v >= 0, cap))
        return np.array(z)

    def record(self, t):
        return np.concatenate([[t], self.fronts(), [float(n.sum()) for n in self.densities()]])


def _exact_lattice(case, seed, device):
    runs = _lattice_runs(case, seed)
    kind = case["kind"]
    t0 = TUNE_STEPS if case.get("autotune") else 0
    total = t0 + case["steps"]
    if kind == "ensemble":
        out = []
        for r in runs:
            m = _Model([r], device)
            for _ in range(total):
                m.step()
            out += [n.flatten() for n in m.densities()]
        return torch.cat(out)
    m = _Model(runs, device)
    every = case.get("log_every", 0)
    log = [m.record(0)] if every else None
    for t in range(1, total + 1):
        m.step(velocity=bool(case.get("velocity")) and t == total)
        if every and t % every == 0:
            log.append(m.record(t))
    dens = m.densities()
    if kind == "droplets":
        if case["precision"] != "f64":
            return torch.stack(dens, dim=1).flatten()
        return [tuple(d[r].cpu().numpy() for d in dens) for r in range(case["runs"])]
    pops = torch.stack([F[:, 0] for F in m.F])
    if kind == "slabs":
        return [pops[..., x0:x1].contiguous() for x0, x1 in S.slab_bounds(case["nx"], case["parts"])]
    if case["precision"] == "f16s":   # stored as f - w_i rho_ref on fluid nodes
        ref = torch.tensor(W.fp16_shift(runs[0]), dtype=torch.float64, device=device).view(2, 1, 1, 1)
        wt = torch.tensor(_WT, dtype=torch.float64, device=device).view(1, 9, 1, 1)
        pops = torch.where(m.fluid[None], pops - wt * ref, torch.zeros_like(pops))
    out = dict(populations=pops, densities=tuple(d[0] for d in dens))
    if case.get("velocity"):
        out["velocity"] = tuple(u[0] for u in m.u)
    if every:
        out["log"] = np.stack(log)
    elif case["precision"] != "f16s":
        out["interface"] = m.fronts()
    return out


def _unpack(p):
    o, out = 0, []
    for a, b in ((6, 128), (128, 128), (128, 128), (128, 3)):
        out += [p[o:o + a * b].reshape(a, b), p[o + a * b:o + a * b + b]]
        o += a * b + b
    return out


def _mlp64(theta, x):
    w = _unpack(theta)
    for i in range(4):
        x = x @ w[2 * i] + w[2 * i + 1]
        if i < 3:
            x = 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))
    return x


def _grad64(theta, x, t):
    theta = theta.detach().requires_grad_(True)
    loss = ((_mlp64(theta, x) - t) ** 2).mean()
    return torch.autograd.grad(loss, theta)[0], loss.detach()


def _exact_fit(case, seed, device):
    seed = int(seed) % (1 << 31)
    X, T = _samples(case["samples"], seed)
    norm = lambda a: (a - a.mean(0)) / np.where(a.std(0) > 0, a.std(0), 1.0)   # noqa: E731
    x = torch.as_tensor(norm(X).astype(np.float32), device=device).double()
    t = torch.as_tensor(norm(T).astype(np.float32), device=device).double()
    theta = torch.as_tensor(M.init_params(seed), device=device).double()
    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    rng = np.random.Generator(np.random.PCG64(seed))
    losses = []
    for s in range(1, case["steps"] + 1):
        idx = torch.as_tensor(rng.choice(len(X), size=min(case["batch"], len(X)), replace=False), device=device)
        g, loss = _grad64(theta, x[idx], t[idx])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        theta = theta - 2e-3 * (m / (1 - 0.9 ** s)) / (torch.sqrt(v / (1 - 0.999 ** s)) + 1e-8)
        losses.append(float(loss))
    return dict(losses=np.array(losses), params=theta.cpu().numpy())


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        X, T = _normalised(case["rows"], seed)
        theta = torch.as_tensor(_net_params(seed), device=device).double()
        x, t = (torch.as_tensor(a, device=device).double() for a in (X, T))
        if kind == "forward":
            return _mlp64(theta, x)
        g, loss = _grad64(theta, x, t)
        return dict(grad=g, loss=loss.reshape(1))
    if kind == "fit":
        return _exact_fit(case, seed, device)
    return _exact_lattice(case, seed, device)
