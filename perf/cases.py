"""The work whose speed counts: what a user of the solver has it do, through its public entry points.

A case is a dict of plain values; `kind` names the call:

  evolve   Solver.evolve         a trajectory of `steps` RK4 steps
  steady   Solver.steady_state   a whole solve to ||f(rho)||_F < tol
  rkf45    Solver.rkf45          the same by adaptive RKF45
  batch    batch_steady_state    many graphs of uneven size in one call
  predict  Gnn.predict           the populations a warm start begins from
  train    Gnn.train             the warm-start network's training
  rank     populations, pagerank, hub_classes of one graph

The graphs are the two seeded generators of graphs.py: `heavy` (preferential
attachment, lognormal weights, the stand-in for the airline network) and `er`
(Erdos-Renyi with link probability p, unit weights: most nodes linked, so the
solver takes its dense forms). Another seed is another graph, another state.
"""
import math
import types

import numpy as np
import torch

from paper_2003_04930_gb300 import Solver, graphs
from paper_2003_04930_gb300.qpr import QPR_FP64, QPR_MIXED, Gnn, batch_steady_state
from paper_2003_04930_gb300.warmstart import TRAINED_PARAMS

ALPHA, DT = 0.85, 0.01
PRECISION = {"fp64": QPR_FP64, "mixed": QPR_MIXED}


def listed():
    return [
        # The plain method's small check: 16 nodes to t = 50. Nothing but latency.
        dict(name="evolve_fp64_er_n16", kind="evolve", graph="er", p=0.25, precision="fp64", n=16, omega=0.8, steps=5000),
        # The default precision on the airline-sized graph: exact FP64, sparse H.
        dict(name="evolve_fp64_n922", kind="evolve", graph="heavy", precision="fp64", n=922, omega=0.5, steps=160),
        # The default precision where most nodes are linked: dense H, a size off every tile.
        dict(name="evolve_fp64_dense_n500", kind="evolve", graph="er", p=0.25, precision="fp64", n=500, omega=0.8, steps=40),
        # The headline: the airline-sized graph to its steady state from I/N, mixed precision.
        dict(name="steady_mixed_n922", kind="steady", graph="heavy", precision="mixed", n=922, omega=0.8, tol=1e-8),
        # A graph above what one CTA can stage, odd-sized, to its steady state.
        dict(name="steady_mixed_n1999", kind="steady", graph="heavy", precision="mixed", n=1999, omega=0.8, tol=1e-8),
        # The metric's second size, where every stage streams from HBM.
        dict(name="steady_mixed_n4096", kind="steady", graph="heavy", precision="mixed", n=4096, omega=0.8, tol=1e-6),
        # Mixed precision where most nodes are linked: the tensor-core form.
        dict(name="steady_mixed_dense_n900", kind="steady", graph="er", p=0.25, precision="mixed", n=900, omega=0.8, tol=1e-8),
        # The paper's own integrator on the airline-sized graph.
        dict(name="rkf45_mixed_n922", kind="rkf45", graph="heavy", n=922, omega=0.8, tol=1e-8),
        # Labels for the warm-start network: uneven graphs, each its own omega, to 1e-6.
        dict(name="batch_mixed_12", kind="batch", count=12, n_lo=32, n_hi=512, omega_lo=0.4, omega_hi=0.95, tol=1e-6),
        # A warm start's inference on the airline-sized graph.
        dict(name="predict_n922", kind="predict", n=922, omega=0.8),
        # The warm-start network's training: uneven graphs, mini-batches of 8.
        dict(name="train_16", kind="train", count=16, n_lo=64, n_hi=1024, epochs=4),
        # What is read off a solved state: populations and ranks, the classical PageRank, the hubs.
        dict(name="rank_n922", kind="rank", n=922),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "sparse64", "dense64", "steady", "large", "dense", "rkf45", "batch", "predict", "train", "rank"])
    omega = round(rng.uniform(0.5, 1.0), 3)
    if kind == "small":
        return dict(kind="evolve", graph="er", p=round(rng.uniform(0.2, 0.5), 2), precision="fp64", n=_log(rng, 5, 64),
                    omega=omega, steps=_log(rng, 500, 5000))
    if kind == "sparse64":
        return dict(kind="evolve", graph="heavy", precision="fp64", n=_log(rng, 100, 1500), omega=omega, steps=_log(rng, 20, 160))
    if kind == "dense64":
        return dict(kind="evolve", graph="er", p=round(rng.uniform(0.2, 0.5), 2), precision="fp64", n=_log(rng, 65, 700),
                    omega=omega, steps=_log(rng, 10, 40))
    if kind == "steady":
        return dict(kind="steady", graph="heavy", precision="mixed", n=_log(rng, 48, 1900), omega=omega,
                    tol=rng.choice([1e-6, 1e-8]))
    if kind == "large":
        return dict(kind="steady", graph="heavy", precision="mixed", n=_log(rng, 1500, 3500),
                    omega=round(rng.uniform(0.7, 0.95), 3), tol=1e-6)
    if kind == "dense":
        return dict(kind="steady", graph="er", p=round(rng.uniform(0.2, 0.35), 2), precision="mixed", n=_log(rng, 130, 900),
                    omega=round(rng.uniform(0.75, 1.0), 3), tol=rng.choice([1e-6, 1e-8]))
    if kind == "rkf45":
        return dict(kind="rkf45", graph="heavy", n=_log(rng, 300, 1500), omega=round(rng.uniform(0.7, 0.95), 3), tol=1e-8)
    if kind == "batch":
        hi = _log(rng, 64, 512)
        return dict(kind="batch", count=rng.randint(3, 12), n_lo=min(32, hi // 2), n_hi=hi, omega_lo=0.4, omega_hi=0.95, tol=1e-6)
    if kind == "predict":
        return dict(kind="predict", n=_log(rng, 32, 4096), omega=omega)
    if kind == "train":
        hi = _log(rng, 128, 1024)
        return dict(kind="train", count=rng.randint(4, 16), n_lo=64, n_hi=hi, epochs=rng.randint(1, 4))
    return dict(kind="rank", n=_log(rng, 32, 4096))


# ---- inputs ----

def _graph(case, seed, n=None):
    n = n or case["n"]
    if case.get("graph") == "er":
        return graphs.erdos_renyi(n, case["p"], seed)
    return graphs.heavy_tailed(n, seed)


def _uneven(case, seed):
    """`count` graphs, their sizes and omegas spread evenly over their ranges so that another seed is as much work."""
    rng = np.random.default_rng(seed)
    count = case["count"]
    ns = [int(case["n_lo"] + (case["n_hi"] - case["n_lo"]) * (k + 0.5) / count) for k in range(count)]
    lo, hi = case.get("omega_lo", 0.1), case.get("omega_hi", 0.95)
    omegas = [float(lo + (hi - lo) * ((k * 7) % count + rng.uniform(0.3, 0.7)) / count) for k in range(count)]
    return [(graphs.heavy_tailed(n, seed + 1000 + k), omegas[k]) for k, n in enumerate(ns)], rng


def _populations(n, rng):
    p = rng.lognormal(0.0, 1.0, n)
    return p / p.sum()


def _state(case, seed, n):
    """rho0: I/N for a solve; a random mixed state, well inside the cone, for a trajectory."""
    if case["kind"] != "evolve":
        return torch.eye(n, dtype=torch.complex128, device="cuda") / n
    gen = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn(n, 8, dtype=torch.complex128, device="cuda", generator=gen)
    a = w @ w.mH
    return 0.5 * a / a.diagonal().real.sum() + 0.5 * torch.eye(n, dtype=torch.complex128, device="cuda") / n


def _largest_step(case, g):
    """The step a caller takes to be stable: the edge of the integrators' stability region on a bound of H's spectrum."""
    h, v, norm = _dense_h(g), torch.ones(g.n, dtype=torch.float64, device=_where(g.n)), 0.0
    for _ in range(100):
        v = h @ (v / v.norm())
        norm = v.norm()
    return 2.4 / ((1.0 - case["omega"]) * 2.1 * float(norm) + 2.0 * case["omega"])


def _solved(n, seed):
    """A state as a solve leaves it: uneven populations, small coherences."""
    rho = torch.diag(torch.from_numpy(_populations(n, np.random.default_rng(seed)))).to("cuda", torch.complex128)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(n, n, dtype=torch.complex128, device="cuda", generator=gen) * (0.01 / n)
    return rho + (a - torch.diag(a.diagonal())) / 2 + (a - torch.diag(a.diagonal())).mH / 2


def prepare(case, seed):
    kind = case["kind"]
    s = types.SimpleNamespace(case=case)
    if kind in ("batch", "train"):
        s.problems, rng = _uneven(case, seed)
        if kind == "train":
            s.net, s.theta = Gnn(seed=0), np.load(TRAINED_PARAMS).astype(np.float32)
            s.problems = [(g, om, _populations(g.n, rng)) for g, om in s.problems]
        return s
    g = _graph(case, seed)
    if kind == "predict":
        s.net, s.g = Gnn(seed=0), g
        s.net.set_params(np.load(TRAINED_PARAMS).astype(np.float32))
    elif kind == "rank":
        s.solver, s.rho = Solver.from_edges(g, alpha=ALPHA, omega=0.8), _solved(case["n"], seed)
    else:
        s.solver = Solver.from_edges(g, alpha=ALPHA, omega=case["omega"], precision=PRECISION[case.get("precision", "mixed")])
        s.rho0 = _state(case, seed, g.n)
        s.largest = _largest_step(case, g)
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "evolve":
        return s.solver.evolve(s.rho0.clone(), min(DT, s.largest), case["steps"])
    if kind == "steady":
        rho = s.rho0.clone()
        stats = s.solver.steady_state(rho, min(DT, s.largest), case["tol"], 400000)
        return {"rho": rho, "steps": stats["steps"]}
    if kind == "rkf45":
        rho = s.rho0.clone()
        stats = s.solver.rkf45(rho, tol=case["tol"], max_steps=400000, step_tol=1e-6, h_max=s.largest, order=5)
        return {"rho": rho, "steps": stats["accepted"]}
    if kind == "batch":
        rhos = [torch.eye(g.n, dtype=torch.complex128, device="cuda") / g.n for g, _ in s.problems]
        _, stats = batch_steady_state([(g, om, r) for (g, om), r in zip(s.problems, rhos)], alpha=ALPHA, dt=DT, tol=case["tol"])
        return {"rho": rhos, "steps": [d["steps"] for d in stats]}
    if kind == "predict":
        return s.net.predict(s.g, case["omega"], ALPHA)
    if kind == "train":
        s.net.set_params(s.theta)
        losses = s.net.train(s.problems, epochs=case["epochs"], batch=8, lr=1e-3, seed=1, alpha=ALPHA)
        return {"losses": losses, "params": s.net.get_params()}
    p, rank = s.solver.populations(s.rho, with_rank=True)
    pi = s.solver.pagerank()
    classes, counts = s.solver.hub_classes(p)
    return {"p": p, "rank": rank, "pi": pi, "classes": classes, "counts": counts}


# ---- what a pass cannot do without ----

def work(case):
    kind = case["kind"]

    def stage(n, graph, p=0.25):
        """Flops of one f(rho): the real product H [Re | Im] over the nonzeros, and about 20 operations an element."""
        nnz = n * n * (1 - (1 - p) ** 2) if graph == "er" else 16.0 * n
        return 4.0 * nnz * n + 20.0 * n * n

    def solve(n, tol):
        """The typical step count of a solve from I/N at dt = 0.01 (2226 at N = 922, omega = 0.8, 1e-8)."""
        return 2300.0 if tol < 1e-7 else 1700.0

    def rho_bytes(n):
        return 2 * 16.0 * n * n  # read and written once

    if kind in ("evolve", "steady", "rkf45"):
        n = case["n"]
        stages = 4 * case["steps"] if kind == "evolve" else 4 * solve(n, case["tol"]) if kind == "steady" else 6 * 360
        return {"bytes": rho_bytes(n), "flops": stages * stage(n, case.get("graph"), case.get("p", 0.25))}
    if kind in ("batch", "train"):
        ns = [case["n_lo"] + (case["n_hi"] - case["n_lo"]) * (k + 0.5) / case["count"] for k in range(case["count"])]
        if kind == "batch":
            return {"bytes": sum(rho_bytes(n) for n in ns), "flops": sum(4 * solve(n, case["tol"]) * stage(n, "heavy") for n in ns)}
        passes = 3.0 * case["epochs"]  # a backward pass is twice the forward's products
        return {"bytes": sum(24.0 * 8 * n + 8.0 * n for n in ns) + 2 * 4.0 * 25921, "flops": passes * sum(_forward_flops(n) for n in ns)}
    n = case["n"]
    if kind == "predict":
        return {"bytes": 24.0 * 8 * n + 8.0 * n + 4.0 * 25921, "flops": _forward_flops(n)}
    return {"bytes": 32.0 * n + 16.0 * 8 * n, "flops": 64 * 2 * 8.0 * n}  # the diagonal, the links; about 64 power iterations


def _forward_flops(n):
    return n * (2.0 * 2 * 64 * (8 + 3 * 64) + 2.0 * 16 * (8 + 3 * 64))


# ---- the same in 64 bits, in plain torch ----

def _adjacency(g):
    """A_ij = w for the link j -> i (duplicates sum; no self-loops)."""
    a = torch.zeros(g.n, g.n, dtype=torch.float64)
    keep = g.src != g.dst
    a.index_put_((torch.from_numpy(g.dst[keep]), torch.from_numpy(g.src[keep])), torch.from_numpy(g.w[keep]), accumulate=True)
    return a.to(_where(g.n))


def _where(n):
    """Small problems on the host: there a launch costs more than the arithmetic."""
    return "cpu" if n <= 64 else "cuda"


def _dense_h(g):
    a = _adjacency(g)
    return -torch.maximum(a, a.T)


def _google(g):
    """G = alpha S + (1 - alpha) F, dangling columns as F's."""
    a, n = _adjacency(g), g.n
    f = (1.0 - torch.eye(n, dtype=torch.float64, device=a.device)) / (n - 1)
    out = a.sum(0)
    s = torch.where(out > 0, a / torch.where(out > 0, out, 1.0), f)
    return ALPHA * s + (1 - ALPHA) * f


class _Rhs:
    """f(rho) of Eq. 1 on rho as [Re | Im], n x 2n."""

    def __init__(self, g, omega):
        self.n, self.omega = g.n, omega
        h = _dense_h(g)
        self.h = h.to_sparse_csr() if int((h != 0).sum()) * 16 < g.n * g.n else h
        self.g = _google(g)

    def __call__(self, y):
        n, om = self.n, self.omega
        x = self.h @ y
        a, b = x[:, :n], x[:, n:]
        f = torch.cat([(1 - om) * (b + b.T), (om - 1) * (a - a.T)], 1) - om * y
        f.diagonal().add_(om * (self.g @ y.diagonal()))
        return f


def _rk4(f, y, dt):
    """y after one step, and ||f(y)||_F."""
    k1 = f(y)
    k2 = f(y + (dt / 2) * k1)
    k3 = f(y + (dt / 2) * k2)
    k4 = f(y + dt * k3)
    return y + (dt / 6) * (k1 + 2 * k2 + 2 * k3 + k4), k1.norm()


def _unit(y):
    return y / y.diagonal().sum()


def _steady(g, omega, tol):
    """The first state of the RK4 trajectory from I/N with ||f||_F < tol, and its step."""
    f = _Rhs(g, omega)
    y = torch.eye(g.n, 2 * g.n, dtype=torch.float64, device=_where(g.n)) / g.n
    dt = min(DT, _largest_step({"omega": omega}, g))
    done, block = 0, 64
    while done < 400000:
        start, norms = y, []
        for _ in range(block):
            y, r = _rk4(f, y, dt)
            norms.append(r)
        # (the trace stays 1 to rounding within a block)
        below = (torch.stack(norms) < tol).nonzero()
        if len(below):
            y = start
            for _ in range(int(below[0])):
                y, _ = _rk4(f, y, dt)
            return _unit(y), done + int(below[0])
        done += block
        y = _unit(y)
    return None, None


def _rkf45(g, omega, tol, h_max, step_tol=1e-6):
    """Adaptive RKF45, fifth order kept: one step of the linear f is a polynomial in h L."""
    f = _Rhs(g, omega)
    y = torch.eye(g.n, 2 * g.n, dtype=torch.float64, device=_where(g.n)) / g.n
    h, steps = min(DT, h_max), 0
    for _ in range(20000):
        u = f(y)
        if float(u.norm()) < tol:
            return y, steps
        z, fac = y, (1.0, 1 / 2, 1 / 6, 1 / 24, 1 / 120, 1 / 2080)
        us = []
        for k in range(6):
            u = h * (u if k == 0 else f(us[-1]))
            us.append(u)
            z = z + fac[k] * u
        d = us[5] / 2080 - us[4] / 780
        err = float(torch.hypot(d[:, :g.n], d[:, g.n:]).max())
        if err <= step_tol * h:
            y, steps = _unit(z), steps + 1
        h = min(h_max, h * min(4.0, max(0.1, (step_tol * h / (2 * err)) ** 0.25 if err > 0 else 4.0)))
    return None, None


def _complex(y):
    n = y.shape[0]
    return torch.complex(y[:, :n].contiguous(), y[:, n:].contiguous())


class _Net:
    """The warm-start network, its matrices rounded to BF16 as they are used, everything else in 64 bits."""

    SIZES = [8, 64, 64, 64]

    @staticmethod
    def graph(g, omega):
        a, gm, n = _adjacency(g), _google(g), g.n
        pi = torch.full((n,), 1.0 / n, dtype=torch.float64, device=a.device)
        for _ in range(200):
            pi = gm @ pi
            pi = pi / pi.sum()
        one = torch.ones(n, dtype=torch.float64, device=a.device)
        out = a.sum(0)
        x = torch.stack([one, omega * one, torch.log1p(a.sum(1)), torch.log1p(out), torch.log1p((a > 0).sum(1).double()),
                         torch.log1p((a > 0).sum(0).double()), torch.log(n * pi), (out == 0).double()], 1)
        b = a + a.T
        s = b.sum(1, keepdim=True)
        return x, torch.where(s > 0, b / torch.where(s > 0, s, 1.0), 0.0)

    @classmethod
    def logp(cls, theta, x, pm):
        at, h = 0, x
        for d in cls.SIZES:
            ws, wn, b = theta[at:at + d * 64].view(d, 64), theta[at + d * 64:at + 2 * d * 64].view(d, 64), theta[at + 2 * d * 64:at + 2 * d * 64 + 64]
            h = torch.relu(h @ _bf16(ws) + (pm @ h) @ _bf16(wn) + b)
            at += 2 * d * 64 + 64
        return torch.log_softmax(h @ theta[at:at + 64] + theta[at + 64], 0)


def _bf16(w):
    """BF16 rounding whose gradient is that of the rounded matrix."""
    return w + (w.detach().float().bfloat16().double() - w.detach())


def _splitmix(s):
    m = (1 << 64) - 1
    s = (s + 0x9E3779B97F4A7C15) & m
    z = ((s ^ (s >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return s, z ^ (z >> 31)


def _train(samples, theta0, epochs, batch, lr, rs):
    theta = torch.from_numpy(theta0).double().cuda()
    m, v, t = torch.zeros_like(theta), torch.zeros_like(theta), 0
    data = [(*(t.cuda() for t in _Net.graph(g, om)), torch.from_numpy(p).cuda()) for g, om, p in samples]
    order, losses = list(range(len(data))), []
    for _ in range(epochs):
        for i in range(len(order) - 1, 0, -1):
            rs, r = _splitmix(rs)
            order[i], order[r % (i + 1)] = order[r % (i + 1)], order[i]
        total = 0.0
        for b0 in range(0, len(order), batch):
            part = order[b0:b0 + batch]
            w = theta.clone().requires_grad_(True)
            loss = sum(-(p * _Net.logp(w, x, pm)).sum() for x, pm, p in (data[i] for i in part))
            g, = torch.autograd.grad(loss, w)
            total, g, t = total + float(loss), g / len(part), t + 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            theta = theta - lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        losses.append(total / len(order))
    return np.array(losses), theta


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "train"):
        problems, rng = _uneven(case, seed)
        if kind == "batch":
            if sum(g.n for g, _ in problems) > 5000:
                return None
            got = [_steady(g, om, case["tol"]) for g, om in problems]
            return {"rho": [None if y is None else _complex(y) for y, _ in got], "steps": [k for _, k in got]}
        losses, theta = _train([(g, om, _populations(g.n, rng)) for g, om in problems], np.load(TRAINED_PARAMS).astype(np.float32),
                               case["epochs"], 8, 1e-3, 1)
        return {"losses": losses, "params": theta}
    g = _graph(case, seed)
    if kind == "predict":
        x, pm = _Net.graph(g, case["omega"])
        return _Net.logp(torch.from_numpy(np.load(TRAINED_PARAMS).astype(np.float32)).double().to(x.device), x, pm).exp()
    if kind == "rank":
        rho = _solved(case["n"], seed)
        gm = _google(g)
        pi = torch.full((g.n,), 1.0 / g.n, dtype=torch.float64, device=gm.device)
        for _ in range(400):
            pi = gm @ pi
            pi = pi / pi.sum()
        return {"p": rho.diagonal().real.contiguous(), "rank": None, "pi": pi, "classes": None, "counts": None}
    if kind == "steady":
        if g.n > 2000:
            return None
        y, k = _steady(g, case["omega"], case["tol"])
        return None if y is None else {"rho": _complex(y), "steps": k}
    if kind == "rkf45":
        y, k = _rkf45(g, case["omega"], case["tol"], _largest_step(case, g))
        return None if y is None else {"rho": _complex(y), "steps": k}
    f = _Rhs(g, case["omega"])
    rho = _state(case, seed, g.n).to(_where(g.n))
    y = torch.cat([rho.real, rho.imag], 1)
    y = _unit(torch.cat([(y[:, :g.n] + y[:, :g.n].T) / 2, (y[:, g.n:] - y[:, g.n:].T) / 2], 1))
    dt = min(DT, _largest_step(case, g))
    for _ in range(case["steps"]):
        y, _ = _rk4(f, y, dt)
        y = _unit(y)
    return _complex(y)
