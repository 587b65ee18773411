"""Performance cases of the solver: what programs have it do, through its public entry points.

Each case is a dict of plain values:

  what        "project" (the capped-simplex projection on device arrays), "solve" (one network),
              "batch" (many uneven networks together) or "serve" (tickets of the scheduler)
  n, m | deg  nodes and, for a projection, columns, else out-degree (ring graphs) or the number
              of nearest neighbours (kNN graphs)
  iters       PDHG iterations of one pass (a fixed number, so that a pass is the same work
              whatever the rounding of the stop test)
  before      iterations that the program has run on the network already; 0: a cold solve
              each pass, else each pass changes the capacities by +-10 % and re-solves warm
  utility     "log", "pow" (one exponent) or "powij" (an exponent for each pair)

Networks are the repository's own recipes (ring plus random chords, the paper's kNN graphs),
drawn here from the seed. FP32 and BF16 iterates come back from the library widened to
doubles; a program that goes on in single precision (or holds flows in BF16) takes them in the
type that they were computed in, and so does ``run``.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2501_17996_gb300 import binding

RHO = 1.9
K_ADAPT = 100


# ------------------------------------------------------------------------------ the cases

def listed():
    return [
        # the operator inside a caller's own iteration: small, queued on a stream, no
        # allocation, no wait; ragged columns (n not a multiple of the row stride)
        {"name": "project-small", "what": "project", "n": 103, "m": 1024, "entry": "noalloc"},
        # the operator at the paper's largest column length, with the distance read back
        {"name": "project-large", "what": "project", "n": 10000, "m": 30000, "entry": "alloc"},
        # the smallest network: launches and waits are all there is
        {"name": "solve-tiny", "what": "solve", "graph": "ring", "n": 10, "deg": 4, "utility": "log",
         "precision": "fp32", "iters": 100, "before": 0, "out": "TFY"},
        # the paper's smallest size (n = 100, m = 1000), all outputs
        {"name": "solve-mid", "what": "solve", "graph": "ring", "n": 100, "deg": 10, "utility": "log",
         "precision": "fp32", "iters": 200, "before": 0, "out": "TFY"},
        # FP64 iterates with an exponent for each pair: the reference runs of small networks
        {"name": "solve-fp64", "what": "solve", "graph": "ring", "n": 203, "deg": 9, "utility": "powij",
         "precision": "fp64", "iters": 100, "before": 0, "out": "TFY"},
        # the paper's kNN family at n = 1000 (renumbered nodes, local gathers)
        {"name": "solve-knn", "what": "solve", "graph": "knn", "n": 1000, "deg": 10, "utility": "log",
         "precision": "fp32", "iters": 200, "before": 0, "out": "T"},
        # a resident network whose capacities change and which is solved again warm
        {"name": "resolve-1000", "what": "solve", "graph": "ring", "n": 1000, "deg": 8, "utility": "log",
         "precision": "fp32", "iters": 100, "before": 400, "out": "TY"},
        # BF16-stored flows, power utility
        {"name": "solve-bf16", "what": "solve", "graph": "ring", "n": 3001, "deg": 10, "utility": "pow",
         "precision": "bf16", "iters": 100, "before": 0, "out": "T"},
        # the largest served network, cold
        {"name": "solve-3000", "what": "solve", "graph": "ring", "n": 3000, "deg": 8, "utility": "log",
         "precision": "fp32", "iters": 100, "before": 0, "out": "T"},
        # n = 10^4, m = 10^5, far into a solve, where nearly all of its iterations are
        {"name": "resolve-large", "what": "solve", "graph": "ring", "n": 10000, "deg": 10, "utility": "pow",
         "precision": "fp32", "iters": 200, "before": 400, "out": "T"},
        # 64 uneven networks solved together
        {"name": "batch-64", "what": "batch", "count": 64, "n": 50, "n_hi": 400, "iters": 100},
        # tickets: twelve resident networks of several sizes, re-solved warm
        {"name": "serve-12", "what": "serve", "count": 12, "n": 100, "n_hi": 1000, "iters": 50,
         "before": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above."""
    what = rng.choice(["project", "solve", "solve", "solve", "solve", "batch", "serve"])
    if what == "project":
        n = _log_int(rng, 8, 20000)
        return {"what": what, "n": n, "m": _log_int(rng, 64, min(200000, 300_000_000 // n)),
                "entry": rng.choice(["noalloc", "alloc"])}
    if what == "batch":
        lo = _log_int(rng, 10, 200)
        return {"what": what, "count": rng.randint(2, 64), "n": lo, "n_hi": lo + rng.randint(1, 300),
                "iters": rng.choice([50, 100])}
    if what == "serve":
        lo = _log_int(rng, 40, 400)
        return {"what": what, "count": rng.randint(1, 16), "n": lo, "n_hi": lo + rng.randint(1, 800),
                "iters": rng.choice([20, 50]), "before": rng.choice([50, 100])}
    precision = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp64"])
    graph = rng.choice(["ring", "ring", "knn"])
    n = _log_int(rng, 12, {"fp32": 5000, "bf16": 5000, "fp64": 1200}[precision])
    deg = rng.randint(3, min(16, n - 2))
    return {"what": what, "graph": graph, "n": n, "deg": deg, "precision": precision,
            "utility": rng.choice(["log", "pow", "powij"]), "iters": rng.choice([50, 100, 150]),
            "before": rng.choice([0, 0, 200]), "out": "TFY" if graph == "ring" and n <= 1000 else rng.choice(["T", "TY"])}


# ------------------------------------------------------------------------------ the inputs

def _ring(n, deg, rng):
    """Directed ring plus deg - 1 distinct random out-edges of each node."""
    off = np.ones((n, deg), dtype=np.int64)
    for j in range(1, deg):   # distinct offsets, drawn again where they collide
        new = rng.integers(2, n, size=n)
        while True:
            again = (off[:, :j] == new[:, None]).any(axis=1)
            if not again.any():
                break
            new[again] = rng.integers(2, n, size=int(again.sum()))
        off[:, j] = new
    tail = np.repeat(np.arange(n), deg)
    head = (tail + off.ravel()) % n
    return tail.astype(np.int32), head.astype(np.int32)


def _knn(n, q, rng):
    """Bidirectional edges between q-nearest neighbours of uniform points in the unit square,
    joined by a ring of the points sorted along a line so that the network is connected."""
    x = rng.uniform(size=(n, 2))
    g = torch.as_tensor(x, device="cuda")
    nbr = torch.cdist(g, g).topk(min(q + 1, n), largest=False).indices[:, 1:].cpu().numpy()
    i = np.repeat(np.arange(n), nbr.shape[1])
    order = np.argsort(np.floor(x[:, 1] * math.sqrt(n)) * 2.0 +
                       np.where(np.floor(x[:, 1] * math.sqrt(n)) % 2 == 0, x[:, 0], 1.0 - x[:, 0]))
    a = np.concatenate([i, nbr.ravel(), order, np.roll(order, -1)])
    b = np.concatenate([nbr.ravel(), i, np.roll(order, -1), order])
    key = np.unique(a[a != b] * n + b[a != b])
    return (key // n).astype(np.int32), (key % n).astype(np.int32)


def _network(case, seed, n=None, deg=None, utility=None):
    n, deg = n or case["n"], deg or case["deg"]
    graph, utility = case.get("graph", "ring"), utility or case.get("utility", "log")
    rng = np.random.default_rng([seed, n, deg])
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    if graph == "knn":
        tail, head = _knn(n, deg, rng)
        cap = np.exp(rng.uniform(math.log(0.5), math.log(5.0), size=tail.size))
        w = torch.rand((n, n), dtype=torch.float64, device="cuda", generator=gen)
        w = torch.exp(w * (math.log(3.0) - math.log(0.3)) + math.log(0.3))
    else:
        tail, head = _ring(n, deg, rng)
        cap = rng.lognormal(0.0, 0.5, size=tail.size) if utility == "pow" else rng.uniform(1.0, 10.0, size=tail.size)
        w = 0.5 + torch.rand((n, n), dtype=torch.float64, device="cuda", generator=gen)
    w.fill_diagonal_(0.0)
    gamma = None
    if utility == "pow":
        gamma = 0.5 if rng.uniform() < 0.5 or n > 1500 else float(rng.uniform(0.3, 0.7))
    elif utility == "powij":
        gamma = (0.3 + 0.4 * torch.rand((n, n), dtype=torch.float64, device="cuda", generator=gen)).cpu().numpy()
    sign = rng.choice([-1.0, 1.0], size=tail.size)
    return SimpleNamespace(n=n, tail=tail, head=head, cap=cap, cap2=cap * (1.0 + 0.1 * sign),
                           kind="log" if utility == "log" else "pow", w=w.cpu().numpy(), gamma=gamma)


def _many(case, seed):
    """The networks of a batch or a serving process: uneven sizes and degrees, half log."""
    rng = np.random.default_rng([case["count"], case["n"], case["n_hi"]])   # sizes: the case's own
    got = []
    for b in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n"]), math.log(case["n_hi"])))))
        deg = int(rng.integers(4, 17)) if case["what"] == "batch" else 8
        got.append(_network(case, seed + 1000 * (b + 1), n=n, deg=max(2, min(deg, n - 2)),
                            utility="log" if case["what"] == "serve" or b % 2 == 0 else "pow"))
    return got


def _columns(case, seed):
    """Columns of the projection as an iteration meets them: most entries below the
    multiplier, the multiplier of the iteration before as the guess."""
    n, m = case["n"], case["m"]
    ld = (n + 3) // 4 * 4
    gen = torch.Generator(device="cuda").manual_seed(seed)
    Q = torch.randn((m, ld), device="cuda", generator=gen)
    cap = torch.rand(m, device="cuda", generator=gen) * 4.0 + 0.5
    mu = torch.rand(m, device="cuda", generator=gen) * 0.5
    return Q, cap, mu, ld


def _options(case):
    return {"stop_mode": "none", "max_iters": case["iters"]}


def prepare(case, seed):
    what = case["what"]
    if what == "project":
        Q, cap, mu, ld = _columns(case, seed)
        return SimpleNamespace(case=case, Q=Q, cap=cap, guess=mu, ld=ld, mu=torch.empty_like(mu),
                               F=torch.empty_like(Q), stream=torch.cuda.current_stream().cuda_stream)
    if what == "solve":
        inst = _network(case, seed)
        p = binding.Problem(inst)
        if case["before"]:
            p.solve(want_T=False, stop_mode="none", max_iters=case["before"], precision=case["precision"])
        return SimpleNamespace(case=case, p=p, caps=[inst.cap, inst.cap2], turn=0)
    insts = _many(case, seed)
    ps = [binding.Problem(i) for i in insts]
    if case.get("before"):
        binding.mcf_solve_batch(ps, binding.mcf_options_default(stop_mode="none", max_iters=case["before"]))
    return SimpleNamespace(case=case, ps=ps, caps=[[i.cap for i in insts], [i.cap2 for i in insts]], turn=0)


# ------------------------------------------------------------------------------ one pass

_KEPT = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp64": torch.float64}


def run(state):
    case, what = state.case, state.case["what"]
    if what == "project":
        state.mu.copy_(state.guess)
        a = (case["n"], case["m"], state.ld, state.Q.data_ptr(), state.cap.data_ptr(), state.F.data_ptr(),
             state.mu.data_ptr(), state.stream)
        if case["entry"] == "noalloc":
            binding.mcf_project_capped_simplex_noalloc(*a, want_dist2=False)
            return {"F": state.F, "mu": state.mu}
        return {"F": state.F, "mu": state.mu, "dist2": binding.mcf_project_capped_simplex(*a)}
    if what == "solve":
        warm = {}
        if case["before"]:
            state.turn ^= 1
            state.p.update_capacities(state.caps[state.turn])
            warm = {"warm_start": 1}
        out = case["out"]
        r = state.p.solve(want_T=True, want_F="F" in out, want_Y="Y" in out, precision=case["precision"],
                          **warm, **_options(case))
        kept = _KEPT[case["precision"]]
        got = {k: torch.from_numpy(r[k]).to(kept) for k in out}
        return {**got, "iters": r["iters"], "utility": r["utility"], "dual_bound": r["dual_bound"]}
    if what == "batch":
        _, rs = binding.mcf_solve_batch(state.ps, binding.mcf_options_default(**_options(case)), want_T=True)
    else:
        state.turn ^= 1
        for p, cap in zip(state.ps, state.caps[state.turn]):
            p.update_capacities(cap)
        tickets = [p.submit(warm_start=1, **_options(case)) for p in state.ps]
        rs = [binding.mcf_wait(t, -1, p.n, p.m, want_T=True) for t, p in zip(tickets, state.ps)]
    return {"T": torch.cat([torch.from_numpy(r["T"]).float().ravel() for r in rs]),
            "iters": torch.tensor([r["iters"] for r in rs])}


# ------------------------------------------------------------------------------ its bounds

def _iteration(n, m, sf, sp):
    """Bytes and operations that one PDHG iteration cannot do without: F read and written, Y
    read and written, F A^T kept between iterations, w read; the projection and the two
    incidence products per flow, the prox per pair."""
    return 2.0 * sf * n * m + 5.0 * sp * n * n + 16.0 * m, 14.0 * n * m + 20.0 * n * n


def work(case):
    what = case["what"]
    if what == "project":
        n, m = case["n"], case["m"]
        return {"bytes": 8.0 * n * m + 12.0 * m, "flops": 6.0 * n * m}
    if what == "solve":
        n = case["n"]
        m = n * case["deg"] * (1.15 if case["graph"] == "knn" else 1.0)
        sf, sp = {"fp32": (4, 4), "bf16": (2, 4), "fp64": (8, 8)}[case["precision"]]
        b, f = _iteration(n, m, sf, sp)
        b, f, out = b * case["iters"], f * case["iters"], 8.0 * n * n
    else:
        b = f = out = 0.0
        for i in range(case["count"]):   # the sizes' mean over the log-uniform range
            n = math.exp(math.log(case["n"]) + (i + 0.5) / case["count"] * math.log(case["n_hi"] / case["n"]))
            bi, fi = _iteration(n, n * (10 if what == "batch" else 8), 4, 4)
            b, f, out = b + bi * case["iters"], f + fi * case["iters"], out + 8.0 * n * n
    return {"bytes": b + out, "flops": f}


# ------------------------------------------------------------------------------ in 64 bits

def _project64(Q, c, mu):
    """Multipliers of the capped-simplex projection of the rows of Q: Newton on the convex,
    decreasing, piecewise linear sum (q - mu)_+ - c, from a point left of the root."""
    mu = mu.clone()
    for _ in range(200):
        s = (Q - mu[:, None]).clamp_(min=0.0)
        cnt = (s > 0).sum(1)
        step = torch.where(cnt > 0, (s.sum(1) - c) / cnt.clamp(min=1), torch.zeros_like(mu))
        new = torch.maximum(mu + step.clamp(min=0.0), mu)
        done = torch.equal(new, mu) or bool(((new - mu) <= 1e-15 * new.abs()).all())
        mu = new
        if done:
            break
    return mu


def _prox64(v, beta, w, gamma):
    if gamma is None:
        s = torch.sqrt(v * v + 4.0 * beta * w)
        return torch.where(v <= 0, 0.5 * (v - s), -2.0 * beta * w / (v + s))
    c1 = gamma / (1.0 - gamma)
    k = c1 * beta * (1.0 / gamma - 1.0) * (w * gamma) ** (1.0 / (1.0 - gamma))
    lo = (-v).clamp(min=0.0)
    top = k ** (1.0 / (c1 + 2.0))
    size = v.abs().clamp(min=1e-300)
    t = torch.where(v >= 0, torch.minimum(top, (k / size) ** (1.0 / (c1 + 1.0))),
                    lo + torch.minimum(top, k / size ** (c1 + 1.0)))
    for _ in range(100):   # Newton from the right of the root: monotone
        p = t ** c1
        new = torch.maximum(t - (p * t * (t + v) - k) / (p * ((c1 + 2.0) * t + (c1 + 1.0) * v)), lo)
        new = torch.minimum(new, t)
        if torch.equal(new, t):
            break
        t = new
    return -t


class _Exact:
    """The paper's Algorithm 2.1 in 64 bits on dense arrays, one row for each edge or node."""

    def __init__(self, inst):
        g = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
        n, m = inst.n, inst.tail.size
        self.n, self.tail, self.head, self.cap = n, g(inst.tail).long(), g(inst.head).long(), g(inst.cap)
        self.w = g(inst.w).t().contiguous()
        self.gamma = None
        if inst.kind == "pow":
            self.gamma = g(np.broadcast_to(np.asarray(inst.gamma, dtype=np.float64), (n, n)).copy()).t().contiguous()
        deg = torch.bincount(self.tail, minlength=n) + torch.bincount(self.head, minlength=n)
        self.eta = 1.0 / math.sqrt(2.0 * float(deg.max()))
        self.eye = torch.eye(n, dtype=torch.bool, device="cuda")
        self.w[self.eye] = 1.0
        self.F = torch.zeros((m, n), dtype=torch.float64, device="cuda")
        self.Y = torch.where(self.eye, 0.0, -1.0).double()
        self.omega = 1.0
        self.mu = torch.zeros(m, dtype=torch.float64, device="cuda")

    def into_nodes(self, F):
        return torch.zeros((self.n, self.n), dtype=torch.float64, device="cuda").index_add_(
            0, self.head, F).index_add_(0, self.tail, F, alpha=-1.0)

    def iterate(self, count):
        for k in range(count):
            alpha, beta = self.eta / self.omega, self.eta * self.omega
            Q = self.F + alpha * (self.Y[self.head] - self.Y[self.tail])
            mu = _project64(Q, self.cap, torch.zeros_like(self.mu))
            Fhat = (Q - mu[:, None]).clamp_(min=0.0)
            V = self.Y - beta * self.into_nodes(2.0 * Fhat - self.F)
            Yhat = torch.where(self.eye, 0.0, _prox64(V, beta, self.w, self.gamma))
            dF, dY = RHO * (Fhat - self.F), RHO * (Yhat - self.Y)
            f, y = float(dF.norm()), float(dY.norm())
            self.F, self.Y = self.F + dF, self.Y + dY
            if k % K_ADAPT == 0 and f > 1e-5 and y > 1e-5:
                self.omega = math.sqrt(y / f) * math.sqrt(self.omega)
        return {"T": -self.into_nodes(Fhat).t(), "F": Fhat.t(), "Y": Yhat.t()}


def exact(case, seed):
    what = case["what"]
    if what == "project":
        Q, cap, _, ld = _columns(case, seed)
        Q = Q.double()
        Q[:, case["n"]:] = 0.0
        mu = _project64(Q, cap.double(), torch.zeros(case["m"], dtype=torch.float64, device="cuda"))
        F = (Q - mu[:, None]).clamp_(min=0.0)
        got = {"F": F, "mu": mu}
        return got if case["entry"] == "noalloc" else {**got, "dist2": float((F - Q).square().sum())}
    if what == "solve":
        if case["n"] ** 2 * case["deg"] * (case["iters"] + case["before"]) > 1.2e10:
            return None
        if case["precision"] == "bf16":
            return None   # the stored type, not the arithmetic, sets its error
        inst = _network(case, seed)
        x = _Exact(inst)
        if case["before"]:
            x.iterate(case["before"])
            x.cap = torch.as_tensor(inst.cap2, device="cuda")
        r = x.iterate(case["iters"])
        keep = {k: r[k].contiguous() for k in case["out"]}
        return {**keep, "iters": None, "utility": None, "dual_bound": None}
    insts = _many(case, seed)
    if sum(i.n * i.tail.size for i in insts) * case["iters"] > 1e10:
        return None
    Ts = []
    for i in insts:
        x = _Exact(i)
        if case.get("before"):
            x.iterate(case["before"])
            x.cap = torch.as_tensor(i.cap2, device="cuda")
        Ts.append(x.iterate(case["iters"])["T"].ravel())
    return {"T": torch.cat(Ts), "iters": None}
