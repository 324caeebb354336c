"""What a program that uses this package has it do, as cases that can be timed.

A case is one of four kinds of pass through the public entry points:

  solve  a Solver that a program keeps: back to f = 0, a solve with a sweep
         budget, the flows read out into device memory
  batch  a Batch that a program keeps: the same for many small or uneven
         instances at once
  grad   autograd.unrolled_objective and its gradients with respect to the
         capacities and the demands
  fresh  an instance that has just arrived in host memory: create the
         solver, solve, read the flows back to host memory, destroy it

Instances are synthetic and made from the seed alone: grids, nearest-neighbour
graphs and random digraphs; demands as integers in [1, 10] or lognormal;
capacities 1.2 times the load of a witness routing (or 0.7 times, infeasible
in most cases).  An FP32 solve's flows are FP32 values, which the library
widens on read-out; they are kept as float32 here.
"""

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2108_07549_gb300 import pdr
from paper_2108_07549_gb300.autograd import unrolled_objective

ALGOS = {"eso": pdr.ALGO_ESO, "agd": pdr.ALGO_AGD, "gdm": pdr.ALGO_GDM, "ck": pdr.ALGO_CK}
LARGEST = 8.0e9  # edge-commodity updates of one pass of the largest listed case


def listed():
    return [
        # the smallest call: a toy network inside a larger program, latency and launches only
        {"name": "grid5_k10", "kind": "solve", "graph": "grid", "n": 25, "K": 10, "sweeps": 300,
         "algo": "eso", "precision": "fp32"},
        # a small sparse network: several solves of this size per decision
        {"name": "digraph200_k50", "kind": "solve", "graph": "digraph3", "n": 200, "K": 50, "sweeps": 300,
         "algo": "eso", "precision": "fp32"},
        # a regional network with a hundred demands
        {"name": "knn500_k100", "kind": "solve", "graph": "knn", "n": 500, "K": 100, "sweeps": 300,
         "algo": "eso", "precision": "fp32"},
        # a planning network whose flows stay in L2
        {"name": "knn2500_k500", "kind": "solve", "graph": "knn", "n": 2500, "K": 500, "sweeps": 200,
         "algo": "eso", "precision": "fp32"},
        # the largest grid: every sweep streams from HBM
        {"name": "grid100_k10000", "kind": "solve", "graph": "grid", "n": 10000, "K": 10000, "sweeps": 20,
         "algo": "eso", "precision": "fp32"},
        # a large random graph: the rows a vertex gathers lie far apart
        {"name": "digraph20k_k2000", "kind": "solve", "graph": "digraph5", "n": 20000, "K": 2000, "sweeps": 20,
         "algo": "eso", "precision": "fp32"},
        # the momentum method (Alg. 4) on a grid with many commodities
        {"name": "gdm_grid25_k4000", "kind": "solve", "graph": "grid", "n": 625, "K": 4000, "sweeps": 40,
         "algo": "gdm", "precision": "fp32"},
        # the same regional network where the program needs FP64 flows
        {"name": "fp64_knn500_k100", "kind": "solve", "graph": "knn", "n": 500, "K": 100, "sweeps": 150,
         "algo": "eso", "precision": "fp64"},
        # many small scenarios of a study, each with its own network
        {"name": "batch_small", "kind": "batch", "count": 96, "n_min": 100, "n_max": 500, "k_min": 10, "k_max": 100,
         "sweeps": 100, "algo": "eso", "precision": "fp32"},
        # a queue of requests of very uneven size
        {"name": "batch_uneven", "kind": "batch", "count": 24, "n_min": 100, "n_max": 5000, "k_min": 10,
         "k_max": 1000, "sweeps": 30, "algo": "eso", "precision": "fp32"},
        # sensitivities to capacities and demands for a capacity upgrade
        {"name": "grad_digraph5k_k600", "kind": "grad", "graph": "digraph5", "n": 5000, "K": 600, "sweeps": 20,
         "ckpt": 10, "algo": "eso", "precision": "fp32"},
        # a request served from host memory to host memory, K not a multiple of a vector
        {"name": "fresh_grid30_k501", "kind": "fresh", "graph": "grid", "n": 900, "K": 501, "sweeps": 100,
         "algo": "eso", "precision": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edges(graph, n):
    if graph == "grid":
        a = math.isqrt(n)
        return 4 * a * (a - 1)
    return n * {"digraph3": 3, "digraph4": 4, "digraph5": 5, "knn": 6}[graph]


def draw(rng):
    kind = rng.choices(["solve", "batch", "grad", "fresh"], [0.67, 0.17, 0.08, 0.08])[0]
    if kind == "batch":
        n_max = _log(rng, 200, 5000)
        k_max = _log(rng, 20, 1000)
        count = max(8, min(96, int(2.0e9 / (40 * 2 * n_max * k_max)), int(4.8e4 / n_max * 8)))
        return {"kind": kind, "count": count, "n_min": min(100, n_max // 2), "n_max": n_max,
                "k_min": 10, "k_max": k_max, "sweeps": rng.randint(20, 40 if n_max * k_max > 1e5 else 100),
                "algo": "eso", "precision": "fp32"}
    graph = rng.choice(["grid", "knn", "digraph3", "digraph5"])
    if kind == "solve":
        size = math.exp(rng.uniform(math.log(8e2), math.log(3e8)))  # edges x commodities
        n = _log(rng, 25, 20000 if graph != "knn" else 4000)
        if graph == "grid":
            n = min(10000, max(5, math.isqrt(n)) ** 2)
        K = int(min(10007, max(10, size / _edges(graph, n))))
        precision = rng.choices(["fp32", "fp64"], [0.8, 0.2])[0]
        algo = rng.choices(["eso", "gdm", "agd", "ck"], [0.7, 0.1, 0.1, 0.1])[0]
        if precision == "fp64":  # FP64 where it is used: the smaller networks
            K = int(min(K, max(10, 3e6 / _edges(graph, n))))
        cost = _edges(graph, n) * K * (8 if precision == "fp64" else 1)
        sweeps = max(10, min(rng.randint(50, 300), int(0.9 * LARGEST / cost)))
        return {"kind": kind, "graph": graph, "n": n, "K": K, "sweeps": sweeps, "algo": algo, "precision": precision}
    n = _log(rng, 100, 8000 if graph != "knn" else 3000)
    if graph == "grid":
        n = math.isqrt(n) ** 2
    K = int(min(1500, max(10, math.exp(rng.uniform(math.log(1e4), math.log(1.5e7))) / _edges(graph, n))))
    if kind == "grad":
        return {"kind": kind, "graph": graph, "n": n, "K": K, "sweeps": rng.randint(5, 20),
                "ckpt": rng.choice([1, 5, 10]), "algo": rng.choice(["eso", "eso", "ck"]), "precision": "fp32"}
    K = int(max(10, min(K, 4e6 / _edges(graph, n))))
    return {"kind": kind, "graph": graph, "n": n, "K": K, "sweeps": rng.randint(50, 150), "algo": "eso",
            "precision": "fp32"}


# --------------------------------------------------------------------------- inputs


def _csr(n, src, dst):
    order = np.argsort(src, kind="stable")
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=row_ptr[1:])
    return row_ptr, dst[order].astype(np.int32)


def _walk(row_ptr, col, s, steps, rng, goal=None):
    """Follows an arc per step from every s (the one that leads nearest to its goal, or any); the vertices it
    ends on and the arcs it took."""
    deg = np.diff(row_ptr)
    cur, took = s.astype(np.int64), []
    for _ in range(steps):
        if goal is None:
            e = row_ptr[cur] + (rng.random(cur.shape[0]) * deg[cur]).astype(np.int64)
            move = np.ones(cur.shape[0], bool)
        else:
            pts, aim = goal
            width = int(deg.max())
            at = row_ptr[cur][:, None] + np.arange(width)
            ok = np.arange(width)[None, :] < deg[cur][:, None]
            heads = col[np.where(ok, at, 0)]
            dist = np.where(ok, ((pts[heads] - aim[:, None, :]) ** 2).sum(-1), np.inf)
            best = dist.argmin(1)
            rows = np.arange(cur.shape[0])
            move = dist[rows, best] < ((pts[cur] - aim) ** 2).sum(-1)
            e = at[rows, best]
        took.append((e, move))
        cur = np.where(move, col[np.where(move, e, 0)].astype(np.int64), cur)
    return cur, took


def _instance(graph, n, K, seed, factor=1.2):
    """A network, K commodities and capacities of `factor` times the load of a witness routing."""
    rng = np.random.default_rng([seed, n, K])
    s = rng.integers(0, n, K)
    goal, steps = None, 6
    if graph == "grid":
        a = math.isqrt(n)
        r, c = np.divmod(np.arange(n), a)
        arcs = [(v, v + off) for v, off in ((np.flatnonzero(c < a - 1), 1), (np.flatnonzero(c > 0), -1),
                                            (np.flatnonzero(r < a - 1), a), (np.flatnonzero(r > 0), -a))]
        row_ptr, col = _csr(n, np.concatenate([x for x, _ in arcs]), np.concatenate([y for _, y in arcs]))
        goal, steps = np.stack([r, c], 1).astype(np.float64), 2 * a
    elif graph == "knn":
        pts = rng.random((n, 2))
        near = torch.cdist(torch.from_numpy(pts).cuda(), torch.from_numpy(pts).cuda())
        near = near.topk(4, largest=False).indices[:, 1:].cpu().numpy().reshape(-1)
        tail = np.repeat(np.arange(n), 3)
        near = np.where(near == tail, (tail + 1) % n, near)
        row_ptr, col = _csr(n, np.concatenate([tail, near]), np.concatenate([near, tail]))
        goal, steps = pts, int(2 * math.sqrt(n)) + 2
    else:
        out = int(graph[-1])
        tail = np.repeat(np.arange(n), out)
        row_ptr, col = _csr(n, tail, (tail + rng.integers(1, n, n * out)) % n)
    aim = None
    if goal is not None:
        aim = (goal, goal[(s + rng.integers(1, n, K)) % n])
    t, took = _walk(row_ptr, col, s, steps, rng, aim)
    stuck = t == s  # a walk that ended where it began: its first arc's head
    first = row_ptr[s]
    t = np.where(stuck, col[first], t)
    d = rng.integers(1, 11, K).astype(np.float64) if graph != "grid" else rng.lognormal(1.0, 0.5, K)
    load = np.zeros(col.shape[0])
    for e, move in took:
        np.add.at(load, e[move & ~stuck], d[move & ~stuck])
    np.add.at(load, first[stuck], d[stuck])
    return SimpleNamespace(n=n, row_ptr=row_ptr, col=col, u=load * factor, s=s.astype(np.int32),
                           t=t.astype(np.int32), d=d)


def _members(case, seed):
    """The instances of a batch: random out-degree-4 digraphs, a fifth of them short of capacity."""
    rng = np.random.default_rng([seed, case["count"]])
    # the sizes belong to the case, so that every seed's pass does the same work
    sizes = np.random.default_rng([7, case["count"], case["n_max"], case["k_max"]])
    n = sizes.integers(case["n_min"], case["n_max"] + 1, case["count"])
    K = sizes.integers(case["k_min"], case["k_max"] + 1, case["count"])
    return [_instance("digraph4", int(a), int(b), int(rng.integers(1 << 30)), 0.7 if i % 5 == 4 else 1.2)
            for i, (a, b) in enumerate(zip(n, K))]


def _options(case):
    return dict(precision=pdr.PREC_FP64 if case["precision"] == "fp64" else pdr.PREC_FP32, algo=ALGOS[case["algo"]],
                max_sweeps=case["sweeps"])


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "batch":
        insts = _members(case, seed)
        state["batch"] = pdr.Batch(insts, **_options(case))
        state["views"] = [state["batch"].solver(i) for i in range(case["count"])]
        state["flows"] = torch.empty(sum(v.m * v.K for v in state["views"]), dtype=torch.float64, device="cuda")
        return state
    inst = _instance(case["graph"], case["n"], case["K"], seed)
    if case["kind"] == "fresh":
        state["inst"] = inst
        return state
    state["solver"] = pdr.Solver.from_instance(inst, **_options(case))
    if case["kind"] == "solve":
        state["flows"] = torch.empty((state["solver"].m, state["solver"].K), dtype=torch.float64, device="cuda")
    else:
        state["u"] = torch.from_numpy(inst.u).to("cuda", torch.float32).requires_grad_()
        state["d"] = torch.from_numpy(inst.d).to("cuda", torch.float32).requires_grad_()
    return state


# --------------------------------------------------------------------------- one pass


def _flows_into(solver, flows, offset=0):
    """pdr_flows into device memory."""
    solver._check(pdr.load().pdr_flows(solver._h, ctypes.c_void_p(flows.data_ptr() + 8 * offset)))


def _numbers(results, kind):
    return {"z": np.array([r["z"] for r in results], kind),
            "cap_rel": np.array([r["cap_rel"] for r in results], kind),
            "cons_rel": np.array([r["cons_rel"] for r in results], kind),
            "sweeps": np.array([r["sweeps"] for r in results], np.int64),
            "verdict": np.array([r["verdict"] for r in results], np.int64)}


def run(state):
    case = state["case"]
    if case["kind"] == "grad":
        L = unrolled_objective(state["solver"], state["u"], state["d"], case["sweeps"], case["ckpt"])
        gu, gd = torch.autograd.grad(L, [state["u"], state["d"]])
        return {"L": L, "gu": gu, "gd": gd}
    if case["kind"] == "fresh":
        with pdr.Solver.from_instance(state["inst"], **_options(case)) as solver:
            result = solver.solve()
            flows = solver.flows()
        return {"flows": flows.astype(np.float32), **_numbers([result], np.float32)}
    if case["kind"] == "batch":
        state["batch"].reset()
        results = state["batch"].solve()
        at = 0
        for view in state["views"]:
            _flows_into(view, state["flows"], at)
            at += view.m * view.K
        return {"flows": state["flows"].float(), **_numbers(results, np.float32)}
    state["solver"].reset()
    result = state["solver"].solve()
    _flows_into(state["solver"], state["flows"])
    if case["precision"] == "fp64":
        return {"flows": state["flows"], **_numbers([result], np.float64)}
    return {"flows": state["flows"].float(), **_numbers([result], np.float32)}


def work(case):
    """Every sweep takes the flows in and gives new flows; the heights between them need not leave the chip."""
    if case["kind"] == "batch":
        sizes = np.random.default_rng([7, case["count"], case["n_max"], case["k_max"]])
        n = sizes.integers(case["n_min"], case["n_max"] + 1, case["count"])
        K = sizes.integers(case["k_min"], case["k_max"] + 1, case["count"])
        elements = float((4 * n * K).sum())
    else:
        elements = float(_edges(case["graph"], case["n"])) * case["K"]
    size = 8 if case["precision"] == "fp64" else 4
    sweeps = case["sweeps"] * (2.0 if case["kind"] == "grad" else 1.0)  # the gradient goes back through each
    return {"bytes": 2.0 * size * elements * sweeps + 8.0 * elements * (case["kind"] != "grad"),
            "flops": 8.0 * elements * sweeps}


# --------------------------------------------------------------------------- the same in 64 bits


class _Plain:
    """The sweep in plain float64 torch operations."""

    def __init__(self, inst, u=None, d=None, dev="cuda"):
        self.n, self.K, self.m = inst.n, inst.s.shape[0], inst.col.shape[0]
        self.src = torch.from_numpy(np.repeat(np.arange(inst.n), np.diff(inst.row_ptr))).to(dev)
        self.col = torch.from_numpy(inst.col.astype(np.int64)).to(dev)
        self.s = torch.from_numpy(inst.s.astype(np.int64)).to(dev)
        self.t = torch.from_numpy(inst.t.astype(np.int64)).to(dev)
        self.u = torch.from_numpy(inst.u).to(dev) if u is None else u
        self.d = torch.from_numpy(inst.d).to(dev) if d is None else d
        deg = torch.bincount(self.src, minlength=self.n) + torch.bincount(self.col, minlength=self.n)
        self.deg = deg.double()
        self.inv = torch.where(deg > 0, 1.0 / self.deg.clamp(min=1), torch.zeros_like(self.deg))
        self.k = torch.arange(self.K, device=dev)
        self.order = self.k.double() + 1.0

    def excess(self, f):
        x = torch.zeros((self.n, self.K), dtype=torch.float64, device=f.device)
        x = x.index_add(0, self.col, f).index_add(0, self.src, -f)
        return x.index_put((self.s, self.k), self.d, accumulate=True).index_put((self.t, self.k), -self.d,
                                                                              accumulate=True)

    def objective(self, f, x):
        psi = (f.sum(1) - self.u).clamp(min=0)
        return 0.5 * (psi * psi).sum() + 0.5 * (x * x * self.inv[:, None]).sum()

    def sweep(self, f, ck):
        """The exact minimiser of every edge's problem: the root over the sorted row."""
        h = self.excess(f) * self.inv[:, None]
        c = f + 0.5 * (h[self.src] - h[self.col])
        den = 0.0 if ck else 2.0
        with torch.no_grad():
            row = c.clamp(min=0).sort(dim=1, descending=True).values
            cand = (row.cumsum(1) - self.u[:, None]) / (den + self.order)
            root = cand.max(dim=1).values.clamp(min=0)
            active = (c > root[:, None]).double()
            count = active.sum(1)
        if not c.requires_grad:
            return (c - root[:, None]).clamp(min=0)
        theta = ((c * active).sum(1) - self.u) / (den + count).clamp(min=1)
        theta = torch.where((root > 0) & (count > 0), theta, torch.zeros_like(theta))
        return (c - theta[:, None]) * active

    def solve(self, sweeps, algo):
        f = torch.zeros((self.m, self.K), dtype=torch.float64, device=self.u.device)
        if algo in ("eso", "ck"):
            for _ in range(sweeps):
                f = self.sweep(f, algo == "ck")
            return f
        momentum = algo == "gdm"
        beta = torch.full((self.m, 1), 0.1 if momentum else 0.25, dtype=torch.float64, device=f.device)
        v = torch.zeros_like(f)
        for t in range(sweeps):
            h = self.excess(f) * self.inv[:, None]
            drop = h[self.src] - h[self.col]
            psi = (f.sum(1, keepdim=True) - self.u[:, None]).clamp(min=0)
            step = torch.maximum(-f, beta * (drop - psi))
            new = ((f + step).sum(1, keepdim=True) - self.u[:, None]).clamp(min=0)
            dz = 0.5 * (new * new - psi * psi) + (step * (step - drop)).sum(1, keepdim=True)
            accept = dz <= 0
            if momentum:
                v = torch.where(accept, 0.9 * v + step, v)
                f = torch.where(accept, (f + v).clamp(min=0), f)
            else:
                f = torch.where(accept, f + step, f)
            beta = torch.where(accept, beta, (0.5 * beta).clamp(min=1.0 / self.K))
            if t % 10 == 0:
                beta = (2.0 * beta).clamp(max=0.2 if momentum else 0.5)
        return f


def _exact_solve(inst, case):
    plain = _Plain(inst)
    f = plain.solve(case["sweeps"], case["algo"])
    x = plain.excess(f)
    over = (f.sum(1) - plain.u).clamp(min=0)
    scale = plain.u.clamp(min=float(inst.u[inst.u > 0].mean()) if (inst.u > 0).any() else 1.0)
    return f, float(plain.objective(f, x)), float((over / scale).max()), float((x.abs() / plain.d).max())


def exact(case, seed):
    elements = work(case)["flops"] / 8.0
    if elements > 4.0e9 or (case["kind"] == "solve" and elements / case["sweeps"] > 6.0e7):
        return None
    if case["algo"] in ("agd", "gdm") and case["precision"] == "fp32":
        return None  # a step is taken or not by the sign of a difference near 0: 64 bits take another path
    if case["kind"] == "grad":
        inst = _instance(case["graph"], case["n"], case["K"], seed)
        u = torch.from_numpy(inst.u).to("cuda", torch.float32).double().requires_grad_()
        d = torch.from_numpy(inst.d).to("cuda", torch.float32).double().requires_grad_()
        plain = _Plain(inst, u, d)
        f = torch.zeros((plain.m, plain.K), dtype=torch.float64, device="cuda")
        for _ in range(case["sweeps"]):
            f = plain.sweep(f, case["algo"] == "ck")
        L = plain.objective(f, plain.excess(f))
        gu, gd = torch.autograd.grad(L, [u, d])
        return {"L": L.detach(), "gu": gu, "gd": gd}
    insts = _members(case, seed) if case["kind"] == "batch" else [
        _instance(case["graph"], case["n"], case["K"], seed)]
    got = [_exact_solve(inst, case) for inst in insts]
    flows = got[0][0] if case["kind"] != "batch" else torch.cat([g[0].reshape(-1) for g in got])
    out = {"flows": flows.cpu().numpy() if case["kind"] == "fresh" else flows, "sweeps": None, "verdict": None}
    for i, key in enumerate(("z", "cap_rel", "cons_rel")):
        out[key] = np.array([g[1 + i] for g in got])
    return out
