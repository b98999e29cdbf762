"""Performance cases: the work users have this library do, through its public
entry points, from the smallest problems (latency) to the largest (throughput).

Each case is one call sequence of a real program on a handle that the program
keeps: reset and iterate a tree-structured problem (or a batch of them) for a
fixed budget of half-steps and read the potentials, check and round a finished
iterate, iterate a junction tree, or take one gradient of the warm-start
network.  Iterates are deterministic for a fixed budget, so outputs can be
compared value by value.

FP32 handles return potentials as float32 device rows; the scalars their check
and rounding report carry FP32-grade iterates, so they are returned as float32.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2406_10849_gb300 as T
from paper_2406_10849_gb300 import treeot


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one small chain solved in double precision: every launch counts (an interactive or
        # inner-loop solve; 5 nodes on a 64-point grid, stored costs)
        dict(name="chain_fp64", kind="tree", shape="chain", trees=1, nodes_lo=5, nodes_hi=5, n_lo=64, n_hi=64,
             dim=1, support="grid", cost="matrix", precision="fp64", mode="auto", persistent=False,
             eps_lo=0.01, eps_hi=0.01, call="solve", steps=128, lowp_start=0),
        # one barycenter of eight images on a 32 x 32 grid: a single mid-size request to a service
        dict(name="star_32x32", kind="tree", shape="star", trees=1, nodes_lo=9, nodes_hi=9, n_lo=1024, n_hi=1024,
             dim=2, support="grid", cost="points", precision="fp32", mode="auto", persistent=False,
             eps_lo=0.005, eps_hi=0.005, call="solve", steps=128, lowp_start=0),
        # the paper's own experiment: a batch of small barycenters on 1-D grids of 10 to 640 points
        dict(name="barycenters_1d", kind="tree", shape="star", trees=45, nodes_lo=4, nodes_hi=17, n_lo=10, n_hi=640,
             dim=1, support="grid", cost="points", precision="fp32", mode="auto", persistent=False,
             eps_lo=0.002, eps_hi=0.03, call="solve", steps=128, lowp_start=0),
        # a batch of small random trees, with the persistent launch allowed (many small requests at once)
        dict(name="trees_small", kind="tree", shape="random", trees=64, nodes_lo=4, nodes_hi=16, n_lo=64, n_hi=512,
             dim=2, support="cloud", cost="points", precision="fp32", mode="auto", persistent=True,
             eps_lo=0.002, eps_hi=0.05, call="half_steps", steps=32, lowp_start=0),
        # the batched workload: uneven random trees on 2-D point clouds, costs recomputed in the kernel
        dict(name="trees_batched", kind="tree", shape="random", trees=128, nodes_lo=4, nodes_hi=32, n_lo=128,
             n_hi=2048, dim=2, support="cloud", cost="points", precision="fp32", mode="auto", persistent=False,
             eps_lo=0.002, eps_hi=0.05, call="half_steps", steps=16, lowp_start=0),
        # one tree with ragged stored cost matrices (costs that are no point distance; row lengths
        # that are no multiple of four)
        dict(name="tree_ragged_matrix", kind="tree", shape="random", trees=1, nodes_lo=12, nodes_hi=12, n_lo=201,
             n_hi=1203, dim=3, support="cloud", cost="matrix", precision="fp32", mode="auto", persistent=False,
             eps_lo=0.02, eps_hi=0.02, call="solve", steps=64, lowp_start=0),
        # the headline workload: a 64-node tree, 4096 points per node, 4.2 GB of stored costs
        dict(name="tree_64x4096_matrix", kind="tree", shape="random", trees=1, nodes_lo=64, nodes_hi=64, n_lo=4096,
             n_hi=4096, dim=3, support="cloud", cost="matrix", precision="fp32", mode="auto", persistent=False,
             eps_lo=0.01, eps_hi=0.01, call="half_steps", steps=8, lowp_start=0),
        # the same kind of tree in the BF16 absorbed phase (the fast form of a stored-cost solve)
        dict(name="tree_bf16_matrix", kind="tree", shape="random", trees=1, nodes_lo=32, nodes_hi=32, n_lo=2048,
             n_hi=2048, dim=3, support="cloud", cost="matrix", precision="fp32", mode="bf16", persistent=False,
             eps_lo=0.01, eps_hi=0.01, call="half_steps", steps=20, lowp_start=4),
        # a batch of barycenters that share one Gibbs kernel, in the tensor-core phase (training data
        # for the warm start, image batches)
        dict(name="stars_bf16", kind="tree", shape="star", trees=500, nodes_lo=9, nodes_hi=9, n_lo=1024, n_hi=1024,
             dim=2, support="grid", cost="points", precision="fp32", mode="bf16", persistent=False,
             eps_lo=0.005, eps_hi=0.005, call="half_steps", steps=32, lowp_start=2),
        # the end of a solve: the FP64-grade check and the rounding to feasible plans of a batch
        dict(name="check_round", kind="finish", shape="random", trees=24, nodes_lo=4, nodes_hi=16, n_lo=128,
             n_hi=1400, dim=2, support="cloud", cost="points", eps_lo=0.005, eps_hi=0.05, steps=6),
        # Wasserstein least squares on its junction tree through the general separator update
        dict(name="junction_wls", kind="junction", cliques=12, d=20, steps=32),
        # one gradient of the warm-start network at its training shape, and a prediction
        dict(name="mlp_gradient", kind="mlp", inputs=1025, hidden=512, outputs=1024, batch=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any kind, sizes over the whole range."""
    kind = rng.choice(["chain", "star", "bary1d", "small", "batched", "ragged", "large", "bf16", "stars", "finish",
                       "junction", "mlp"])
    base = dict(kind="tree", trees=1, dim=2, support="cloud", cost="points", precision="fp32", mode="auto",
                persistent=False, eps_lo=0.005, eps_hi=0.03, call="half_steps", lowp_start=0)
    if kind == "chain":
        J, n = rng.randint(3, 12), _log_int(rng, 16, 150)
        base.update(shape="chain", nodes_lo=J, nodes_hi=J, n_lo=n, n_hi=n, dim=1, support="grid",
                    cost=rng.choice(["matrix", "points"]), precision="fp64", call="solve",
                    steps=2 * rng.randint(16, 64))
    elif kind == "star":
        J, side = rng.randint(3, 12), rng.randint(8, 40)
        base.update(shape="star", nodes_lo=J, nodes_hi=J, n_lo=side * side, n_hi=side * side, support="grid",
                    call="solve", steps=2 * rng.randint(16, 64))
    elif kind == "bary1d":
        lo = _log_int(rng, 5, 60)
        base.update(shape="star", trees=_log_int(rng, 1, 60), nodes_lo=3, nodes_hi=rng.randint(4, 24), n_lo=lo,
                    n_hi=_log_int(rng, 100, 1000), dim=1, support="grid", call="solve", steps=2 * rng.randint(16, 64))
    elif kind == "small":
        base.update(shape="random", trees=_log_int(rng, 2, 64), nodes_lo=4, nodes_hi=rng.randint(5, 16),
                    n_lo=_log_int(rng, 20, 100), n_hi=_log_int(rng, 200, 600), dim=rng.randint(1, 3),
                    persistent=rng.random() < 0.5, eps_lo=0.002, eps_hi=0.05, steps=rng.randint(4, 32))
    elif kind == "batched":
        base.update(shape="random", trees=_log_int(rng, 8, 100), nodes_lo=4, nodes_hi=rng.randint(8, 32), n_lo=128,
                    n_hi=_log_int(rng, 600, 2048), dim=rng.choice([2, 2, 3]), eps_lo=0.002, eps_hi=0.05,
                    steps=rng.randint(4, 16))
    elif kind == "ragged":
        J = rng.randint(3, 20)
        base.update(shape="random", nodes_lo=J, nodes_hi=J, n_lo=_log_int(rng, 30, 300),
                    n_hi=_log_int(rng, 400, 1500), dim=3, cost="matrix", eps_lo=0.02, eps_hi=0.02,
                    call=rng.choice(["solve", "half_steps"]), steps=2 * rng.randint(4, 32))
    elif kind == "large":
        J, n = rng.randint(4, 40), rng.randint(1800, 4097)
        base.update(shape="random", nodes_lo=J, nodes_hi=J, n_lo=n, n_hi=n, dim=3, cost="matrix", eps_lo=0.01,
                    eps_hi=0.01, steps=rng.randint(2, 8))
    elif kind == "bf16":
        J, n = rng.randint(4, 24), rng.randint(500, 2600)
        base.update(shape="random", nodes_lo=J, nodes_hi=J, n_lo=n, n_hi=n, dim=3, cost="matrix", mode="bf16",
                    eps_lo=0.01, eps_hi=0.01, steps=rng.randint(8, 20), lowp_start=4)
    elif kind == "stars":
        J, side = rng.randint(5, 10), rng.randint(16, 33)
        base.update(shape="star", trees=_log_int(rng, 20, 400), nodes_lo=J, nodes_hi=J, n_lo=side * side,
                    n_hi=side * side, support="grid", mode="bf16", eps_lo=0.005, eps_hi=0.005,
                    steps=rng.randint(8, 32), lowp_start=2)
    elif kind == "finish":
        base = dict(kind="finish", shape="random", trees=_log_int(rng, 1, 24), nodes_lo=4, nodes_hi=rng.randint(5, 16),
                    n_lo=_log_int(rng, 30, 200), n_hi=_log_int(rng, 300, 1400), dim=rng.randint(1, 3),
                    support="cloud", cost=rng.choice(["points", "points", "matrix"]), eps_lo=0.005, eps_hi=0.05,
                    steps=rng.randint(3, 6))
    elif kind == "junction":
        base = dict(kind="junction", cliques=rng.randint(2, 16), d=_log_int(rng, 5, 24), steps=rng.randint(8, 32))
    else:
        n = rng.randint(8, 33) ** 2
        base = dict(kind="mlp", inputs=n + 1, hidden=rng.choice([128, 256, 384, 512]), outputs=n,
                    batch=rng.randint(16, 256))
    return base


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _edges(shape, J, rng):
    if shape == "chain":
        return np.array([[i, i + 1] for i in range(J - 1)], np.int32)
    if shape == "star":
        return np.array([[0, i] for i in range(1, J)], np.int32)
    # random tree: node i joins a uniform earlier node, labels shuffled
    order = rng.permutation(J)
    return np.array([[order[rng.integers(0, i)], order[i]] for i in range(1, J)], np.int32)


def _grid(n, dim):
    side = int(round(n ** (1.0 / dim)))
    if side ** dim != n:
        raise ValueError("grid supports need a perfect power")
    t = np.arange(side) / max(side - 1, 1)
    axes = np.meshgrid(*([t] * dim), indexing="ij")
    return np.stack([a.reshape(-1) for a in axes], 1).astype(np.float32)


def _mixtures(x, rng, count, comps=3):
    """`count` Gaussian-mixture densities at the support points, each normalised."""
    x = x.astype(np.float64)
    dim = x.shape[1]
    out = np.zeros((count, x.shape[0]))
    w = rng.dirichlet(np.ones(comps), count)
    mean = rng.uniform(0.15, 0.85, (count, comps, dim))
    sig = rng.uniform(0.05, 0.15, (count, comps))
    for c in range(comps):
        r2 = sum((x[None, :, k] - mean[:, c, k][:, None]) ** 2 for k in range(dim))
        out += (w[:, c] / sig[:, c] ** dim)[:, None] * np.exp(-r2 / (2.0 * sig[:, c] ** 2)[:, None])
    # far tails: a floor of 1e-30 of the mass keeps every marginal a full-support density
    out += 1e-30 * out.sum(1, keepdims=True)
    return out / out.sum(1, keepdims=True)


def _problems(case, seed):
    # the trees' shapes and sizes belong to the case; points, marginals and eps come from the seed
    shapes = np.random.default_rng([case["trees"], case["nodes_hi"], case["n_lo"], case["n_hi"], 10849])
    rng = np.random.default_rng([seed, 2406])
    out = []
    shared = None
    for _ in range(case["trees"]):
        J = int(shapes.integers(case["nodes_lo"], case["nodes_hi"] + 1))
        edges = _edges(case["shape"], J, shapes)
        deg = np.bincount(edges.reshape(-1), minlength=J)
        fixed = deg == 1
        if case["support"] == "grid":
            if case["n_lo"] == case["n_hi"]:
                n0 = case["n_lo"]
            else:
                n0 = int(round(math.exp(shapes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
            if shared is None or shared.shape[0] != n0:
                shared = _grid(n0, case["dim"])
            n = np.full(J, n0, np.int32)
            coords = [shared] * J
        else:
            n = shapes.integers(case["n_lo"], case["n_hi"] + 1, J).astype(np.int32)
            coords = [rng.random((int(k), case["dim"])).astype(np.float32) for k in n]
        if case["support"] == "grid":
            ids = np.flatnonzero(fixed)
            m = _mixtures(shared, rng, len(ids))
            marg = {int(j): m[k] for k, j in enumerate(ids)}
        elif case["cost"] == "matrix":
            marg = {}
            for j in np.flatnonzero(fixed):
                v = rng.dirichlet(np.ones(int(n[j])))
                marg[int(j)] = v / v.sum()
        else:
            marg = {int(j): _mixtures(coords[j], rng, 1)[0] for j in np.flatnonzero(fixed)}
        eps = math.exp(rng.uniform(math.log(case["eps_lo"]), math.log(case["eps_hi"])))
        scale = 0.5 if case["support"] == "grid" and case["dim"] == 2 else 1.0
        out.append(SimpleNamespace(
            num_nodes=J, num_edges=J - 1, edges=edges, n=n, fixed=fixed, marginals=marg, eps=eps, coords=coords,
            cost_scale=scale, cost_kind="dense" if case["cost"] == "matrix" else "sqeuclid"))
    return out


def _squared(xa, xb, scale, dtype=torch.float64):
    """scale * |x - y|^2 in FP64 on the GPU, between FP32 support points."""
    a = torch.as_tensor(xa, device="cuda").to(torch.float64)
    b = torch.as_tensor(xb, device="cuda").to(torch.float64)
    acc = 0.0
    for k in range(a.shape[1]):
        acc = acc + (a[:, k, None] - b[None, :, k]) ** 2
    return (acc * scale).to(dtype)


def _matrices(problems):
    return [[_squared(p.coords[a], p.coords[b], p.cost_scale, torch.float32) for a, b in p.edges] for p in problems]


def _items(problems):
    pr = np.array([i for i, p in enumerate(problems) for _ in range(2 * p.num_edges)], np.int32)
    de = np.array([d for p in problems for d in range(2 * p.num_edges)], np.int32)
    return pr, de


def _owner(p, d):
    return int(p.edges[d // 2][d % 2])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        net = T.MLP(case["inputs"], case["hidden"], case["outputs"], case["batch"], seed)
        net.set_input_log(case["inputs"] - 1, 1e-30, 1.0 / 16.0)
        x, target = _mlp_data(case, seed)
        return SimpleNamespace(case=case, net=net, x=x, target=target,
                               grads=torch.zeros(net.num_params, device="cuda"),
                               y=torch.zeros(case["batch"], case["outputs"], device="cuda"))
    if kind == "junction":
        return SimpleNamespace(case=case, solver=treeot.JunctionSolver(_wls(case, seed)))
    problems = _problems(case, seed)
    dense = _matrices(problems) if case["cost"] == "matrix" else None
    if kind == "finish":
        solver = T.Solver(problems, T.options(precision="fp32"), device_costs=dense)
        for i, p in enumerate(problems):
            solver.set_potentials({k: v.cpu().numpy() for k, v in _iterate(p, case["steps"]).items()}, i)
        return SimpleNamespace(case=case, solver=solver, side=(case["steps"]) % 2)
    opts = dict(precision=case["precision"], apply_mode=case["mode"], persistent=case["persistent"])
    if case["mode"] == "bf16":
        opts.update(lowp_start=case["lowp_start"], refine_tol=0.0)
    if case["call"] == "solve":  # a fixed budget of half-steps, then the check
        opts.update(tol=0.0, max_half_steps=case["steps"])
    solver = T.Solver(problems, T.options(**opts), device_costs=dense)
    pr, de = _items(problems)
    rows = None
    if case["precision"] == "fp32":
        rows = torch.zeros(len(pr), max(int(p.n.max()) for p in problems), device="cuda")
    return SimpleNamespace(case=case, solver=solver, problems=problems, pr=pr, de=de, rows=rows)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state.case
    if case["kind"] == "mlp":
        loss = state.net.backward(state.x, state.target, state.grads)
        state.net.forward(state.x, state.y)
        return {"loss": np.float32(loss), "grads": state.grads, "y": state.y}
    s = state.solver
    if case["kind"] == "junction":
        s.reset()
        s.half_steps(case["steps"])
        return {"cost": s.transport_cost(), "plans": [s.plan(c) for c in range(case["cliques"])]}
    if case["kind"] == "finish":
        check, rounded = s.check(), s.round(state.side)
        f32 = lambda rows, key: np.array([r[key] for r in rows], np.float32)
        return {"transport_cost": f32(check, "transport_cost"), "residual_sum": f32(check, "residual_sum_l1"),
                "residual_max": f32(check, "max_marginal_l1"), "rounded_cost": f32(rounded, "rounded_transport_cost")}
    s.reset()
    out = {}
    if case["call"] == "solve":
        _, res = s.solve()
        if case["precision"] == "fp64":
            out["transport_cost"] = np.array([r["transport_cost"] for r in res])
        else:
            out["transport_cost"] = np.array([r["transport_cost"] for r in res], np.float32)
    else:
        s.half_steps(case["steps"])
    if case["precision"] == "fp64":
        out["potentials"] = [s.potential(int(p), int(d)) for p, d in zip(state.pr, state.de)]
    else:
        out["potentials"] = s.get_potentials_batch(state.pr, state.de, state.rows)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _sizes(case):
    """(elements of every edge's plan, length of all directed-edge vectors), expected over the draws of a case."""
    J = 0.5 * (case["nodes_lo"] + case["nodes_hi"])
    lo, hi = case["n_lo"], case["n_hi"]
    if case["support"] == "grid" and lo < hi:  # one log-uniform size per tree
        w = math.log(hi / lo)
        m1, m2 = (hi - lo) / w, (hi * hi - lo * lo) / (2.0 * w)
    else:
        m1 = 0.5 * (lo + hi)
        m2 = m1 * m1
    return case["trees"] * (J - 1) * m2, case["trees"] * (J - 1) * 2 * m1


def work(case):
    if case["kind"] == "mlp":
        i, h, o, b = case["inputs"], case["hidden"], case["outputs"], case["batch"]
        p = i * h + h * h + h * o + 2 * h + o
        # forward twice, two products per layer backward (no gradient of the inputs)
        macs = 2 * b * (i * h + h * h + h * o) + b * (i * h + 2 * h * h + 2 * h * o)
        return {"bytes": 4.0 * (2 * p + b * (i + 2 * o)), "flops": 2.0 * macs}
    if case["kind"] == "junction":
        J, d = case["cliques"], case["d"]
        elems = J * d ** 3
        return {"bytes": 8.0 * elems + 8.0 * elems + 8.0 * J * (d * d + d) * case["steps"],
                "flops": 4.0 * elems * (case["steps"] + 2)}
    elems, vec = _sizes(case)
    dim = case["dim"]
    # per plan element: the squared distance (recomputed costs), the exponent's argument, its
    # exponential and the sum
    per = (3 * dim - 1 if case["cost"] == "points" else 0) + 4
    if case["kind"] == "finish":
        return {"bytes": 8.0 * vec * 2 + (4.0 * elems if case["cost"] == "matrix" else 0.0),
                "flops": per * elems * 4.0}
    size = 8.0 if case["precision"] == "fp64" else 4.0
    nbytes = size * vec * case["steps"] + size * vec
    if case["cost"] == "matrix":
        low = max(0, case["steps"] - case["lowp_start"]) if case["mode"] == "bf16" else 0
        nbytes += 4.0 * elems * (case["steps"] - low) + 2.0 * elems * low
    return {"bytes": nbytes, "flops": per * elems * case["steps"]}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------

def _log_gamma(p, j):
    if p.fixed[j]:
        return torch.log(torch.as_tensor(p.marginals[j], device="cuda"))
    return torch.zeros(int(p.n[j]), dtype=torch.float64, device="cuda")


def _colours(p):
    nb = [[] for _ in range(p.num_nodes)]
    for a, b in p.edges:
        nb[int(a)].append(int(b))
        nb[int(b)].append(int(a))
    col, todo = {0: 0}, [0]
    while todo:
        v = todo.pop()
        for w in nb[v]:
            if w not in col:
                col[w] = 1 - col[v]
                todo.append(w)
    return nb, col


def _costs64(p):
    f32 = p.cost_kind == "dense"  # stored costs are FP32 values
    out = {}
    for a, b in p.edges:
        c = _squared(p.coords[a], p.coords[b], p.cost_scale, torch.float32 if f32 else torch.float64).to(torch.float64)
        out[(int(a), int(b))] = c
    return out


def _iterate(p, steps, costs=None):
    """`steps` half-steps of bipartite iterative scaling from zero potentials, in FP64."""
    nb, col = _colours(p)
    costs = _costs64(p) if costs is None else costs
    neg = {k: c / -p.eps for k, c in costs.items()}
    lg = [_log_gamma(p, j) for j in range(p.num_nodes)]
    f = {}
    for a, b in p.edges:
        f[(int(a), int(b))] = torch.zeros(int(p.n[a]), dtype=torch.float64, device="cuda")
        f[(int(b), int(a))] = torch.zeros(int(p.n[b]), dtype=torch.float64, device="cuda")

    def message(j, k):
        g = f[(k, j)] / p.eps + lg[k]
        if (j, k) in neg:
            return torch.logsumexp(neg[(j, k)] + g[None, :], 1)
        return torch.logsumexp(neg[(k, j)] + g[:, None], 0)

    for t in range(steps):
        new = {}
        for j in range(p.num_nodes):
            if col[j] != t % 2:
                continue
            m = {k: message(j, k) for k in nb[j]}
            if p.fixed[j]:
                new[(j, nb[j][0])] = -p.eps * m[nb[j][0]]
            else:
                s = sum(m.values()) / len(nb[j])
                z = torch.logsumexp(s, 0)
                for k in nb[j]:
                    new[(j, k)] = p.eps * (s - z - m[k])
        f.update(new)
    return f


def _plans(p, f, costs):
    out = {}
    for (a, b), c in costs.items():
        arg = (f[(a, b)][:, None] + f[(b, a)][None, :] - c) / p.eps + _log_gamma(p, a)[:, None] + _log_gamma(p, b)
        out[(a, b)] = torch.exp(arg)
    return out


def _transport(plans, costs):
    return sum(float((plans[k] * costs[k]).sum()) for k in costs)


def _exact_finish(case, seed):
    out = {"transport_cost": [], "residual_sum": [], "residual_max": [], "rounded_cost": []}
    side = case["steps"] % 2
    for p in _problems(case, seed):
        nb, col = _colours(p)
        costs = _costs64(p)
        plans = _plans(p, _iterate(p, case["steps"], costs), costs)
        q = {}
        for (a, b), m in plans.items():
            q[(a, b)], q[(b, a)] = m.sum(1), m.sum(0)
        terms, target = [], []
        for j in range(p.num_nodes):
            mine = [q[(j, k)] for k in nb[j]]
            mean = sum(mine) / len(mine)
            if p.fixed[j]:
                mean = torch.as_tensor(p.marginals[j], device="cuda")
            terms += [float((v - mean).abs().sum()) for v in mine]
            target.append(mean / mean.sum())
        out["transport_cost"].append(_transport(plans, costs))
        out["residual_sum"].append(sum(terms))
        out["residual_max"].append(max(terms))
        cost = 0.0
        for (a, b), m in plans.items():
            c = costs[(a, b)]
            j, k = (a, b) if col[a] == side else (b, a)
            if j != a:
                m, c = m.t(), c.t()
            m = m * torch.clamp(target[j] / m.sum(1), max=1.0)[:, None]
            m = m * torch.clamp(target[k] / m.sum(0), max=1.0)[None, :]
            er, ec = target[j] - m.sum(1), target[k] - m.sum(0)
            cost += float((m * c).sum())
            if float(er.abs().sum()) > 0:
                cost += float(er @ (c @ ec)) / float(er.abs().sum())
        out["rounded_cost"].append(cost)
    return {k: np.array(v) for k, v in out.items()}


def _wls(case, seed):
    """Wasserstein least squares on a uniform grid: cliques {x_0, x_j, x_{J+1}}, the end points'
    separator free, every x_j constrained to a density."""
    J, d = case["cliques"], case["d"]
    rng = np.random.default_rng([seed, 849])
    x = np.arange(d) / (d - 1.0)
    costs = []
    for j in range(1, J + 1):
        t = j / (J + 1.0)
        costs.append(((x[None, :, None] - (1 - t) * x[:, None, None] - t * x[None, None, :]) ** 2
                      + (10.0 / J) * (x[:, None, None] - x[None, None, :]) ** 2).astype(np.float32))
    mu = _mixtures(x[:, None].astype(np.float32), rng, J, 2)
    return SimpleNamespace(
        d=np.full(J + 2, d, np.int32), clique_vars=[(0, j, J + 1) for j in range(1, J + 1)], clique_costs=costs,
        sep_vars=[(0, J + 1)] + [(j,) for j in range(1, J + 1)],
        sep_cliques=[list(range(J))] + [[j] for j in range(J)], sep_gamma=[None] + [(j,) for j in range(1, J + 1)],
        sep_mu=[None] + [mu[j] for j in range(J)], eps=0.2 / (4.0 * J * math.log(d)))


def _exact_junction(case, seed):
    """The trivially nested junction tree is a star of separators: its centre {x_0, x_{J+1}} has d^2
    points and clique j is the edge to the leaf {x_j}."""
    w = _wls(case, seed)
    J, d = case["cliques"], case["d"]
    cost = [torch.as_tensor(c, device="cuda").to(torch.float64).permute(0, 2, 1).reshape(d * d, d)
            for c in w.clique_costs]
    mu = [torch.as_tensor(m, device="cuda") for m in w.sep_mu[1:]]
    fc = [torch.zeros(d * d, dtype=torch.float64, device="cuda") for _ in range(J)]
    fl = [torch.zeros(d, dtype=torch.float64, device="cuda") for _ in range(J)]
    for t in range(case["steps"]):
        if t % 2 == 0:
            m = [torch.logsumexp((fl[j][None, :] - cost[j]) / w.eps + torch.log(mu[j]), 1) for j in range(J)]
            s = sum(m) / J
            z = torch.logsumexp(s, 0)
            fc = [w.eps * (s - z - m[j]) for j in range(J)]
        else:
            fl = [-w.eps * torch.logsumexp((fc[j][:, None] - cost[j]) / w.eps, 0) for j in range(J)]
    plans = [torch.exp((fc[j][:, None] + fl[j][None, :] - cost[j]) / w.eps) * mu[j] for j in range(J)]
    total = sum(float((plans[j] * cost[j]).sum()) for j in range(J))
    return {"cost": total, "plans": [b.reshape(d, d, d).permute(0, 2, 1).contiguous() for b in plans]}


def _mlp_data(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 17)
    b, i, o = case["batch"], case["inputs"], case["outputs"]
    x = torch.rand(b, i, generator=g, device="cuda")
    x[:, :-1] = torch.exp(-20.0 * x[:, :-1])
    x[:, :-1] /= x[:, :-1].sum(1, keepdim=True)
    x[:, -1] = x[:, -1] - 0.5
    return x, 0.05 * torch.randn(b, o, generator=g, device="cuda")


def _mlp_weights(case, seed):
    """The network's seeded initialisation: uniform weights from a SplitMix64 stream, zero biases."""
    i, h, o = case["inputs"], case["hidden"], case["outputs"]
    out, count = [], 0
    for rows, cols in ((h, i), (h, h), (o, h)):
        k = np.arange(count + 1, count + rows * cols + 1, dtype=np.uint64)
        with np.errstate(over="ignore"):
            z = np.uint64(seed) + k * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
        u = (z >> np.uint64(11)).astype(np.float64) / 9007199254740992.0
        out.append(((2.0 * u - 1.0) / math.sqrt(cols)).astype(np.float32).astype(np.float64).reshape(rows, cols))
        count += rows * cols
    return out


def _exact_mlp(case, seed):
    x, target = (v.to(torch.float64) for v in _mlp_data(case, seed))
    x[:, :-1] = torch.log(torch.clamp(x[:, :-1], min=1e-30)) / 16.0
    w = [torch.as_tensor(v, device="cuda").requires_grad_() for v in _mlp_weights(case, seed)]
    b = [torch.zeros(v.shape[0], dtype=torch.float64, device="cuda", requires_grad=True) for v in w]
    gelu = torch.nn.functional.gelu
    y = gelu(gelu(x @ w[0].t() + b[0]) @ w[1].t() + b[1]) @ w[2].t() + b[2]
    loss = ((y - target) ** 2).mean()
    loss.backward()
    grads = []
    for k in range(3):
        for v in (w[k].grad.reshape(-1), b[k].grad):
            grads += [v, torch.zeros(-v.numel() % 8, dtype=torch.float64, device="cuda")]
    return {"loss": float(loss.detach()), "grads": torch.cat(grads), "y": y.detach()}


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "junction":
        return _exact_junction(case, seed)
    if case["kind"] == "finish":
        return _exact_finish(case, seed)
    problems = _problems(case, seed)
    width = max(int(p.n.max()) for p in problems)
    potentials, cost = [], []
    for p in problems:
        costs = _costs64(p)
        f = _iterate(p, case["steps"], costs)
        rows = [f[(_owner(p, d), _owner(p, d ^ 1))] for d in range(2 * p.num_edges)]
        if case["precision"] == "fp32":
            rows = [torch.nn.functional.pad(v, (0, width - v.numel())) for v in rows]
        potentials += rows
        if case["call"] == "solve":
            cost.append(_transport(_plans(p, f, costs), costs))
    out = {"potentials": torch.stack(potentials) if case["precision"] == "fp32" else potentials}
    if case["call"] == "solve":
        out["transport_cost"] = np.array(cost)
    return out
