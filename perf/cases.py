"""What the library is used for, as calls that can be timed: propagation of
batches of search nodes, batched searches, proofs over the shared queue, and
the learned policy's scoring and training.

Every case works on the scheduling model that the package builds
(Model.from_rcpsp): tasks with durations U[1,10], resources of capacity
U[5,10], demands U[0,5] and precedences with probability 0.1; below 10 tasks
one resource of capacity 4, durations U[1,5], demands U[1,3] and probability
0.2.  Sizes are those of the tests and of bench.py: 8 to 120 tasks, one store
to ten thousand, one model to 256.

    listed()              the cases
    draw(rng)             one more case of the same ranges
    prepare(case, seed)   models, stores, policies and batches on the GPU
    run(state)            one pass through the public entry points
    work(case)            bytes and operations that a pass cannot do without
    exact(case, seed)     computed numbers in 64 bits, from numpy alone
"""
import math

import numpy as np
import torch

import paper_2207_12116_gb300 as pccp

FEATURES, HIDDEN = 12, 128
GROUP = 16             # mean candidates of a training group
PROOF_NODES = 20000    # models whose optimum takes longer are left out of a proof batch
STRATEGY = {"input_order": pccp.PCCP_INPUT_ORDER, "first_fail": pccp.PCCP_FIRST_FAIL,
            "learned": pccp.PCCP_LEARNED}


def listed():
    return [
        # one node of the smallest family: what a program that drives its own
        # search pays for each call
        {"name": "propagate_8_tasks_1", "kind": "propagate", "tasks": 8, "stores": 1},
        # the benchmark's batch: 10,000 nodes of a 30-task model
        {"name": "propagate_30_tasks_10000", "kind": "propagate", "tasks": 30, "stores": 10000},
        # an ordinary batch of an odd size: the children of a few nodes of a
        # 60-task model, as strong-branching probes make them
        {"name": "propagate_60_tasks_777", "kind": "propagate", "tasks": 60, "stores": 777},
        # the largest family, bench.py --family j120
        {"name": "propagate_120_tasks_1216", "kind": "propagate", "tasks": 120, "stores": 1216},
        # the end-to-end call: stores in page-locked host memory
        {"name": "host_30_tasks_10000", "kind": "host", "tasks": 30, "stores": 10000},
        # a plain solve to the optimum, one team, input order
        {"name": "solve_8_tasks", "kind": "search", "low": 8, "high": 8, "models": 1, "nodes": 0,
         "strategy": "input_order"},
        # the uneven batch in the sequential order, a node limit per model
        {"name": "batch_30_60_tasks_256", "kind": "search", "low": 30, "high": 60, "models": 256,
         "nodes": 500, "strategy": "first_fail"},
        # the same kind of batch with learned branching on 60-task models
        {"name": "learned_60_tasks_64", "kind": "search", "low": 60, "high": 60, "models": 64,
         "nodes": 200, "strategy": "learned"},
        # the large family's batch (a part of it: models are slow to build)
        {"name": "batch_120_tasks_24", "kind": "search", "low": 120, "high": 120, "models": 24,
         "nodes": 50, "strategy": "first_fail"},
        # proofs that nothing beats a known optimum, every team over one
        # queue: how labels are measured and complete batches end
        {"name": "proof_6_10_tasks_256", "kind": "proof", "low": 6, "high": 10, "models": 256},
        # features and scores of the branch variables of a batch of nodes
        {"name": "rank_30_tasks_4000", "kind": "rank", "tasks": 30, "stores": 4000},
        # one training step on a mini-batch of 256 nodes' candidates
        {"name": "train_256_groups", "kind": "train", "groups": 256},
    ]


def _log(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["propagate", "propagate", "propagate", "host", "search", "search", "proof",
                       "rank", "train"])
    if kind in ("propagate", "host", "rank"):
        tasks = _log(rng, 8, 120) if kind == "propagate" else _log(rng, 8, 60)
        most = {"propagate": 10000, "host": 10000, "rank": 4000}[kind]
        # no more cells than 10,000 stores of a 30-task model hold
        most = max(1, min(most, 9_000_000 // (tasks * tasks)))
        return {"kind": kind, "tasks": tasks, "stores": _log(rng, 2, max(2, most))}
    if kind == "search":
        strategy = rng.choice(["input_order", "first_fail", "learned"])
        low = _log(rng, 12, 60)
        high = min(60, low + rng.randint(0, 20))
        models = _log(rng, 1, 200)
        return {"kind": kind, "low": low, "high": high, "models": models,
                "nodes": rng.randint(30, 200), "strategy": strategy}
    if kind == "proof":
        low = rng.randint(6, 9)
        return {"kind": kind, "low": low, "high": rng.randint(low, 9), "models": _log(rng, 1, 256)}
    return {"kind": kind, "groups": _log(rng, 8, 512)}


# ------------------------------------------------------------------- inputs

class Instance:
    """A scheduling instance as Model.from_rcpsp takes it."""

    def __init__(self, n, g):
        small = n < 10
        dur, use, cap = ((1, 5), (1, 3), (4, 4)) if small else ((1, 10), (0, 5), (5, 10))
        self.n = n
        self.durations = tuple(int(x) for x in g.integers(dur[0], dur[1] + 1, n))
        self.capacity = tuple(int(x) for x in g.integers(cap[0], cap[1] + 1, 1 if small else 4))
        self.usage = tuple(tuple(int(x) for x in g.integers(use[0], min(use[1], c) + 1, n))
                           for c in self.capacity)
        pairs = np.argwhere(np.triu(g.random((n, n)) < (0.2 if small else 0.1), 1))
        self.precedences = tuple((int(i), int(j)) for i, j in pairs)
        self.horizon = int(sum(self.durations))


def _rng(seed, *more):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, *more])


def _nodes(inst, count, g):
    """Restrictions (store, task, lo, hi) of `count` search nodes: the root,
    then 0 to 15 decisions in input order, each a random side of a random cut."""
    out = []
    for s in range(count):
        left = int(g.integers(0, 16)) if s > 0 else 0
        cuts = g.random(2 * left)
        k = 0
        for t in range(inst.n):
            lo, hi = 0, inst.horizon
            while k < left and lo < hi:
                cut = lo + int(cuts[2 * k] * (hi - lo))
                if cuts[2 * k + 1] < 0.5:
                    hi = cut
                else:
                    lo = cut + 1
                k += 1
            if lo > 0 or hi < inst.horizon:
                out.append((s, t, lo, hi))
            if k >= left:
                break
    return np.array(out, dtype=np.int64).reshape(-1, 4)


def _stores(model, inst, count, g):
    """Stores [2 (lb, ub), count, n_vars] of random search nodes on the GPU, and
    their depths."""
    r = _nodes(inst, count, g)
    root = torch.from_numpy(np.stack([model.lb0, model.ub0])).cuda()
    stores = root[:, None].repeat(1, count, 1)
    t = torch.from_numpy(r).cuda()
    stores[0, t[:, 0], t[:, 1]] = t[:, 2].int()
    stores[1, t[:, 0], t[:, 1]] = t[:, 3].int()
    depth = torch.bincount(t[:, 0], minlength=count).int()
    return stores, depth


def _weights(g):
    return {"w1": g.normal(0, math.sqrt(2 / FEATURES), (HIDDEN, FEATURES)).astype(np.float32),
            "b1": g.normal(0, 0.1, HIDDEN).astype(np.float32),
            "w2": g.normal(0, math.sqrt(2 / HIDDEN), (HIDDEN, HIDDEN)).astype(np.float32),
            "b2": g.normal(0, 0.1, HIDDEN).astype(np.float32),
            "w3": g.normal(0, math.sqrt(1 / HIDDEN), HIDDEN).astype(np.float32), "b3": 0.0}


def _one(case, seed):
    inst = Instance(case["tasks"], _rng(seed, 1))
    return inst, pccp.Model.from_rcpsp(inst)


def _train_inputs(case, seed):
    g = _rng(seed, 3)
    sizes = g.integers(2, 2 * GROUP - 1, case["groups"])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    f = g.random((int(off[-1]), FEATURES)).astype(np.float32)
    score = g.normal(0, 1, int(off[-1]))
    target = np.concatenate([np.exp(score[a:b]) / np.exp(score[a:b]).sum()
                             for a, b in zip(off[:-1], off[1:])]).astype(np.float32)
    return _weights(g), f, off, target


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("propagate", "host", "rank"):
        inst, model = _one(case, seed)
        s["model"] = model
        stores, depth = _stores(model, inst, case["stores"], _rng(seed, 2))
        if kind == "rank":
            s["policy"] = pccp.Policy(_weights(_rng(seed, 3)))
        if kind == "host":
            # in place in host memory.  The contents of a failed store are
            # unspecified, so the batch is made of those that hold (the root
            # does), repeated to its size; a pass over them again moves the
            # same bytes and leaves the same fixed points
            n = case["stores"]
            closed = stores.clone()
            status, _ = pccp.propagate(model, closed[0], closed[1])
            holds = (status == pccp.PCCP_FIXPOINT).nonzero().flatten()
            stores = stores[:, holds[torch.arange(n, device=holds.device) % holds.numel()]]
            s["lb"], s["ub"] = (x.cpu().pin_memory() for x in stores)
            s["status"] = torch.empty(n, dtype=torch.int32, pin_memory=True)
            s["iterations"] = torch.empty(n, dtype=torch.int32, pin_memory=True)
        else:
            s["stores"], s["depth"] = stores, depth
        return s
    if kind == "search":
        g = _rng(seed, 1)
        s["models"] = [pccp.Model.from_rcpsp(Instance(int(g.integers(case["low"], case["high"] + 1)), g))
                       for _ in range(case["models"])]
        s["most"] = case["high"]
        s["strategy"], s["nodes"] = STRATEGY[case["strategy"]], case["nodes"]
        s["policy"] = pccp.Policy(_weights(_rng(seed, 3))) if case["strategy"] == "learned" else None
        return s
    if kind == "proof":
        # optima by the sequential search, then the same models with the
        # makespan below them
        g = _rng(seed, 1)
        sizes = g.integers(case["low"], case["high"] + 1, case["models"])
        insts = [Instance(int(n), g) for n in sizes]
        rows = [pccp.rcpsp.build_rows(i) for i in insts]
        models = [pccp.Model.from_rows(r) for r in rows]
        found = pccp.solve_batch(models, strategy=pccp.PCCP_FIRST_FAIL, node_limit=PROOF_NODES)
        below = []
        for r, f in zip(rows, found):
            # without a proved optimum nothing is left to search: makespan 0
            proved = f["status"] == pccp.PCCP_RES_OPTIMAL
            r["ub0"][r["objective"]] = f["objective"] - 1 if proved else 0
            below.append(pccp.Model.from_rows(r))
        s["models"] = below
        s["batch"] = pccp.Batch(below)
        return s
    w, f, off, target = _train_inputs(case, seed)
    s["policy"] = pccp.Policy(w)
    s["f"], s["off"], s["target"] = (torch.from_numpy(x).cuda() for x in (f, off, target))
    return s


# --------------------------------------------------------------------- runs

def _table(results, names):
    return {k: np.array([int(r[k]) for r in results], dtype=np.int64) for k in names}


def run(s):
    kind = s["kind"]
    if kind == "propagate":
        stores = s["stores"].clone()  # propagation is in place
        status, _ = pccp.propagate(s["model"], stores[0], stores[1])
        # a failed store's contents are unspecified
        stores.masked_fill_((status != pccp.PCCP_FIXPOINT)[None, :, None], 0)
        return {"status": status, "stores": stores}
    if kind == "host":
        pccp.propagate_host(s["model"], s["lb"], s["ub"], s["status"], s["iterations"])
        return {"status": s["status"], "lb": s["lb"], "ub": s["ub"]}
    if kind == "search":
        if len(s["models"]) == 1:
            r = [pccp.solve(s["models"][0], strategy=s["strategy"], node_limit=s["nodes"],
                            policy=s["policy"])]
        else:
            r = pccp.solve_batch(s["models"], strategy=s["strategy"], node_limit=s["nodes"],
                                 policy=s["policy"])
        out = _table(r, ("status", "has_solution", "nodes", "fails", "solutions", "max_depth"))
        out["objective"] = np.array([r_["objective"] if r_["has_solution"] else -1 for r_ in r])
        # the starts (the other variables follow from them), -1 without a solution
        out["starts"] = np.full((len(r), s["most"]), -1)
        for i, (m, r_) in enumerate(zip(s["models"], r)):
            if r_["has_solution"]:
                out["starts"][i, :len(m.branch)] = r_["witness"][m.branch]
        return out
    if kind == "proof":
        # no solution lies below the bound, so the trees are the same in any order
        s["batch"].solve_async(strategy=pccp.PCCP_FIRST_FAIL, deterministic=False)
        return _table(s["batch"].results(), ("status", "has_solution", "nodes", "fails",
                                             "solutions"))
    if kind == "rank":
        f = pccp.policy_features(s["model"], s["stores"][0], s["stores"][1], s["depth"])
        return {"features": f, "scores": s["policy"].score(f.reshape(-1, FEATURES))}
    loss = s["policy"].train_step(s["f"], s["off"], s["target"], lr=2e-3)
    return {"loss": np.array([loss], dtype=np.float32), "weights": _arrays(s["policy"].weights()),
            "gradients": _arrays(s["policy"].gradients())}


def _arrays(w):
    # without b3: it moves every candidate's score alike, so its gradient is
    # rounding alone
    return {k: v for k, v in w.items() if k != "b3"}


# --------------------------------------------------------------------- work

def _rows(n):
    """Operands of one evaluation of every row of an n-task model: two for a
    precedence, three for an overlap, one for each term of a resource row."""
    resources = 1 if n < 10 else 4
    return 2 * (0.05 * n * n + n) + 3 * n * (n - 1) + resources * n * n * (1.0 if n < 10 else 0.83)


def work(case):
    kind = case["kind"]
    if kind in ("propagate", "host"):
        n = case["tasks"]
        cells = case["stores"] * (n * n + n + 1)
        # bounds read and written once, one status; every row evaluated once
        return {"bytes": 16 * cells + 4 * case["stores"], "flops": 2 * case["stores"] * _rows(n)}
    if kind == "search":
        n = (case["low"] + case["high"]) / 2
        nodes = case["models"] * (case["nodes"] or 60)
        # each table and root box once, each witness once; every row once a node
        return {"bytes": case["models"] * (4 * _rows(n) + 12 * (n * n + n)),
                "flops": 2 * nodes * _rows(n)}
    if kind == "proof":
        n = (case["low"] + case["high"]) / 2
        # trees of a thousand nodes are ordinary
        return {"bytes": case["models"] * (4 * _rows(n) + 12 * (n * n + n)),
                "flops": 2 * case["models"] * 1000 * _rows(n)}
    net = 2 * (FEATURES * HIDDEN + HIDDEN * HIDDEN + HIDDEN)
    if kind == "rank":
        n, rows = case["tasks"], case["stores"] * case["tasks"]
        # the bounds of the starts and of the makespan, features out, scores out
        return {"bytes": 8 * case["stores"] * (n + 1) + rows * 4 * (FEATURES + 1),
                "flops": rows * net}
    rows = GROUP * case["groups"]
    params = HIDDEN * (FEATURES + HIDDEN + 3) + 1
    # features and targets in; parameters, both moments and gradients
    return {"bytes": rows * 4 * (FEATURES + 1) + 4 * 7 * params, "flops": 3 * rows * net}


# -------------------------------------------------------------------- exact

def _forward(w, f):
    w = {k: np.asarray(v, dtype=np.float64) for k, v in w.items()}
    h1 = np.maximum(f @ w["w1"].T + w["b1"], 0)
    h2 = np.maximum(h1 @ w["w2"].T + w["b2"], 0)
    return w, h1, h2, h2 @ w["w3"] + w["b3"]


def _exact_features(case, seed):
    inst = Instance(case["tasks"], _rng(seed, 1))
    n, h, count = inst.n, inst.horizon, case["stores"]
    r = _nodes(inst, count, _rng(seed, 2))
    lb, ub = np.zeros((count, n)), np.full((count, n), float(h))
    lb[r[:, 0], r[:, 1]], ub[r[:, 0], r[:, 1]] = r[:, 2], r[:, 3]
    depth = np.bincount(r[:, 0], minlength=count).astype(np.float64)
    after, before, d = np.ones(n), np.zeros(n), np.array(inst.durations, dtype=np.float64)
    for i, j in inst.precedences:  # every task also precedes the makespan
        after[i] += 1
        before[j] += 1
    demand = sum(np.array(u, dtype=np.float64) / c for u, c in zip(inst.usage, inst.capacity))
    f = np.empty((count, n, FEATURES))
    f[..., 0], f[..., 1], f[..., 2] = lb / (h + 1), ub / (h + 1), (ub - lb) / (h + 1)
    f[..., 3] = np.log2(1 + ub - lb) / 16
    f[..., 4], f[..., 5], f[..., 6] = after / 8, after * d / (h + 1), before / 8
    f[..., 7] = 2 * (n - 1) / 64
    f[..., 8] = demand / 4
    f[..., 9] = np.arange(n) / n
    f[..., 10] = (depth / (depth + 32))[:, None]
    f[..., 11] = 0  # the makespan's lower bound is still the root's
    return f


def exact(case, seed):
    if case["kind"] == "rank":
        f = _exact_features(case, seed)
        return {"features": f, "scores": _forward(_weights(_rng(seed, 3)), f.reshape(-1, FEATURES))[3]}
    if case["kind"] != "train":
        return None
    w, f, off, target = _train_inputs(case, seed)
    f, target = f.astype(np.float64), target.astype(np.float64)
    w, h1, h2, s = _forward(w, f)
    groups = len(off) - 1
    ds, loss = np.empty_like(s), 0.0
    for a, b in zip(off[:-1], off[1:]):
        z = s[a:b] - s[a:b].max()
        log_p = z - np.log(np.exp(z).sum())
        loss -= (target[a:b] * log_p).sum() / groups
        ds[a:b] = (np.exp(log_p) - target[a:b]) / groups
    d2 = (h2 > 0) * ds[:, None] * w["w3"]
    d1 = (h1 > 0) * (d2 @ w["w2"])
    grad = {"w1": d1.T @ f, "b1": d1.sum(0), "w2": d2.T @ h1, "b2": d2.sum(0), "w3": h2.T @ ds}
    # Adam's first step: the moments' corrections cancel
    new = {k: w[k] - 2e-3 * g / (np.abs(g) + 1e-8) for k, g in grad.items()}
    return {"loss": np.array([loss]), "weights": new, "gradients": grad}
