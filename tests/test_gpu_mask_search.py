"""Searches of models in mask form: the team-per-model search and the shared
queue keep saved fixed points of the path in a ring and continue from them.
Counts, optima and witnesses equal the oracle's (the queue's on proof trees,
which no order changes) at the edges of the word layouts, for one- and many-warp
teams, with rings shorter than the path, for models without a path matrix (a
cycle of precedences), and where a shape leaves the search to intervals."""
import numpy as np
import pytest

import oracle
from oracle.rcpsp import rcpsp_model
import paper_2207_12116_gb300 as pccp
from tests.gpu_util import compare_batch
from tests.test_gpu_mask import HUGE, SMALL, WIDE, instance
from tests.test_gpu_solve import same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [2, 3, 10, 11, 17, 31, 32, 33, 45, 64, 65]


def proof(n, demand=SMALL):
    """An instance of n tasks (of a few), a bound below its optimum and the
    oracle's proof, the largest of at most `most` nodes."""
    best, most = None, 1500 if n < 31 else 400
    for seed in range(12 if n < 31 else 3):
        inst = instance(n, demand, seed=seed)
        om = rcpsp_model(inst)
        low = int(oracle.propagate(om, om.lb0, om.ub0)[1][om.objective])
        for ub in range(low - 1, low + 12):
            p = oracle.solve(om, obj_ub=ub, node_limit=most, strategy=oracle.FIRST_FAIL)
            if p["status"] != oracle.RES_INFEASIBLE:
                break
            if best is None or p["nodes"] > best[2]["nodes"]:
                best = inst, ub, p
    return best


@pytest.mark.parametrize("n", SIZES)
def test_sequential_order(n):
    inst = instance(n)
    om, m = rcpsp_model(inst), pccp.Model.from_rcpsp(inst)
    for strategy, ostrategy in ((pccp.PCCP_INPUT_ORDER, oracle.INPUT_ORDER),
                                (pccp.PCCP_FIRST_FAIL, oracle.FIRST_FAIL)):
        o = oracle.solve(om, node_limit=300, strategy=ostrategy)
        for threads in (0, 32, 96, 512, 1024):
            same(pccp.solve(m, node_limit=300, strategy=strategy, threads=threads), o)


@pytest.mark.parametrize("teams", [0, 4, 16])
def test_batch_of_all_layouts(teams):
    insts = [instance(n, d) for n in SIZES for d in (SMALL, WIDE, HUGE)]
    models = [pccp.Model.from_rcpsp(i) for i in insts]
    kw = {} if teams == 0 else {"teams_per_cta": teams, "threads": 32}
    try:
        res = pccp.solve_batch(models, node_limit=200, strategy=pccp.PCCP_FIRST_FAIL, **kw)
    except RuntimeError:
        assert teams == 16  # no shape holds so many teams of the largest model
        return
    for inst, r in zip(insts, res):
        same(r, oracle.solve(rcpsp_model(inst), node_limit=200, strategy=oracle.FIRST_FAIL))


@pytest.mark.parametrize("n", SIZES)
def test_parallel_proofs(n):
    inst, ub, p = proof(n)
    m = pccp.Model.from_rcpsp(inst)
    for kw in ({}, {"threads": 32, "donate_nodes": 1}, {"threads": 96}, {"threads": 512, "blocks": 3}):
        r = pccp.solve(m, obj_ub=ub, deterministic=False, strategy=pccp.PCCP_FIRST_FAIL, **kw)
        assert r["status"] == pccp.PCCP_RES_INFEASIBLE
        assert (r["nodes"], r["fails"], r["solutions"]) == (p["nodes"], p["fails"], 0)


@pytest.mark.parametrize("kw", [{}, {"teams_per_cta": 2, "threads": 64}, {"threads": 32, "donate_nodes": 1}])
def test_parallel_batch_proofs(kw):
    """Copies of two models with proofs of some size, one bound for both, among
    small models that the bound may leave a solution."""
    (big, ub, p), (wide, _, _) = proof(17), proof(17, HUGE)
    insts = [big] * 4 + [wide] + [instance(n, d, seed=s) for n in (2, 9, 10) for d in (SMALL, HUGE)
                                  for s in range(3)]
    res = pccp.solve_batch([pccp.Model.from_rcpsp(i) for i in insts], obj_ub=ub, deterministic=False,
                           strategy=pccp.PCCP_FIRST_FAIL, node_limit=200000, **kw)
    for k, (inst, r) in enumerate(zip(insts, res)):
        o = p if k < 4 else oracle.solve(rcpsp_model(inst), obj_ub=ub, node_limit=50000,
                                         strategy=oracle.FIRST_FAIL)
        if o["status"] == oracle.RES_INFEASIBLE:
            assert (r["nodes"], r["fails"], r["solutions"]) == (o["nodes"], o["fails"], 0)
        elif o["status"] == oracle.RES_OPTIMAL:
            assert r["objective"] == o["objective"]


@pytest.mark.parametrize("n", [9, 33])
def test_learned_search_from_saved_fixed_points(n):
    """The learned order, by a plain solve and by a batch, spans the same tree at
    every team size, and its optimum is the oracle's where it completes."""
    inst = instance(n)
    om, m, pol = rcpsp_model(inst), pccp.Model.from_rcpsp(inst), pccp.Policy.random(3)
    runs = [pccp.solve(m, strategy=pccp.PCCP_LEARNED, policy=pol, node_limit=400, threads=t)
            for t in (0, 32, 128, 512)]
    runs += pccp.solve_batch([m, m], strategy=pccp.PCCP_LEARNED, policy=pol, node_limit=400)
    assert len({(r["nodes"], r["fails"], r["solutions"], r["objective"]) for r in runs}) == 1
    if runs[0]["status"] == pccp.PCCP_RES_OPTIMAL:
        assert runs[0]["objective"] == oracle.solve(om)["objective"]


def cyclic(seed):
    """Start times within a cycle of precedences, overlap Booleans and one
    resource: no path matrix."""
    n, d = 5, [2, 3, 1, 2, 3]
    lb0, ub0 = [0] * (n + 1) + [0] * (n * n), [12] * (n + 1) + [1] * (n * n)
    temporal = [(0, 1, 1), (1, 2, 1), (2, 0, -9 + seed % 3)] + [(i, n, d[i]) for i in range(n)]
    reified = [(n + 1 + n * i + j, i, j, d[i]) for i in range(n) for j in range(n) if i != j]
    use = [1 + (seed + i) % 3 for i in range(n)]
    linear = [(4 - use[j], [(use[i], n + 1 + n * i + j) for i in range(n) if i != j]) for j in range(n)]
    return lb0, ub0, temporal, linear, reified, n, list(range(n))


@pytest.mark.parametrize("seed", range(4))
def test_cycle_of_precedences(seed):
    lb0, ub0, temporal, linear, reified, objective, branch = cyclic(seed)
    m = pccp.Model.from_lists(lb0, ub0, temporal, linear, reified, objective, branch)
    om = oracle.Model(lb0, ub0, temporal, linear, reified, objective, branch)
    o = oracle.solve(om)
    same(pccp.solve(m), o)
    same(pccp.solve(m, threads=64), o)
    c = oracle.solve(om, mode=oracle.COUNT_ALL, obj_ub=o["objective"])
    r = pccp.solve(m, mode=pccp.PCCP_COUNT_ALL, obj_ub=o["objective"], deterministic=False, donate_nodes=1)
    assert (r["nodes"], r["fails"], r["solutions"]) == (c["nodes"], c["fails"], c["solutions"])


@pytest.mark.parametrize("sizes", [(40, 70), (33, 64), (64, 64), (96, 32, 31), (65, 1, 65)])
def test_groups_of_like_and_unlike_size(sizes):
    """Resource rows over groups of Booleans of several words: like groups'
    words lie side by side, unlike groups' one group after another."""
    g = np.random.default_rng(sum(sizes))
    n, k = 6, sum(sizes)
    lb0, ub0 = [0] * n + [0] * k, [9] * n + [1] * k
    pairs = [(int(a), int(b)) for a, b in (g.permutation(n)[:2] for _ in range(k))]
    reified = [(n + i, a, b, 1 + i % 4) for i, (a, b) in enumerate(pairs)]
    linear, at = [], 0
    for size in sizes:
        for _ in range(2):
            linear.append((size, [(int(g.integers(1, 6)), n + at + i) for i in range(size)]))
        at += size
    temporal = [(0, 1, 1), (2, 3, 2)]
    m = pccp.Model.from_lists(lb0, ub0, temporal, linear, reified)
    om = oracle.Model(lb0, ub0, temporal, linear, reified)
    lb, ub = np.tile(np.int32(lb0), (48, 1)), np.tile(np.int32(ub0), (48, 1))
    lb[:, :n] = g.integers(0, 5, (48, n))
    ub[:, :n] = lb[:, :n] + g.integers(0, 5, (48, n))
    dlb, dub = torch.from_numpy(lb).cuda(), torch.from_numpy(ub).cuda()
    st, _ = pccp.propagate(m, dlb, dub)
    compare_batch(om, lb, ub, st.cpu().numpy(), dlb.cpu().numpy(), dub.cpu().numpy())
