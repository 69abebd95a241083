"""The general kernels (intervals, no mask form) on scheduling models: bool_store
-1 keeps the Booleans as intervals, so the default launch of every call is
theirs.  And the mask searches with many small slots, whose rings hold fewer
fixed points than the path is deep."""
import numpy as np
import pytest

import oracle
from oracle.rcpsp import rcpsp_model
import paper_2207_12116_gb300 as pccp
from synthetic import config_instance, draw_partial_assignments
from tests.gpu_util import compare_batch
from tests.test_gpu_mask import instance
from tests.test_gpu_solve import same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def intervals(inst):
    m = pccp.Model.from_rcpsp(inst, bool_store=-1)
    assert m.info.bool_vars == 0
    return m


@pytest.mark.parametrize("family, count", [("tiny8", 200), ("j30", 200), ("j120", 12)])
@pytest.mark.parametrize("kw", [{}, {"skip_stable": False}, {"skip_stable": True}])
def test_propagation(family, count, kw):
    inst = config_instance(family, 1)
    om, rows, m = rcpsp_model(inst), pccp.rcpsp.build_rows(inst), intervals(inst)
    lb, ub = pccp.rcpsp.node_stores(rows, draw_partial_assignments(inst.n, inst.horizon, count, seed=5))
    dlb, dub = torch.from_numpy(lb).cuda(), torch.from_numpy(ub).cuda()
    st, _ = pccp.propagate(m, dlb, dub, config=pccp.launch_config(**kw) if kw else None)
    compare_batch(om, lb, ub, st.cpu().numpy(), dlb.cpu().numpy(), dub.cpu().numpy())


@pytest.mark.parametrize("kw", [{}, {"teams_per_cta": 4, "threads": 64}, {"teams_per_cta": 3, "threads": 256}])
def test_batched_search(kw):
    insts = [config_instance("tiny8", s) for s in range(6)] + [config_instance("mixed30_60", s) for s in range(4)]
    res = pccp.solve_batch([intervals(i) for i in insts], strategy=pccp.PCCP_FIRST_FAIL, node_limit=60, **kw)
    for inst, r in zip(insts, res):
        same(r, oracle.solve(rcpsp_model(inst), strategy=oracle.FIRST_FAIL, node_limit=60))


@pytest.mark.parametrize("donate", [0, 1])
def test_parallel_search(donate):
    insts = [config_instance("tiny8", s) for s in range(8)]
    oms, models = [rcpsp_model(i) for i in insts], [intervals(i) for i in insts]
    best = [oracle.solve(om) for om in oms]
    for r, o in zip(pccp.solve_batch(models, deterministic=False, donate_nodes=donate), best):
        assert r["status"] == pccp.PCCP_RES_OPTIMAL and r["objective"] == o["objective"]
    for m, om, o in zip(models, oms, best):
        p = oracle.solve(om, obj_ub=o["objective"] - 1)
        r = pccp.solve(m, obj_ub=o["objective"] - 1, deterministic=False, donate_nodes=donate)
        assert (r["status"], r["nodes"], r["fails"]) == (pccp.PCCP_RES_INFEASIBLE, p["nodes"], p["fails"])


@pytest.mark.parametrize("teams", [1, 3, 5, 15])
def test_many_small_slots_of_the_mask_search(teams):
    insts = [instance(20, seed=s) for s in range(6)] + [instance(n) for n in (2, 3, 17)]
    res = pccp.solve_batch([pccp.Model.from_rcpsp(i) for i in insts], node_limit=300, threads=32,
                           teams_per_cta=teams)
    for inst, r in zip(insts, res):
        same(r, oracle.solve(rcpsp_model(inst), node_limit=300))
    if teams == 15:  # of a fifteenth of 227 KB: no room for as many stores as the path is deep
        store = 8 * (21 + 20 * 19 // 32) + 4 * (20 * 19 // 32)
        assert max(r["max_depth"] for r in res[:6]) > 227 * 1024 // 15 // store


def test_a_16th_team_is_refused():
    models = [pccp.Model.from_rcpsp(config_instance("tiny8", s)) for s in range(3)]
    for deterministic in (True, False):
        with pytest.raises(pccp.PccpError) as e:
            pccp.solve_batch(models, threads=32, teams_per_cta=16, deterministic=deterministic)
        assert e.value.code == pccp.PCCP_ERR_INVALID
