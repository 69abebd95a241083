"""Loops that a call asks for by name run also on models in mask form: the
eventless loop (skip_stable off: every row in every iteration), change tracking
(skip_stable on) and the two orders of the temporal rows in searches, through
every entry point; results stay the oracle's."""
import pytest

import oracle
from oracle.rcpsp import rcpsp_model
import paper_2207_12116_gb300 as pccp
from synthetic import config_instance, draw_partial_assignments
from tests.gpu_util import compare_batch
from tests.test_gpu_solve import same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# every row in every iteration (tables that fit shared memory are not tracked by default)
EVERY_ROW = [{"skip_stable": False}, {"temporal_levels": True}, {"temporal_levels": False}]


def every_row(m, r):
    return r["rows_evaluated"] == r["iterations"] * m.rows


@pytest.mark.parametrize("seed", range(3))
def test_eventless_propagation(seed):
    inst = config_instance("j30", seed)
    om, rows = rcpsp_model(inst), pccp.rcpsp.build_rows(inst)
    m = pccp.Model.from_rows(rows)
    lb, ub = pccp.rcpsp.node_stores(rows, draw_partial_assignments(inst.n, inst.horizon, 60, seed=seed))
    dlb, dub = torch.from_numpy(lb).cuda(), torch.from_numpy(ub).cuda()
    work = torch.zeros((len(lb), 2), dtype=torch.int32, device="cuda")
    st, it = pccp.propagate(m, dlb, dub, work=work, config=pccp.launch_config(skip_stable=False))
    st, it, work = (t.cpu().numpy() for t in (st, it, work))
    compare_batch(om, lb, ub, st, dlb.cpu().numpy(), dub.cpu().numpy())
    assert (work[:, 0] == it * m.rows)[st == pccp.PCCP_FIXPOINT].all()


@pytest.mark.parametrize("kw", EVERY_ROW)
def test_searches(kw):
    insts = [config_instance("tiny8", s) for s in range(5)]
    oms, models = [rcpsp_model(i) for i in insts], [pccp.Model.from_rcpsp(i) for i in insts]
    want = [oracle.solve(om) for om in oms]
    batch = pccp.Batch(models)
    batch.solve_async(**kw)
    runs = [pccp.solve(m, **kw) for m in models], pccp.solve_batch(models, **kw), batch.results(), \
        pccp.solve_batch(models, noalloc=True, **kw)
    for res in runs:
        for m, o, r in zip(models, want, res):
            same(r, o)
            assert every_row(m, r)
    batch.solve_async(deterministic=False, **kw)
    for m, o, r in zip(models, want, batch.results()):
        assert r["objective"] == o["objective"] and every_row(m, r)
    for m, o in zip(models, want):
        r = pccp.solve(m, deterministic=False, **kw)
        assert r["objective"] == o["objective"] and every_row(m, r)
    # and the default again, on the same batch
    batch.solve_async()
    for o, r in zip(want, batch.results()):
        same(r, o)


def test_change_tracking_in_a_batch():
    """One-warp teams, whose loop has one order: the batch's counts are those of the
    same models kept as intervals, which have no other form."""
    insts = [config_instance("tiny8", s) for s in range(7)]
    runs = []
    for store in (0, -1):
        models = [pccp.Model.from_rcpsp(i, bool_store=store) for i in insts]
        batch = pccp.Batch(models, threads=32, teams_per_cta=2)
        batch.solve_async(skip_stable=True)
        runs.append(batch.results())
    for inst, a, b in zip(insts, *runs):
        same(a, oracle.solve(rcpsp_model(inst)))
        assert (a["iterations"], a["rows_evaluated"]) == (b["iterations"], b["rows_evaluated"])
