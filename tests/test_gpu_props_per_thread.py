"""Batched searches whose team size follows from props_per_thread, with numbers
of teams a CTA that do not divide its threads into whole warps: the oracle's
counts, for models in mask form and with interval stores."""
import pytest

import oracle
from oracle.rcpsp import rcpsp_model
import paper_2207_12116_gb300 as pccp
from tests.test_gpu_mask import instance
from tests.test_gpu_solve import same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bool_store", [0, -1])
@pytest.mark.parametrize("teams", [3, 5, 6, 7])
def test_team_sizes_from_rows(bool_store, teams):
    insts = [instance(n, seed=s) for n in (17, 18) for s in range(2 * teams)]
    models = [pccp.Model.from_rcpsp(i, bool_store=bool_store) for i in insts]
    assert min(m.rows for m in models) > 1024 // 3  # more rows than a team may have threads
    for per in (1, 8):
        res = pccp.solve_batch(models, strategy=pccp.PCCP_FIRST_FAIL, node_limit=60,
                               teams_per_cta=teams, props_per_thread=per)
        for inst, r in zip(insts, res):
            same(r, oracle.solve(rcpsp_model(inst), node_limit=60, strategy=oracle.FIRST_FAIL))
