"""The team size of a solve of one model: any number below one leaves it to the
library, also for models in mask form."""
import pytest

import oracle
from oracle.rcpsp import rcpsp_model
import paper_2207_12116_gb300 as pccp
from synthetic import config_instance
from tests.test_gpu_solve import same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", [0, -1])
@pytest.mark.parametrize("threads", [0, -1, -32])
def test_no_team_size(store, threads):
    inst = config_instance("tiny8", 3)
    m = pccp.Model.from_rcpsp(inst, bool_store=store)
    same(pccp.solve(m, threads=threads), oracle.solve(rcpsp_model(inst)))
