"""Rows that a mask search reports as evaluated where the temporal rows have a cycle:
one warp of a team runs them, and they count once whatever the team's size."""
import pytest

import oracle
import paper_2207_12116_gb300 as pccp
from tests.test_gpu_solve import same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_temporal_rows_count_once():
    # three intervals in a cycle of temporal rows, one Boolean in one row
    lb0, ub0 = [0] * 4, [6, 6, 6, 1]
    temporal, linear = [(0, 1, 1), (1, 2, 1), (2, 0, -4)], [(1, [(1, 3)])]
    m = pccp.Model.from_lists(lb0, ub0, temporal, linear, (), 2, [0, 1, 2])
    o = oracle.solve(oracle.Model(lb0, ub0, temporal, linear, (), 2, [0, 1, 2]))
    runs = [pccp.solve(m, threads=t) for t in (32, 64, 256, 512)]
    for r in runs:
        same(r, o)
    assert len({r["rows_evaluated"] for r in runs}) == 1
