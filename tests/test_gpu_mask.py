"""Models whose Booleans are evaluated as bit masks: the overlap Booleans of a
resource column share words, their reified rows run a word at a time and
their resource rows from coefficient planes.  The layout changes with the
number of tasks (columns packed into one word, one column a word, a word and a
rest, several words) and with the largest coefficient (one or more quads of
planes); fixed points, statuses and searches equal the oracle's at the edges of
each, in one- and many-warp teams, and where a model falls back to intervals."""
import numpy as np
import pytest

import oracle
from oracle.rcpsp import rcpsp_model
import paper_2207_12116_gb300 as pccp
from synthetic import SplitMix64, draw_partial_assignments
from synthetic.rcpsp import RcpspDistribution, draw_rcpsp
from tests.gpu_util import compare_batch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SMALL, WIDE, HUGE = (0, 5), (0, 20), (0, 300)  # demands: one, two and three quads of planes


def instance(n, demand=SMALL, resources=3, seed=0):
    cap = (demand[1], 2 * demand[1])
    return draw_rcpsp(RcpspDistribution(n, n, resources, (1, 9), demand, cap, 0.12), 1000 * n + seed)


def check(inst, count, seed, cfgs):
    om = rcpsp_model(inst)
    rows = pccp.rcpsp.build_rows(inst)
    m = pccp.Model.from_rows(rows)
    lb, ub = pccp.rcpsp.node_stores(rows, [[]] + draw_partial_assignments(inst.n, inst.horizon,
                                                                          count, seed=seed))
    # Boolean inputs of every kind: fixed, empty, outside {0, 1}
    g = SplitMix64.derive(seed, 3)
    for r in range(0, len(lb), 3):
        v = inst.n + g.uniform_int(0, inst.n * inst.n - 1)
        lb[r, v], ub[r, v] = ((1, 1), (0, 0), (2, 3), (-3, -1), (-3, 5))[g.uniform_int(0, 4)]
    for cfg in cfgs:
        dlb, dub = torch.from_numpy(lb).cuda(), torch.from_numpy(ub).cuda()
        st, _ = pccp.propagate(m, dlb, dub, config=cfg)
        torch.cuda.synchronize()
        compare_batch(om, lb, ub, st.cpu().numpy(), dlb.cpu().numpy(), dub.cpu().numpy())


@pytest.mark.parametrize("n", [2, 3, 10, 11, 16, 17, 31, 32, 33, 45, 64, 65, 97])
def test_word_layouts(n):
    cfgs = [None, pccp.launch_config(32, 3), pccp.launch_config(64, 2, temporal_levels=False),
            pccp.launch_config(512, 1)]
    check(instance(n), 40 if n < 60 else 12, n, cfgs)


@pytest.mark.parametrize("n, demand", [(9, WIDE), (33, WIDE), (40, HUGE), (64, HUGE)])
def test_coefficient_planes(n, demand):
    check(instance(n, demand), 24, n, [None, pccp.launch_config(32, 1)])


def test_unaligned_stores_and_work_report():
    """Rows of stores that start at every 16-byte offset, lb and ub apart by
    other offsets, and a work report of at least one evaluation of every row of a
    store that holds."""
    inst = instance(21)
    om, rows = rcpsp_model(inst), pccp.rcpsp.build_rows(inst)
    m = pccp.Model.from_rows(rows)
    lb, ub = pccp.rcpsp.node_stores(rows, draw_partial_assignments(inst.n, inst.horizon, 30, seed=2))
    n, nv = lb.shape
    for a, b in ((0, 0), (1, 1), (1, 2), (3, 0)):
        flat = torch.zeros(2, n * nv + 8, dtype=torch.int32, device="cuda")
        dlb, dub = flat[0, a:a + n * nv].view(n, nv), flat[1, b:b + n * nv].view(n, nv)
        dlb.copy_(torch.from_numpy(lb))
        dub.copy_(torch.from_numpy(ub))
        work = torch.zeros((n, 2), dtype=torch.int32, device="cuda")
        st, _ = pccp.propagate(m, dlb, dub, work=work)
        st = st.cpu().numpy()
        compare_batch(om, lb, ub, st, dlb.cpu().numpy(), dub.cpu().numpy())
        assert (work.cpu().numpy()[st == 0, 0] >= m.rows).all()


def test_models_without_the_form():
    """A Boolean with two reified rows, and a linear row holding a variable
    twice, keep the general evaluation."""
    base = dict(lb0=[0, 0, 0, 0, 0, 0], ub0=[9, 9, 9, 1, 1, 1])
    for reified, linear in (([(3, 0, 1, 2), (3, 1, 2, 3), (4, 0, 2, 2)], [(2, [(1, 3), (2, 4), (1, 5)])]),
                            ([(3, 0, 1, 2), (4, 0, 2, 2)], [(2, [(1, 3), (1, 3), (2, 4)])])):
        m = pccp.Model.from_lists(temporal=[(0, 1, 1)], reified=reified, linear=linear, **base)
        om = oracle.Model(base["lb0"], base["ub0"], [(0, 1, 1)], linear, reified)
        g = SplitMix64(7)
        lb = np.array([[g.uniform_int(0, 4) for _ in range(3)] + [0, 0, 0] for _ in range(64)], np.int32)
        ub = np.array([[g.uniform_int(3, 9) for _ in range(3)] + [1, g.uniform_int(0, 1), 1]
                       for _ in range(64)], np.int32)
        dlb, dub = torch.from_numpy(lb).cuda(), torch.from_numpy(ub).cuda()
        st, _ = pccp.propagate(m, dlb, dub)
        compare_batch(om, lb, ub, st.cpu().numpy(), dlb.cpu().numpy(), dub.cpu().numpy())
