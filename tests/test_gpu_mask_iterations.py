"""Iterations of the mask form where the rows clear Booleans of words that no
reified row has: what shared memory held before the launch does not count."""
import numpy as np
import pytest

import oracle
import paper_2207_12116_gb300 as pccp
from tests.gpu_util import compare_batch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ones():
    """Shared memory of every SM full of set bits: stores of wide intervals from -1 on."""
    wide = pccp.Model.from_lists([-1] * 26000, [(1 << 30) - 1] * 26000)
    n = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    lb = torch.full((n, 26000), -1, dtype=torch.int32, device="cuda")
    ub = torch.full_like(lb, (1 << 30) - 1)

    def fill():
        st, _ = pccp.propagate(wide, lb, ub)
        assert (st == pccp.PCCP_FIXPOINT).all()
    return fill


@pytest.mark.parametrize("free", [40, 64, 200])
@pytest.mark.parametrize("team", [0, 32, 64, 512])
def test_rows_over_free_booleans(ones, free, team):
    # intervals 0 and 1, a reified Boolean 2, and free Booleans in one row that
    # allows a single one of them
    lb0, ub0 = [0, 0] + [0] * (1 + free), [9, 9] + [1] * (1 + free)
    reified = [(2, 0, 1, 3)]
    linear = [(1, [(1, 3 + k) for k in range(free)])]
    m = pccp.Model.from_lists(lb0, ub0, (), linear, reified)
    om = oracle.Model(lb0, ub0, (), linear, reified)
    lb, ub = np.tile(np.int32(lb0), (300, 1)), np.tile(np.int32(ub0), (300, 1))
    for r in range(300):
        lb[r, 3 + r % free] = 1  # the others become 0: nothing else follows
    for budget in (0, 1):
        ones()
        dlb, dub = torch.from_numpy(lb).cuda(), torch.from_numpy(ub).cuda()
        st, it = pccp.propagate(m, dlb, dub, config=pccp.launch_config(team, max_iterations=budget))
        assert (it.cpu().numpy() == 1).all()
        compare_batch(om, lb, ub, st.cpu().numpy(), dlb.cpu().numpy(), dub.cpu().numpy())
