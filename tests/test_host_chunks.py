"""The default chunks of host-memory propagation of models in mask form: whole
multiples of 64 stores, several to a batch of large page-locked stores; and batches
around a chunk's edges give the device call's results."""
import os
import subprocess

import pytest

import paper_2207_12116_gb300 as pccp
from synthetic import draw_partial_assignments

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "launch_rules.h"
int main() {
  for (long long vars : {1ll, 73ll, 931ll, 1641ll, 3661ll, 14521ll, 65535ll})
    for (int sms : {1, 8, 148, 152})
      for (int locked : {0, 1})
        std::printf("%lld %d %d %lld\n", vars, sms, locked,
                    static_cast<long long>(pccp::host_chunk_unit(8 * vars, sms, locked)));
}
"""


def test_units(tmp_path):
    (tmp_path / "unit.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2207_12116_gb300", "csrc"),
                    str(tmp_path / "unit.cc"), "-o", str(tmp_path / "unit")], check=True)
    out = subprocess.run([str(tmp_path / "unit")], check=True, capture_output=True, text=True).stdout
    units = {tuple(int(x) for x in line.split()[:3]): int(line.split()[3]) for line in out.splitlines()}
    assert len(units) == 7 * 4 * 2
    for (vars_, sms, locked), unit in units.items():
        assert unit % 64 == 0 and 64 <= unit <= max(64, 8 * sms)
        assert not locked or unit == 64 or 8 * vars_ * unit <= 12 << 20
    assert units[931, 152, 1] == 1216 and units[3661, 152, 0] == 1216
    # 1,216 stores of 60 tasks: several chunks when their copies can overlap
    assert units[3661, 152, 1] <= 1216 // 3


@pytest.mark.gpu
@pytest.mark.parametrize("locked", [True, False])
@pytest.mark.parametrize("stores", [63, 64, 65, 383, 384, 385, 1300])
def test_batches_around_a_chunk(locked, stores):
    from tests.test_gpu_mask import instance
    inst = instance(60)
    rows = pccp.rcpsp.build_rows(inst)
    m = pccp.Model.from_rows(rows)
    lb, ub = (torch.from_numpy(x) for x in pccp.rcpsp.node_stores(
        rows, draw_partial_assignments(inst.n, inst.horizon, stores, seed=stores)))
    dlb, dub = lb.cuda(), ub.cuda()
    st, _ = pccp.propagate(m, dlb, dub)
    hlb, hub = (lb.pin_memory(), ub.pin_memory()) if locked else (lb.clone(), ub.clone())
    hst, _ = pccp.propagate_host(m, hlb, hub)
    assert torch.equal(hst, st.cpu())
    fx = hst == pccp.PCCP_FIXPOINT
    assert fx.any() and torch.equal(hlb[fx], dlb.cpu()[fx]) and torch.equal(hub[fx], dub.cpu()[fx])
