"""A team's wait for an item of the shared queue, with the limit set to 50 ms:
the wait of either search ends with an error and the stop flag when an item is
reserved and never published, and when a busy team never reports progress; an
item that is there is claimed, and an empty queue without busy teams is the end."""
import ctypes
import subprocess

import pytest

from paper_2207_12116_gb300 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAM = r"""
#define PCCP_QUEUE_WAIT_NS 50000000ull
#include <cuda_runtime.h>
#include <climits>
#include <cstdint>
namespace {
struct InstanceDesc;
struct PolicyDev;
#include "queue_ring.inc"

__global__ void k_wait(QArgs a, int which, long long* out) {
  unsigned long long pos = 0;
  int model = -1, len = -1;
  out[0] = which ? mq_wait_item(a, &pos, &model, &len) : q_wait_item(a, &pos, &model, &len);
  out[1] = static_cast<long long>(pos);
  out[2] = model;
  out[3] = len;
  out[4] = static_cast<long long>(a.g->head);
  out[5] = a.g->busy;
  out[6] = a.g->stop;
  out[7] = a.g->error;
}
}  // namespace

// g: head, tail, t0, progress, {busy, stop}, {error, limited}, donations; seq[4]; hdr[4]
extern "C" int wait_item(int which, void* g, void* seq, void* hdr, long long* out) {
  static_assert(sizeof(QGlobal) == 56, "the queue's state");
  QArgs a{};
  a.g = static_cast<QGlobal*>(g);
  a.seq = static_cast<unsigned long long*>(seq);
  a.hdr = static_cast<int2*>(hdr);
  a.cap = 4;
  a.n_teams = 2;
  k_wait<<<1, 1>>>(a, which, out);
  if (cudaGetLastError() != cudaSuccess) return 1;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("wait")
    (d / "wait.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-I", build.CSRC, str(d / "wait.cu"), "-o", str(d / "wait.so")], check=True)
    return ctypes.CDLL(str(d / "wait.so"))


CASES = {  # head, tail, busy, published -> claimed, head, busy, stop, error
    "reserved, never published": ((0, 1, 0, False), (0, 0, 0, 1, 4)),
    "a busy team without progress": ((2, 2, 1, False), (0, 2, 1, 1, 4)),
    "an item": ((0, 1, 0, True), (1, 1, 1, 0, 0)),
    "the end": ((3, 3, 0, False), (0, 3, 0, 0, 0)),
}


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("case", sorted(CASES))
def test_wait(lib, which, case):
    (head, tail, busy, published), want = CASES[case]
    # slots of the ring below head have been through a round, the others are free
    seq = [k + 4 if k < head else k for k in range(4)]
    if published:
        seq[head] = head + 1
    g = torch.tensor([head, tail, 0, 0, busy, 0, 0], dtype=torch.int64, device="cuda")
    dseq = torch.tensor(seq, dtype=torch.int64, device="cuda")
    hdr = torch.tensor([[5, 7]] * 4, dtype=torch.int32, device="cuda")
    out = torch.zeros(8, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    rc = lib.wait_item(which, *(ctypes.c_void_p(t.data_ptr()) for t in (g, dseq, hdr, out)))
    assert rc == 0
    have, pos, model, length, now_head, now_busy, stop, error = out.cpu().numpy()
    assert (have, now_head, now_busy, stop, error) == want
    if have:
        assert (pos, model, length) == (head, 5, 7)
