"""The propagation kernel of the mask form when its table image never arrives:
the bounded wait gives up, nothing of the image is read, and every store is
reported as an error with its bounds untouched.  The kernel is built here with a
loader that fills the image with a pattern and reports that it gave up."""
import ctypes
import subprocess

import pytest

from paper_2207_12116_gb300 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "pccp_device.cuh"
namespace pccp {
__device__ bool late_image(uint8_t* dst, const uint8_t*, uint32_t bytes, uint64_t*, uint32_t) {
  for (uint32_t i = threadIdx.x; i < bytes; i += blockDim.x) dst[i] = 0x7f;
  __syncthreads();
  return false;
}
}
#define load_image late_image
#include "k_propagate_mask.cuh"

extern "C" int late(int n_stores, int n_vars, int team, int teams, int grid, int* lb, int* ub,
                    int* status, int* iters, int* work, int* counter) {
  pccp::PropArgs a{};
  a.lb = lb;
  a.ub = ub;
  a.status = status;
  a.iters = iters;
  a.work = work;
  a.counter = counter;
  a.image_bytes = 1024;
  a.n_vars = n_vars;
  a.n_stores = n_stores;
  a.team_size = team;
  a.teams = teams;
  a.max_iter = 100;
  a.track_words = 64;
  a.slot_bytes = 1024;
  a.levels = 1;
  const auto kern = team == 32 ? pccp::k_propagate_mask<true, 1024, 1> : pccp::k_propagate_mask<false, 1024, 1>;
  kern<<<grid, team * teams, 1024 + 16 + 1024 * teams>>>(a);
  if (cudaGetLastError() != cudaSuccess) return 1;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-I", build.CSRC, str(d / "late.cu"), "-o", str(d / "late.so")], check=True)
    return ctypes.CDLL(str(d / "late.so"))


@pytest.mark.parametrize("team", [32, 64, 512])
@pytest.mark.parametrize("stores, grid, taken", [(3, 3, False), (700, 5, True)])
def test_stores_are_reported(lib, team, stores, grid, taken):
    teams, n_vars = 2, 9
    bounds = torch.arange(2 * stores * n_vars, dtype=torch.int32, device="cuda").view(2, stores, n_vars)
    before = bounds.clone()
    report = torch.full((4, stores), -7, dtype=torch.int32, device="cuda")
    counter = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = lib.late(stores, n_vars, team, teams, grid,
                  *(ctypes.c_void_p(t.data_ptr()) for t in (bounds[0], bounds[1], report[0], report[1],
                                                            report[2])),
                  ctypes.c_void_p(counter.data_ptr() if taken else 0))
    assert rc == 0
    assert (report[0] == 2).all() and (report[1:] == 0).all()
    assert torch.equal(bounds, before)
