"""The bounded waits of pic_internal.cuh, as kernels of this test's own that include
it: what an aborting kernel waits for on its way out.  Nothing here faults: every
wait ends by its limit or by an arrival of the same kernel."""
import ctypes
import os
import subprocess
import time

import pytest
import torch

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2607_28069_gb300", "csrc")

SOURCE = r"""
#include "pic_internal.cuh"
using namespace pic;

// n waits in a row on a barrier nothing arrives on
__global__ void row_kernel(int n, unsigned long long limit_ns, int32_t *status, int *got) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    fence_mbar_init();
  }
  __syncthreads();
  bool ok = true;
  for (int i = 0; i < n; ++i)
    ok = mbar_wait_while(ok, smem_u32(&bar), 0, status, -1, limit_ns);
  if (threadIdx.x == 0) *got = ok;
}

// a wait of a CTA that has aborted, for a barrier that its other warp arrives on
// only after `late_ns`
__global__ void late_kernel(unsigned long long late_ns, unsigned long long limit_ns, int32_t *status,
                            int *got) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 32) {
    for (const uint64_t t0 = globaltimer_ns(); globaltimer_ns() - t0 < late_ns;) {
    }
    mbar_arrive(smem_u32(&bar));
  } else if (threadIdx.x == 0) {
    *got = mbar_wait_no_flag(smem_u32(&bar), 0, status, -1, limit_ns);
  }
}

extern "C" int late_arrival(unsigned long long late_ns, unsigned long long limit_ns, int32_t *status,
                            int *got) {
  late_kernel<<<1, 64>>>(late_ns, limit_ns, status, got);
  return (int)cudaGetLastError();
}

extern "C" int row_of_waits(int n, unsigned long long limit_ns, int32_t *status, int *got) {
  row_kernel<<<1, 32>>>(n, limit_ns, status, got);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def waits(cuda_lib, tmp_path_factory):
    d = tmp_path_factory.mktemp("waits")
    src, lib = str(d / "waits.cu"), str(d / "libwaits.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    from paper_2607_28069_gb300 import build
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-cudart", "shared", "-I", CSRC, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _ints(n):
    t = torch.zeros(n, dtype=torch.int32, device="cuda")
    return t, ctypes.c_void_p(t.data_ptr())


def test_a_wait_on_the_way_out_waits(waits):
    """What an aborted CTA waits for arrives 200 ms late, and is waited for."""
    status, sp = _ints(2)
    got, gp = _ints(1)
    assert waits.late_arrival(ctypes.c_uint64(200_000_000), ctypes.c_uint64(2_000_000_000), sp, gp) == 0
    torch.cuda.synchronize()
    assert got.item() == 1 and status.tolist() == [0, 0]


def test_a_row_of_waits_runs_out_once(waits):
    """32 waits with a limit of 50 ms: over after one limit, not after 32 of them."""
    status, sp = _ints(2)
    got, gp = _ints(1)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    assert waits.row_of_waits(32, ctypes.c_uint64(50_000_000), sp, gp) == 0
    torch.cuda.synchronize()
    elapsed = time.perf_counter() - t0
    assert got.item() == 0 and status.tolist() == [8, -1]  # PIC_DEV_TIMEOUT
    assert 0.05 <= elapsed < 4 * 0.05
