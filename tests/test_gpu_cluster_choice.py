"""Which decoding steps merge their splits in a cluster: 4 to 16 splits, GQA groups
of up to 8 heads, and only where the GPU holds all clusters at once.  A GPU (or
a part of one) that places no such cluster runs the same plan with the merge
launch: simulated on the host by a library put before the CUDA runtime, which
answers that no cluster fits and refuses launches of clusters."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..")

FAKE = r"""
#include <cuda_runtime_api.h>
#include <dlfcn.h>
#include <stdio.h>
extern "C" cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) {
  *n = 0;
  return cudaSuccess;
}
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  using Fn = cudaError_t (*)(const cudaLaunchConfig_t *, const void *, void **);
  static Fn next = (Fn)dlsym(RTLD_NEXT, "cudaLaunchKernelExC");
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return cudaErrorInvalidClusterSize;
  fprintf(stderr, "fake launch\n");
  return next(c, f, args);
}
"""

STEP = """
import sys, torch
import paper_2607_28069_gb300 as pic
hq, hkv, dim, B, ctx, splits = (int(x) for x in sys.argv[2:8])
gen = torch.Generator(device="cuda").manual_seed(3)
rnd = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()
pages = ctx // 16 + 1
g = pic.Geometry(1, hq, hkv, dim, 5e5)
kc, vc = rnd(1, B * pages, hkv, 16, dim), rnd(1, B * pages, hkv, 16, dim)
bt = torch.arange(B * pages, dtype=torch.int32, device="cuda").view(B, pages)
q, k, v = rnd(B, hq, dim), rnd(B, hkv, dim), rnd(B, hkv, dim)
pos = torch.full((B,), ctx, dtype=torch.int32, device="cuda")
out = torch.empty_like(q)
ws = torch.empty(pic.pic_decode_workspace_size(g, B, ctx + 1, splits), dtype=torch.uint8, device="cuda")
pic.pic_attend_decode(g, 0, q, k, v, pos, bt, B * pages, kc, vc, out, ctx + 1, num_splits=splits, workspace=ws)
assert pic.pic_device_status() == (0, 0)
torch.save([t.cpu() for t in (out, kc, vc)], sys.argv[1])
"""


def _step(path, shape, **env):
    r = subprocess.run([sys.executable, "-c", STEP, path, *map(str, shape)], cwd=ROOT, text=True,
                       capture_output=True, env=dict(os.environ, **env), timeout=300)
    assert r.returncode == 0, r.stderr
    return torch.load(path), r.stderr.count("fake launch")


@pytest.mark.parametrize("shape", [(32, 8, 128, 1, 1000, 16), (16, 2, 64, 3, 500, 7)])
def test_without_clusters_the_merge_launch_runs(cuda_lib, tmp_path, shape):
    from paper_2607_28069_gb300 import build
    src, fake = str(tmp_path / "fake.cpp"), str(tmp_path / "fake.so")
    with open(src, "w") as f:
        f.write(FAKE)
    inc = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", f"-I{inc}", src, "-o", fake, "-ldl"], check=True)
    want, _ = _step(str(tmp_path / "a.pt"), shape)
    got, launches = _step(str(tmp_path / "b.pt"), shape, LD_PRELOAD=fake)
    assert launches == 2  # attention and merge, none of them refused
    assert all(torch.equal(a, b) for a, b in zip(got, want))
