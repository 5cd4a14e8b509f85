"""GPU test of the apply where the device cannot place a cluster: a fake of the launch call (a library loaded before the CUDA
runtime, in a process of its own) refuses every launch with a cluster; the launches per colour give the same bits.
"""
import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FAKE = r"""
#include <cuda_runtime_api.h>
#include <dlfcn.h>
static int refused = 0;
extern "C" int refused_launches() { return refused; }
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  for (unsigned k = 0; k < c->numAttrs; ++k)
    if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) {
      ++refused;
      return cudaErrorLaunchOutOfResources;
    }
  using Call = cudaError_t (*)(const cudaLaunchConfig_t *, const void *, void **);
  static Call real = (Call)dlsym(RTLD_NEXT, "cudaLaunchKernelExC");
  return real(c, f, args);
}
"""

RUN = r"""
import ctypes, os, sys
sys.path[:0] = [{root!r}, os.path.join({root!r}, "tests")]
import torch, synthetic
import paper_2109_05072_gb300 as ceed
from _util import gpu_mesh
out = []
for p, prec in ((2, 0), (7, 0), (3, 1)):
    m = synthetic.HexMesh(2, 2, 2, p, seed=p)
    mesh = gpu_mesh(ceed, m, "gll")
    qd = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, prec)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, prec, qd)
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=1)).cuda()
    y = torch.full_like(x, float("nan"))
    ceed.ceed_apply_diffusion(mesh, qd, prec, x, y)
    ceed.ceed_mesh_status(mesh)
    out.append(y.cpu())
torch.save(out, sys.argv[1])
n = ctypes.CDLL(sys.argv[2]).refused_launches() if len(sys.argv) > 2 else 0
print("refused", n)
"""


def test_launches_per_colour_stand_in(tmp_path):
    cc, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if cc is None or not os.path.exists(nvcc):
        pytest.skip("no C++ compiler or CUDA headers")
    src, lib, run = tmp_path / "fake.cpp", tmp_path / "fake.so", tmp_path / "run.py"
    src.write_text(FAKE)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run([cc, "-shared", "-fPIC", "-I", include, str(src), "-o", str(lib), "-ldl"], check=True)
    run.write_text(RUN.format(root=os.path.dirname(os.path.dirname(os.path.abspath(__file__)))))
    plain, faked = tmp_path / "plain.pt", tmp_path / "faked.pt"
    subprocess.run([sys.executable, str(run), str(plain)], check=True)
    r = subprocess.run([sys.executable, str(run), str(faked), str(lib)], env={**os.environ, "LD_PRELOAD": str(lib)},
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert "refused 3" in r.stdout
    for a, b in zip(torch.load(plain), torch.load(faked)):
        assert torch.equal(a, b)
