"""Double-float FFT of long lines where no thread-block cluster can be placed: the lines go to the
kernels that do without.  The refusal is a fake of the two runtime calls, preloaded into a child
process."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FAKE = r"""
#include <dlfcn.h>
#include <cuda_runtime_api.h>
typedef cudaError_t (*launch_t)(const cudaLaunchConfig_t*, const void*, void**);
extern "C" cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 0;
  return cudaSuccess;
}
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension && c->attrs[i].val.clusterDim.x > 1)
      return cudaErrorLaunchOutOfResources;
  static const launch_t real = (launch_t)dlsym(dlopen("libcudart.so.13", RTLD_NOW), "cudaLaunchKernelExC");
  return real(c, f, args);
}
"""
CHILD = r"""
import numpy as np, torch
import paper_2010_10122_gb300 as wg
rng = np.random.default_rng(1)
for shape in ((1, 3, 3456), (1, 3072, 5), (1, 16, 5632), (1, 4, 13824)):
    for sign in (-1, 1):
        x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
        a = torch.from_numpy(x).cuda()
        wg.wgrid.fft2d(a, sign=sign, impl=2)
        ref = np.fft.fft2(x) if sign < 0 else np.fft.ifft2(x) * (shape[1] * shape[2])
        err = np.linalg.norm(a.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err < 5e-14, (shape, sign, err)
print("transforms done")
"""


def test_long_lines_without_clusters(tmp_path):
    from paper_2010_10122_gb300 import _build
    _build.build()
    (tmp_path / "fake.cpp").write_text(FAKE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    fake = str(tmp_path / "fake.so")
    subprocess.check_call(["g++", "-shared", "-fPIC", "-I" + cuda, str(tmp_path / "fake.cpp"), "-o", fake, "-ldl"])
    env = dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=_build.ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "transforms done" in r.stdout, r.stdout + r.stderr
