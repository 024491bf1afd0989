"""The w phase of FP32 index records: FP64 cosine and sine rounded to float, whatever computes them."""
import ctypes
import subprocess

import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "kernels_index.cu"
namespace wg {
__global__ void k_probe(const double* c, float2* out, double2* ref, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = cis_turn(c[i]);
  sincospi(2.0 * c[i], &ref[i].y, &ref[i].x);
}
}
extern "C" int probe(const double* c, float* out, double* ref, int n) {
  double *dc, *dr; float2* d;
  if (cudaMalloc(&dc, n * 8) || cudaMalloc(&d, n * 8) || cudaMalloc(&dr, n * 16)) return 1;
  cudaMemcpy(dc, c, n * 8, cudaMemcpyHostToDevice);
  wg::k_probe<<<(n + 255) / 256, 256>>>(dc, d, (double2*)dr, n);
  cudaMemcpy(out, d, n * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(ref, dr, n * 16, cudaMemcpyDeviceToHost);
  const int e = (int)cudaDeviceSynchronize();
  cudaFree(dc); cudaFree(d); cudaFree(dr);
  return e;
}
"""


def test_phase_is_the_rounded_double(tmp_path):
    """Random angles, and angles next to the quarter turns, where one of the two is near zero: equal to
    the rounded FP64 values in every bit but the sign of a zero."""
    from paper_2010_10122_gb300 import _build
    (tmp_path / "probe.cu").write_text(PROGRAM)
    so = str(tmp_path / "probe.so")
    subprocess.check_call([_build.nvcc(), *_build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-I" + _build.INCLUDE, "-I" + _build.CSRC, str(tmp_path / "probe.cu"), "-o", so,
                           "-lcudart"])
    rng = np.random.default_rng(1)
    near = np.outer([-0.5, -0.25, 0.0, 0.25, 0.5], np.ones(20000)) + \
        np.sign(rng.standard_normal((5, 20000))) * 2.0 ** rng.uniform(-60, -3, (5, 20000))
    c = np.concatenate([rng.uniform(-0.5, 0.5, 1 << 22), np.clip(near, -0.5, 0.5).reshape(-1),
                        np.arange(-4, 5) / 8.0])
    out, ref = np.empty((c.size, 2), np.float32), np.empty((c.size, 2))
    vp = ctypes.c_void_p
    assert ctypes.CDLL(so).probe(vp(c.ctypes.data), vp(out.ctypes.data), vp(ref.ctypes.data), c.size) == 0
    assert np.abs(ref[:, 0] - np.cos(2 * np.pi * c)).max() < 1e-14      # the reference itself
    assert np.array_equal(out, ref.astype(np.float32)), np.count_nonzero((out != ref.astype(np.float32)).any(1))
