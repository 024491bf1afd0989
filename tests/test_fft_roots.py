"""The double-float FFT's constants and twiddle factors (host arithmetic, no GPU): every one is the
pair of floats next to its value."""
import subprocess

import numpy as np
import pytest

from paper_2010_10122_gb300 import _build

PROGRAM = r"""
#include <cstdio>
#include "fft_engine.cuh"
#include "host_math.h"
using namespace wg;
static void put(int n, int t, float a, float b, float c, float d) { printf("%d %d %a %a %a %a\n", n, t, a, b, c, d); }
template <int N, int K> static void roots() {   // the constants of radix N: e^{-2 pi i K / N}
  if constexpr (K < N) {
    constexpr Konst c{trig::cos2pi(K, N)}, s{trig::neg(trig::sin2pi(K, N))};
    put(N, K, c.h, c.l, s.h, s.l);
    roots<N, K + 1>();
  }
}
int main() {
  roots<3, 0>(); roots<5, 0>(); roots<7, 0>(); roots<8, 0>(); roots<9, 0>(); roots<11, 0>();
  for (int n : {16, 30, 576, 1155, 2048, 3456, 11264, 16384}) {
    const UnitRoots r(n);
    for (int t = 0; t < n; ++t) { float w[4]; r.pair(t, w); put(n, t, w[0], w[1], w[2], w[3]); }
  }
}
"""


@pytest.fixture(scope="module")
def entries(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    (d / "roots.cu").write_text(PROGRAM)
    src = [_build.CSRC + "/host_math.cpp", _build.CSRC + "/kernel_design.cpp"]
    subprocess.check_call([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "-I" + _build.CSRC,
                           str(d / "roots.cu"), *src, "-o", str(d / "roots")])
    out = subprocess.check_output([str(d / "roots")], text=True).split()
    return np.array([float.fromhex(x) if "x" in x else float(x) for x in out]).reshape(-1, 6)


def test_roots_are_the_nearest_float_pairs(entries):
    """High part: the nearest float.  Low part: within half its last bit of the rest, beside the
    reference's own error: three roundings (2^-64) of an angle up to 2 pi, below 2^-59."""
    n, t = entries[:, 0], entries[:, 1]
    angle = 2 * np.longdouble("3.14159265358979323846264338327950288") * t.astype(np.longdouble) / n
    for v, h, l in ((np.cos(angle), entries[:, 2], entries[:, 3]), (-np.sin(angle), entries[:, 4], entries[:, 5])):
        some = np.abs(v) > 2.0 ** -40   # not the zeros of the reference
        assert np.array_equal(h[some], v[some].astype(np.float32))
        half = 0.5 * np.spacing(np.abs(l).astype(np.float32)).astype(np.longdouble)
        assert (np.abs(v - h - l) <= half + 2.0 ** -59).all()
