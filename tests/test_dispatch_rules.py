"""The rules that choose a form of the (de)gridding kernels by sizes (host arithmetic, no GPU), at sizes
measured on both sides of each line."""
import ctypes
import subprocess

import pytest

from paper_2010_10122_gb300 import _build

WRAPPER = r"""
#include "host_math.h"
extern "C" int shares(double densest, double mean, double least, double ctas, int f32) {
  return wg::degrid_shares(densest, mean, least, ctas, f32 != 0);
}
extern "C" int launches(double densest, double mean, double ctas) { return wg::mma_launches(densest, mean, ctas); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(WRAPPER)
    so = str(d / "rules.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I" + _build.CSRC, str(d / "rules.cpp"),
                           _build.CSRC + "/host_math.cpp", _build.CSRC + "/kernel_design.cpp", "-o", so])
    lib = ctypes.CDLL(so)
    lib.shares.argtypes = [ctypes.c_double] * 4 + [ctypes.c_int]
    lib.launches.argtypes = [ctypes.c_double] * 3
    return lib


@pytest.mark.parametrize("densest,mean,least,ctas,f32,lo,hi", [
    # few dense tiles of a small grid: several CTAs (256^2 1523 us with one, 268 with 32; double-float 70 -> 7 ms)
    (24953.6, 3700.4, 1792, 1024, 1, 8, 32), (54227.2, 1184.2, 576, 64512, 0, 8, 32),
    # a few crowded tiles of a large grid: one (2816^2: 575 us, 717 with two; 4000^2 without w; 5760^2 FP64)
    (2947.7, 904.6, 448, 77440, 1, 1, 1), (2056.0, 328.9, 128, 40000, 1, 1, 1), (1584.0, 32.9, 128, 129600, 0, 1, 1),
    # even plans: one
    (2386.8, 2960.3, 1472, 12150, 1, 1, 1), (2848.4, 4659.8, 2304, 20480, 0, 1, 1), (0.0, 0.0, 128, 1, 1, 1, 1)])
def test_degrid_shares(rules, densest, mean, least, ctas, f32, lo, hi):
    assert lo <= rules.shares(densest, mean, least, ctas, f32) <= hi


@pytest.mark.parametrize("densest,mean,ctas,form", [
    (1518, 195, 1024, 4), (14855, 389, 5120, 4),                 # dense small grids: four warps everywhere
    (538, 1727, 4096, 1), (170, 17, 26244, 1), (487, 47, 309760, 1),   # even, or too many tiles: one warp
    (2556, 173, 15625, 5), (5935, 475, 77440, 5), (0, 0, 1, 1)])       # crowded large grids: two launches
def test_mma_launches(rules, densest, mean, ctas, form):
    got = rules.launches(densest, mean, ctas)
    assert got == form
