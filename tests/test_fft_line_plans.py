"""The double-float FFT's plan of a line as the library reports it, and the operations counted for it (host
arithmetic, no GPU)."""
import math

import pytest

import bench
from paper_2010_10122_gb300 import wgrid


@pytest.mark.parametrize("n,forward,kernel,parts", [
    (512, True, "k_fft_pairs", 1), (2048, False, "k_fft_pairs", 1), (3456, True, "k_fft_pairs", 4),
    (13824, True, "k_fft_pairs", 8), (640, True, "k_fft_lines", 1), (640, False, "k_fft_pairs", 1),
    (3168, True, "k_fft_lines", 1), (2016, False, "k_fft_lines", 1),   # sides that stay line by line
    (17280, True, "k_fft_lines_cluster", 4)])                           # above 8 x 2048 points
def test_line_kernels(n, forward, kernel, parts):
    pairs, got, radices = wgrid.fft_df64_line(n, forward)
    assert got == parts and math.prod(radices) * parts == n
    assert bench.df64_pass(n, "degrid" if forward else "grid")[0] == kernel and pairs == (kernel == "k_fft_pairs")


def test_pair_operations():
    # 3456 points as 4 x 864, radices 8 6 6 3: 430 per point (the line kernels' transform: 460); one radix-8
    # stage after another has 7 twiddle products a butterfly
    assert bench.df64_pass(3456, "degrid")[1] == 864 * (176 + 114) + 4 * (
        108 * 600 + 2 * 144 * (432 + 190) + 288 * (150 + 76)) == 1486656
    assert bench.df64_pass(512, "grid")[1] == 64 * 600 + 2 * 64 * (600 + 266)
    with pytest.raises(wgrid.WgridError):
        wgrid.fft_df64_line(13 * 8)
