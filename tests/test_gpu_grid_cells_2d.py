"""Gridding of double-float planes without w (two planes per CTA, one of them in use) against the direct
sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2010_10122_gb300 import synthetic as S  # noqa: E402


@pytest.fixture(scope="module")
def wg():
    from paper_2010_10122_gb300 import _build
    _build.build()
    import paper_2010_10122_gb300 as wg
    return wg


# one visibility, chunks of 64 and a remainder, the narrowest and the widest support, both tile sides, no
# kernel-value table; crowded plans take the other shape
@pytest.mark.parametrize("nrows,nx,ny,alpha,tile,scale,opts", [
    (1, 64, 32, 4, 0, 1.0, {}), (65, 96, 64, 16, 0, 1.0, {}), (129, 128, 222, 8, 32, 1.0, {"compact_index": True}),
    (300, 150, 90, 9, 16, 1.0, {"compact_index": True}), (2000, 64, 64, 12, 0, 0.1, {})])
def test_grids_without_w(wg, oracle_lib, nrows, nx, ny, alpha, tile, scale, opts):
    eps = 1e-2 if alpha == 4 else 1e-6
    obs = S.random_uvw_observation(nrows, 2, nx, ny, 20.0, seed=nrows)
    uvw = obs.uvw * scale
    d = S.complex_normal((nrows, 2), seed=4)
    plan = wg.Plan(uvw, obs.freq, nx, ny, obs.pixsize_x, obs.pixsize_y, eps, "f64", do_wstacking=False,
                   force_alpha=alpha, force_sigma=2.0, tile=tile, fft_impl=2, **opts)
    assert plan.info["nw"] == 1 and plan.info["fft_impl"] == 2
    got = plan.grid(torch.from_numpy(d).cuda())
    ref = oracle_lib.grid(uvw, obs.freq, d, nx, ny, obs.pixsize_x, obs.pixsize_y, do_wstacking=False)
    assert oracle_lib.rel_l2(got.cpu().numpy(), ref) <= eps
