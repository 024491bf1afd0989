"""Degridding of tiles that several CTAs share, against the direct sum."""
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


# visibilities crowded into a few tiles (scale 0.05) beside spread ones: shares that end within a
# pass of a CTA, the last CTA without any; both tile sides, 4, 8 and 16 lanes per visibility, planes in
# batches, and an odd plane count of a visibility's sub-batches
@pytest.mark.parametrize("prec,nrows,crowd,alpha,eps,tile,do_w,opts", [
    ("f32", 3001, 2900, 4, 1e-2, 32, True, {}), ("f32", 3001, 3001, 8, 1e-4, 32, True, {}),
    ("f32", 2999, 2000, 11, 1e-5, 16, True, {"max_workspace": 8 << 20}), ("f32", 1500, 1400, 7, 1e-3, 32, False, {}),
    ("f64", 3001, 2900, 4, 1e-2, 32, True, {}), ("f64", 3001, 3001, 13, 1e-9, 16, True, {}),
    ("f64", 2999, 2000, 8, 1e-5, 32, True, {"compact_index": True, "max_workspace": 4 << 20}),
    ("f64", 1500, 1400, 10, 1e-7, 16, False, {}), ("f64", 2000, 1999, 10, 1e-7, 16, True, {"fft_impl": 1})])
def test_shared_tiles(wg, oracle_lib, prec, nrows, crowd, alpha, eps, tile, do_w, opts):
    nx, ny = 96, 64
    obs = S.random_uvw_observation(nrows, 2, nx, ny, 20.0, seed=nrows)
    uvw = obs.uvw.copy()
    uvw[:crowd, :2] *= 0.05
    img = S.gaussian_image(nx, ny, seed=3)
    plan = wg.Plan(uvw, obs.freq, nx, ny, obs.pixsize_x, obs.pixsize_y, eps, prec, do_wstacking=do_w,
                   force_alpha=alpha, force_sigma=2.0, tile=tile, **opts)
    x = torch.from_numpy(img.astype(np.float32 if prec == "f32" else np.float64)).cuda()
    got = plan.degrid(x)
    assert torch.equal(got, plan.degrid(x))
    ref = oracle_lib.degrid(uvw, obs.freq, x.cpu().numpy().astype(np.float64), obs.pixsize_x, obs.pixsize_y,
                            do_wstacking=do_w)
    assert oracle_lib.rel_l2(got.cpu().numpy(), ref) <= eps
