"""Gridding of double-float planes (register accumulators) against the direct sum."""
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


# visibilities around the 16-lane groups and the chunks of 64 and 128; the narrowest and the widest
# support, 32- and 16-cell tiles; plane counts that leave a group of 8 incomplete, batches of few
# planes and no kernel-value table (compact plan, small workspace); without w; dense plans, where
# four sets of warps share the cells
@pytest.mark.parametrize("nrows,nchan,nx,ny,alpha,eps,tile,do_w,opts", [
    (1, 1, 32, 32, 8, 1e-6, 0, True, {}), (15, 1, 64, 96, 4, 1e-2, 32, True, {}),
    (65, 1, 96, 64, 16, 1e-12, 16, True, {}), (129, 3, 128, 222, 13, 1e-9, 0, False, {}),
    (300, 5, 150, 90, 9, 1e-6, 16, True, {}), (300, 5, 150, 90, 9, 1e-6, 32, True, {}),
    (3000, 1, 64, 64, 12, 1e-8, 0, True, {"compact_index": True, "max_workspace": 4 << 20}),
    (2000, 8, 48, 64, 12, 1e-9, 0, True, {}), (2000, 8, 48, 64, 6, 1e-4, 32, True, {})])
def test_register_gridding(wg, oracle_lib, nrows, nchan, nx, ny, alpha, eps, tile, do_w, opts):
    obs = S.random_uvw_observation(nrows, nchan, nx, ny, 20.0, seed=nrows)
    uvw = obs.uvw * (0.2 if nrows == 2000 else 1.0)   # crowded towards the origin
    rng = np.random.default_rng(nx)
    d = S.complex_normal((nrows, nchan), seed=4)
    wgt = rng.uniform(0.5, 2.0, (nrows, nchan)) if nrows % 2 else None
    geom = (uvw, obs.freq, nx, ny, obs.pixsize_x, obs.pixsize_y)
    vis = torch.from_numpy(d).cuda()
    plan = wg.Plan(*geom, eps, "f64", do_wstacking=do_w, force_alpha=alpha, force_sigma=2.0,
                   tile=tile, **opts)
    w = None if wgt is None else torch.from_numpy(wgt).cuda()
    got = plan.grid(vis, wgt=w)
    assert torch.equal(got, plan.grid(vis, wgt=w))      # reproducible
    ref = oracle_lib.grid(uvw, obs.freq, d, nx, ny, obs.pixsize_x, obs.pixsize_y, wgt=wgt,
                          do_wstacking=do_w)
    assert oracle_lib.rel_l2(got.cpu().numpy(), ref) <= eps
