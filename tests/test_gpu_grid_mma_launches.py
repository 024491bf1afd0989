"""FP32 tensor-core gridding of plans with a few crowded tiles: dense tiles in a launch of their own."""
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


# half of the visibilities in the middle, by the scale of their u and v: even, two launches with many and with
# few dense tiles, four warps for every tile; with and without w; one batch of planes and several
@pytest.mark.parametrize("n,rows,scale,do_w,launches,opts", [
    (512, 20000, 1.0, True, 1, {}), (512, 20000, 0.3, True, None, {}), (768, 20000, 0.05, True, 2, {}),
    (768, 20000, 0.05, True, None, {"max_workspace": 64 << 20}), (1024, 20000, 0.02, False, None, {}),
    (256, 20000, 0.05, True, 1, {})])
def test_crowded_tiles(wg, oracle_lib, n, rows, scale, do_w, launches, opts):
    obs = S.random_uvw_observation(rows, 1, n, n, 12.0, seed=3)
    uvw = obs.uvw.copy()
    uvw[: rows // 2, :2] *= scale
    geom = (uvw, obs.freq, n, n, obs.pixsize_x, obs.pixsize_y)
    vis = torch.from_numpy(S.complex_normal((rows, 1), seed=4).astype(np.complex64)).cuda()
    plan = wg.Plan(*geom, 1e-5, "f32", do_wstacking=do_w, **opts)
    assert plan.info["tile"] == 32 and plan.info["rounding_gain"] <= 40
    got, st = plan.grid(vis, stats=True)
    assert torch.equal(got, plan.grid(vis))      # reproducible
    if launches is not None:
        assert st["n_batches"] == 1 and st["n_kernels"] == launches + 1
    ref = wg.Plan(*geom, 1e-10, "f64", do_wstacking=do_w).grid(vis.to(torch.complex128))
    assert ((got.double() - ref).norm() / ref.norm()).item() <= 1e-5
