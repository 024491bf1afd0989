"""FP32 gridding on the tensor cores (the automatic choice with 32-cell tiles) against the FP64
direct sum (and, for many visibilities, the FP64 plan)."""
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


# visibilities around the groups of 16 and the blocks of 64; supports of 8- and 16-lane groups, odd
# ones and the smallest (sigma 2 where they are forced, so that the planes' rounding is not
# amplified); plane counts that leave a group of planes incomplete; without w; dense small grids
# (four warps per quarter) and sparse ones
@pytest.mark.parametrize("nrows,nchan,nx,ny,alpha,eps,do_w", [
    (1, 1, 32, 32, 8, 1e-5, True), (15, 1, 64, 96, 5, 1e-2, True), (17, 1, 96, 64, 8, 1e-4, True),
    (65, 2, 128, 128, 7, 1e-4, False), (129, 3, 150, 90, 4, 1e-2, True),
    (211, 4, 128, 222, 12, 1e-5, True), (300, 5, 96, 96, 16, 1e-5, True),
    (20000, 8, 64, 64, 8, 1e-5, True), (9000, 16, 96, 128, 11, 1e-5, True), (9000, 16, 128, 96, 0, 1e-5, True)])
def test_tensor_core_gridding(wg, oracle_lib, nrows, nchan, nx, ny, alpha, eps, do_w):
    obs = S.random_uvw_observation(nrows, nchan, nx, ny, 20.0, seed=nrows)
    rng = np.random.default_rng(nx)
    d = S.complex_normal((nrows, nchan), seed=4)
    wgt = rng.uniform(0.5, 2.0, (nrows, nchan)).astype(np.float32) if nrows % 2 else None
    mask = (rng.random((nrows, nchan)) < 0.9).astype(np.uint8) if nrows % 3 == 0 else None
    geom = (obs.uvw, obs.freq, nx, ny, obs.pixsize_x, obs.pixsize_y)
    vis = torch.from_numpy(d.astype(np.complex64)).cuda()
    w32 = None if wgt is None else torch.from_numpy(wgt).cuda()
    plan = wg.Plan(*geom, eps, "f32", mask=mask, do_wstacking=do_w, force_alpha=alpha,
                   force_sigma=2.0 if alpha else 0.0)
    assert plan.info["tile"] == 32
    got = plan.grid(vis, wgt=w32)
    assert torch.equal(got, plan.grid(vis, wgt=w32))      # reproducible
    # the direct sum; where that takes too long, the FP64 plan at 1e-11
    if nrows * nchan * nx * ny < 1e8:
        ref = oracle_lib.grid(obs.uvw, obs.freq, d, nx, ny, obs.pixsize_x, obs.pixsize_y, wgt=wgt,
                              mask=mask, do_wstacking=do_w)
    else:
        fine = wg.Plan(*geom, 1e-11, "f64", mask=mask, do_wstacking=do_w)
        ref = fine.grid(vis.to(torch.complex128), wgt=None if w32 is None else w32.double()).cpu().numpy()
    assert oracle_lib.rel_l2(got.cpu().numpy(), ref) <= eps


def test_large_rounding_gain_takes_the_atomics(wg, oracle_lib):
    obs = S.random_uvw_observation(500, 2, 128, 96, 20.0, seed=5)
    d = S.complex_normal((500, 2), seed=4)
    plan = wg.Plan(obs.uvw, obs.freq, 128, 96, obs.pixsize_x, obs.pixsize_y, 1e-3, "f32", force_alpha=7,
                   force_sigma=1.15)
    assert plan.info["tile"] == 32 and plan.info["rounding_gain"] > 40
    got = plan.grid(torch.from_numpy(d.astype(np.complex64)).cuda())
    ref = oracle_lib.grid(obs.uvw, obs.freq, d, 128, 96, obs.pixsize_x, obs.pixsize_y)
    assert oracle_lib.rel_l2(got.cpu().numpy(), ref) <= 1e-3
