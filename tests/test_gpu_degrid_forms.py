"""Degridding of double-float planes in both forms of the footprint sum, against the direct sum."""
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


# packed sums (supports above 8 with w) and unpacked ones, the first and the last support of each; with a
# kernel-value table and without (a compact plan keeps none); batches of fewer planes than a CTA takes
@pytest.mark.parametrize("alpha,tile,do_w,opts", [
    (8, 0, True, {}), (8, 16, True, {"compact_index": True}), (4, 0, True, {"compact_index": True}),
    (9, 0, True, {}), (9, 32, True, {"compact_index": True}), (12, 0, True, {"compact_index": True}),
    (16, 0, True, {}), (16, 0, True, {"compact_index": True, "max_workspace": 3 << 20}),
    (16, 0, False, {}), (9, 0, False, {"compact_index": True}), (12, 32, False, {}), (6, 0, False, {})])
def test_forms(wg, oracle_lib, alpha, tile, do_w, opts):
    eps = {4: 1e-2, 6: 1e-4, 8: 1e-6}.get(alpha, 1e-6)
    obs = S.random_uvw_observation(700, 3, 96, 64, 20.0, seed=alpha)
    img = S.gaussian_image(96, 64, seed=3)
    plan = wg.Plan(obs.uvw, obs.freq, 96, 64, obs.pixsize_x, obs.pixsize_y, eps, "f64", do_wstacking=do_w,
                   force_alpha=alpha, force_sigma=2.0, tile=tile, fft_impl=2, **opts)
    assert plan.info["fft_impl"] == 2
    got = plan.degrid(torch.from_numpy(img).cuda())
    ref = oracle_lib.degrid(obs.uvw, obs.freq, img, obs.pixsize_x, obs.pixsize_y, do_wstacking=do_w)
    assert oracle_lib.rel_l2(got.cpu().numpy(), ref) <= eps
