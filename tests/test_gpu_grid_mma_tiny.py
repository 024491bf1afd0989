"""FP32 gridding on the tensor cores of data that are very small, throughout or in part."""
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


@pytest.mark.parametrize("lo,hi", [(-120, -120), (-90, -64), (-64, -62), (-10, 10), (-100, 0), (100, 110)])
def test_small_and_wide_magnitudes(wg, lo, hi):
    """Data times random powers of two: the gridded image is as near to the shared-memory atomics' as with
    ordinary data (both round each product and sum in FP32; the slices of the tensor cores drop
    nothing), here within 8 times that distance for the other weights of the cells."""
    obs = S.random_uvw_observation(3000, 4, 128, 96, 20.0, seed=5)
    geom = (obs.uvw, obs.freq, 128, 96, obs.pixsize_x, obs.pixsize_y, 1e-5, "f32")
    plan, atomics = wg.Plan(*geom), wg.Plan(*geom, grid_variant=1)
    assert plan.info["tile"] == 32 and plan.info["rounding_gain"] <= 40
    d = torch.from_numpy(S.complex_normal((3000, 4), seed=4).astype(np.complex64)).cuda()
    e = torch.from_numpy(np.random.default_rng(1).integers(lo, hi + 1, (3000, 4))).cuda()

    def apart(vis, scale):
        a, b = plan.grid(vis).double() * scale, atomics.grid(vis).double() * scale
        return ((a - b).norm() / b.norm()).item()
    assert apart(d * torch.exp2(e.float()), 2.0 ** -hi) <= 8 * apart(d, 1.0)
