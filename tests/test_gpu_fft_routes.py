"""Double-float FFT of complex128 planes whose passes run on different kernels, against numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wg():
    from paper_2010_10122_gb300 import _build
    _build.build()
    import paper_2010_10122_gb300 as wg
    return wg


# both passes line by line forward (640, 800), one of them in either place, both on pairs of lines; sides
# that never go in pairs (3168; 15); passes of few lines and of many
@pytest.mark.parametrize("shape", [(1, 640, 800), (2, 640, 512), (2, 512, 640), (1, 3168, 640), (3, 15, 640),
                                   (1, 128, 128), (9, 128, 128), (1, 96, 1024), (20, 96, 64), (1, 1344, 2048)])
@pytest.mark.parametrize("sign", [-1, 1])
def test_routes(wg, shape, sign):
    rng = np.random.default_rng(sum(shape) + sign)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    a = torch.from_numpy(x).cuda()
    wg.wgrid.fft2d(a, sign=sign, impl=2)
    ref = np.fft.fft2(x) if sign < 0 else np.fft.ifft2(x) * (shape[1] * shape[2])
    assert np.linalg.norm(a.cpu().numpy() - ref) / np.linalg.norm(ref) < 5e-14   # the FFT's own bound
