"""One-shot calls (App. B) on the GPU: their plans serve one call, and in single precision take
the library's FP32 plane FFT instead of cuFFT where that is cheaper in all.  Same grid and
kernel, so the result meets epsilon against the FP64 direct sum like a resident plan's."""
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


# sides with odd halves (ragged column groups), unequal axes, the smallest image, 5- and 7-smooth
# grids; with weights and a mask in turn
@pytest.mark.parametrize("nx,ny,nrows,nchan,eps,do_w", [(32, 32, 7, 1, 1e-5, True), (86, 130, 300, 3, 1e-5, True),
                                                        (150, 98, 211, 2, 1e-4, False), (222, 222, 123, 5, 1e-3, True)])
def test_oneshot_f32_matches_oracle(wg, oracle_lib, nx, ny, nrows, nchan, eps, do_w):
    obs = S.random_uvw_observation(nrows, nchan, nx, ny, 20.0, seed=nx)
    rng = np.random.default_rng(ny)
    I, d = S.gaussian_image(nx, ny, seed=3), S.complex_normal((nrows, nchan), seed=4)
    wgt = rng.uniform(0.5, 2.0, (nrows, nchan)) if nx % 4 else None
    mask = (rng.random((nrows, nchan)) < 0.9).astype(np.uint8) if ny % 4 else None
    w32 = None if wgt is None else wgt.astype(np.float32)
    vis = wg.dirty2ms(obs.uvw, obs.freq, I.astype(np.float32), wgt=w32, pixsize_x=obs.pixsize_x,
                      pixsize_y=obs.pixsize_y, epsilon=eps, do_wstacking=do_w, mask=mask).cpu().numpy()
    img = wg.ms2dirty(obs.uvw, obs.freq, d.astype(np.complex64), wgt=w32, npix_x=nx, npix_y=ny,
                      pixsize_x=obs.pixsize_x, pixsize_y=obs.pixsize_y, epsilon=eps, do_wstacking=do_w,
                      mask=mask).cpu().numpy()
    kw = dict(wgt=wgt, mask=mask, do_wstacking=do_w)
    rv = oracle_lib.degrid(obs.uvw, obs.freq, I, obs.pixsize_x, obs.pixsize_y, **kw)
    ri = oracle_lib.grid(obs.uvw, obs.freq, d, nx, ny, obs.pixsize_x, obs.pixsize_y, **kw)
    assert oracle_lib.rel_l2(vis, rv) <= eps and oracle_lib.rel_l2(img, ri) <= eps
