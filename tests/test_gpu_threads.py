"""Calls of plans that differ in shared memory per CTA, from several host threads at once."""
import threading

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


# supports of one lane group, whose tiles take different amounts of shared memory, on the same kernels
@pytest.mark.parametrize("prec,alphas,opts", [("f32", (5, 8), {}), ("f32", (5, 8), {"grid_variant": 1}),
                                              ("f64", (5, 8), {}), ("f64", (9, 16), {})])
def test_concurrent_calls(wg, prec, alphas, opts):
    obs = S.random_uvw_observation(200, 2, 64, 64, 20.0, seed=1)
    real, cplx = (torch.float32, torch.complex64) if prec == "f32" else (torch.float64, torch.complex128)
    img = torch.from_numpy(S.gaussian_image(64, 64, seed=1)).to(real).cuda()
    vis = torch.from_numpy(S.complex_normal((200, 2), seed=2)).to(cplx).cuda()
    plans = [wg.Plan(obs.uvw, obs.freq, 64, 64, obs.pixsize_x, obs.pixsize_y, 1e-2, prec, force_alpha=a,
                     force_sigma=2.0, **opts) for a in alphas]
    want = [p.degrid(img).cpu().numpy() for p in plans]
    torch.cuda.synchronize()
    failed = []

    def work(k):
        stream = torch.cuda.Stream()
        out = torch.empty((200, 2), dtype=cplx, device="cuda")
        dirty = torch.empty((64, 64), dtype=real, device="cuda")
        try:
            for _ in range(1500):
                plans[k].degrid(img, out=out, stream=stream)
                plans[k].grid(vis, out=dirty, stream=stream)
            stream.synchronize()
            if not np.array_equal(out.cpu().numpy(), want[k]):
                failed.append("result")
        except Exception as e:   # a refused launch
            failed.append(str(e))

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1, 0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
