"""What this library is measured on: the measurement operator R (degrid, image -> visibilities),
its adjoint (grid, visibilities -> image), one pass of an imaging loop and one of a gradient
step, through the public Python entry points, over the sizes, accuracies and options that the
repository's workloads, tests and serving mix use.

A case is
  call   "degrid" | "grid": one call on a resident plan; "oneshot_degrid" | "oneshot_grid": the
         one-shot calls (plan made and destroyed inside); "residual": grid(d - degrid(x)), the
         major cycle of an imager; "step": forward and backward of 0.5 ||degrid(x) - d||^2
  prec, eps                   precision and requested accuracy
  nx, ny, fov                 image sides in pixels; field of view in degrees along the longer side
  ant, times, chans           antennas, integrations and channels of the synthesised observation
                              (ant 0: `times` rows of uniform random uvw instead of an array)
  wgt, mask, compact          weights; a mask (5 % of the visibilities flagged); the compact index
                              that the server's plans use
"""
import math

import numpy as np
import torch

import paper_2010_10122_gb300 as wg
from paper_2010_10122_gb300 import autograd
from paper_2010_10122_gb300 import synthetic as S

_REAL = {"f32": torch.float32, "f64": torch.float64}
_CPLX = {"f32": torch.complex64, "f64": torch.complex128}
C_LIGHT = 299792458.0
FOV_2K = 2048 * 20 / 3600.0        # the wide-field workloads' 11.4 degrees
FOV_8K = 8192 * 4 / 3600.0         # the 8192^2 workload's 9.1 degrees
FOV_4K = 4096 * 4 / 3600.0         # the differentiable workload's 4.6 degrees


def _case(name, call, prec, eps, nx, ny, fov, ant, times, chans, wgt=False, mask=False,
          compact=False):
    return {"name": name, "call": call, "prec": prec, "eps": eps, "nx": nx, "ny": ny, "fov": fov,
            "ant": ant, "times": times, "chans": chans, "wgt": wgt, "mask": mask,
            "compact": compact}


def listed():
    return [
        # The smallest problem in use: 256^2, 1e4 random visibilities in double precision (the
        # tiny workload).  Latency and launches count: a sampler calls it thousands of times.
        _case("tiny_f64_degrid", "degrid", "f64", 1e-10, 256, 256, 12.8, 0, 10000, 1),
        _case("tiny_f64_grid", "grid", "f64", 1e-10, 256, 256, 12.8, 0, 10000, 1),
        # Small requests of the serving mix: single precision at 1e-4, 16 channels, served from
        # compact plans; the gridded data carry weights and flags as calibrated data do.
        _case("serve_512_f32_grid", "grid", "f32", 1e-4, 512, 512, FOV_2K, 64, 4, 16, wgt=True,
              mask=True, compact=True),
        _case("serve_1k_f32_degrid", "degrid", "f32", 1e-4, 1024, 1024, FOV_2K, 64, 20, 16,
              compact=True),
        # Ragged double precision: odd image sides, a 27-antenna array, 7 channels, weights, at
        # the accuracy of the double-precision mode and small enough for the direct sum.
        _case("ragged_f64_grid", "grid", "f64", 1e-12, 354, 250, 8.0, 27, 11, 7, wgt=True),
        # The paper's interface: one call per data set, planning included, ragged sides.
        _case("oneshot_ragged_f32_grid", "oneshot_grid", "f32", 1e-5, 1470, 1038, 9.0, 41, 37, 5),
        # The bench workload: 2048^2 at 20 arcsec, 999,936 visibilities, both directions and
        # both precisions (1e-5 in single, 1e-12 in double precision).
        _case("wide_2k_f32_degrid", "degrid", "f32", 1e-5, 2048, 2048, FOV_2K, 64, 62, 8),
        _case("wide_2k_f32_grid", "grid", "f32", 1e-5, 2048, 2048, FOV_2K, 64, 62, 8),
        _case("wide_2k_f64_degrid", "degrid", "f64", 1e-12, 2048, 2048, FOV_2K, 64, 62, 8),
        _case("wide_2k_f64_grid", "grid", "f64", 1e-12, 2048, 2048, FOV_2K, 64, 62, 8),
        # The differentiable workload: gradient of 0.5 ||degrid(x) - d||^2 for a 4096^2 image and
        # 9,999,360 visibilities.
        _case("diff_4k_f32_step", "step", "f32", 1e-5, 4096, 4096, FOV_4K, 64, 310, 16),
        # The largest: 8192^2 with 64 channels, 5e7 visibilities, the residual image of a major
        # cycle.
        _case("wide_8k_f32_residual", "residual", "f32", 1e-5, 8192, 8192, FOV_8K, 128, 97, 64),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    prec = rng.choice(["f32", "f32", "f64"])
    eps = rng.choice([1e-3, 1e-4, 1e-5, 1e-5] if prec == "f32" else [1e-7, 1e-10, 1e-12, 1e-12])
    top = 6000 if prec == "f32" else 2300
    nx = 2 * int(_log(rng, 128, top / 2))
    ny = nx if rng.random() < 0.5 else 2 * int(nx * rng.uniform(0.4, 1.0) / 2)
    ant = rng.choice([0, 27, 41, 64, 64, 128])
    chans = rng.choice([1, 3, 5, 8, 16, 16, 31, 64])
    vis = _log(rng, 1e4, 2e7 if prec == "f32" else 2e6)
    if ant == 0:
        times = max(1, int(vis / chans))
    else:
        times = max(2, int(round(vis / chans / (ant * (ant - 1) // 2))))
    call = rng.choice(["degrid", "grid", "degrid", "grid", "residual", "step", "oneshot_degrid",
                       "oneshot_grid"])
    oneshot = call.startswith("oneshot")
    fov = rng.uniform(3.0, FOV_2K)
    c = _case("", call, prec, eps, nx, ny, fov, ant, times, chans, wgt=rng.random() < 0.4,
              mask=rng.random() < 0.3, compact=(not oneshot) and rng.random() < 0.3)
    del c["name"]
    return c


def _rows(case):
    return case["times"] * (case["ant"] * (case["ant"] - 1) // 2 if case["ant"] else 1)


def _observation(case, seed):
    pix = math.radians(case["fov"]) / max(case["nx"], case["ny"])
    if case["ant"]:
        obs = S.array_observation(case["ant"], case["times"], case["chans"],
                                  max(case["nx"], case["ny"]), pix, seed=seed)
        return obs.uvw, obs.freq, pix
    # uniform random uvw inside the uv grid, w within half of that, as the tiny workload has it
    freq = np.linspace(1.0e9, 1.4e9, case["chans"]) if case["chans"] > 1 else np.array([1.0e9])
    lim = 0.45 / pix * C_LIGHT / freq.max()
    uvw = np.random.default_rng(seed).uniform(-lim, lim, (case["times"], 3))
    uvw[:, 2] *= 0.5
    return uvw, freq, pix


def _inputs(case, seed):
    uvw, freq, pix = _observation(case, seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    real = _REAL[case["prec"]]
    rows, chans, call = uvw.shape[0], case["chans"], case["call"]
    s = {"case": case, "pix": pix, "img": None, "vis": None, "wgt": None, "mask": None}
    s["uvw"] = torch.from_numpy(np.ascontiguousarray(uvw)).cuda()
    s["freq"] = torch.from_numpy(freq).cuda()
    if call != "grid" and call != "oneshot_grid":
        # 1 % of the pixels hold point sources of log-normal flux
        x = torch.rand((case["nx"], case["ny"]), generator=gen, device="cuda", dtype=torch.float32)
        flux = torch.randn(x.shape, generator=gen, device="cuda", dtype=torch.float32).exp_()
        s["img"] = torch.where(x < 0.01, flux, torch.zeros_like(flux)).to(real)
    if call != "degrid" and call != "oneshot_degrid":
        d = torch.randn((rows, chans, 2), generator=gen, device="cuda", dtype=real)
        s["vis"] = torch.view_as_complex(d)
    if case["wgt"]:
        s["wgt"] = 0.5 + torch.rand((rows, chans), generator=gen, device="cuda",
                                    dtype=torch.float32).to(real)
    if case["mask"]:
        s["mask"] = (torch.rand((rows, chans), generator=gen, device="cuda",
                                dtype=torch.float32) >= 0.05).to(torch.uint8)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if not case["call"].startswith("oneshot"):
        s["plan"] = wg.Plan(s["uvw"], s["freq"], case["nx"], case["ny"], s["pix"], s["pix"],
                            case["eps"], case["prec"], mask=s["mask"],
                            compact_index=case["compact"])
    if case["call"] == "step":
        s["img"].requires_grad_(True)
    return s


def run(s):
    c, call = s["case"], s["case"]["call"]
    if call == "degrid":
        return s["plan"].degrid(s["img"], wgt=s["wgt"])
    if call == "grid":
        return s["plan"].grid(s["vis"], wgt=s["wgt"])
    if call == "oneshot_degrid":
        return wg.dirty2ms(s["uvw"], s["freq"], s["img"], wgt=s["wgt"], pixsize_x=s["pix"],
                           pixsize_y=s["pix"], epsilon=c["eps"], mask=s["mask"])
    if call == "oneshot_grid":
        return wg.ms2dirty(s["uvw"], s["freq"], s["vis"], wgt=s["wgt"], npix_x=c["nx"],
                           npix_y=c["ny"], pixsize_x=s["pix"], pixsize_y=s["pix"],
                           epsilon=c["eps"], mask=s["mask"])
    if call == "residual":
        r = s["vis"] - s["plan"].degrid(s["img"], wgt=s["wgt"])
        return [s["plan"].grid(r, wgt=s["wgt"]), r]
    x = s["img"]
    x.grad = None
    r = autograd.degrid(x, s["plan"], s["wgt"]) - s["vis"]
    loss = 0.5 * torch.view_as_real(r).square().sum()
    loss.backward()
    return [x.grad, r.detach(), loss.detach()]


def work(case):
    """Image, visibilities, weights, mask and uvw once each, and what the w-gridding of the
    paper (Secs. 3-4) cannot do without at this accuracy, whatever the implementation: per
    visibility and direction the alpha^3 complex multiply-adds of its footprint, per w-plane one
    2-D FFT of the sigma = 1.5 oversampled image (alpha and the plane count from the accuracy and
    the field of view)."""
    nvis = _rows(case) * case["chans"]
    pix = case["nx"] * case["ny"]
    e = 4 if case["prec"] == "f32" else 8
    both = case["call"] in ("residual", "step")
    nbytes = pix * e + nvis * 2 * e + _rows(case) * 24 + (nvis * e if case["wgt"] else 0)
    nbytes += nvis if case["mask"] else 0
    if both:
        nbytes += pix * e + nvis * 2 * e + (nvis * e if case["wgt"] else 0)
    alpha = max(4, min(16, int(math.ceil(-math.log10(case["eps"]))) + 2))
    side = max(case["nx"], case["ny"])
    theta = math.radians(case["fov"])
    r2 = 0.25 * theta ** 2 * (1 + (min(case["nx"], case["ny"]) / side) ** 2)
    wmax = 0.25 * side / theta            # wavelengths: about half of the longest baseline
    planes = alpha + 1.5 * wmax * r2 / (1 + math.sqrt(1 - r2))
    cells = 2.25 * pix
    flops = (2 if both else 1) * (planes * 5 * cells * math.log2(cells) + nvis * 4.0 * alpha ** 3)
    return {"bytes": float(nbytes), "flops": float(flops)}


# ------------------------------------------------------------------------------------------
# the direct sum in 64 bits
# ------------------------------------------------------------------------------------------
# row x pixel pairs that a direct sum may take (an FP64 sine and cosine for each, twice)
_PAIRS = 8.0e9


def _cycles(a, j):
    """a * j modulo 1 for integers |j| < 2^20: a split into a part on a 2^-30 lattice, whose
    products are exact, and the rest."""
    hi = torch.round(a * 2.0 ** 30) / 2.0 ** 30
    p = torch.outer(hi, j)
    return p.sub_(torch.round(p)).add_(torch.outer(a - hi, j))


def _phases(s, rows, jx, jy, nm1):
    """Phases e^{-2 pi i [u l + v m - w (n - 1)]} of the rows and pixels at the first channel,
    and their ratio from one channel to the next (the channels are evenly spaced)."""
    c, f = s["case"], s["freq"]
    out = []
    for scale in ((f[0] / C_LIGHT,) if f.numel() == 1 else (f[0] / C_LIGHT, (f[1] - f[0]) / C_LIGHT)):
        t = s["uvw"][rows] * scale
        p = _cycles(t[:, 0] * s["pix"], jx).add_(_cycles(t[:, 1] * s["pix"], jy))
        p.sub_(torch.outer(t[:, 2], nm1))
        p.sub_(torch.round(p)).mul_(-2.0 * math.pi)
        out.append(torch.polar(torch.ones_like(p), p))
        del p
    return out[0], (out[1] if len(out) > 1 else None)


def _lm(case, pix, idx):
    jx = (idx // case["ny"] - case["nx"] // 2).double()
    jy = (idx % case["ny"] - case["ny"] // 2).double()
    r2 = (jx * pix) ** 2 + (jy * pix) ** 2
    n = torch.sqrt(1.0 - r2)
    return jx, jy, n, -r2 / (1.0 + n)


def _direct_degrid(s, img):
    """sum over the nonzero pixels, for all rows and channels"""
    c = s["case"]
    flat = img.detach().double().reshape(-1)
    idx = torch.nonzero(flat).reshape(-1)
    jx, jy, n, nm1 = _lm(c, s["pix"], idx)
    amp = (flat[idx] / n).to(torch.complex128)
    rows = s["uvw"].shape[0]
    out = torch.empty((rows, c["chans"]), dtype=torch.complex128, device="cuda")
    step = max(1, int(1.0e8) // max(1, idx.numel()))
    for r0 in range(0, rows, step):
        r = slice(r0, min(rows, r0 + step))
        p, q = _phases(s, r, jx, jy, nm1)
        for ch in range(c["chans"]):
            if ch:
                p.mul_(q)
            out[r, ch] = p @ amp
    return _weighted(s, out)


def _weighted(s, v):
    if s["wgt"] is not None:
        v = v * s["wgt"].double()
    if s["mask"] is not None:
        v = v * s["mask"].double()
    return v


def _direct_grid(s, vis):
    """sum over all rows and channels, for all pixels"""
    c = s["case"]
    d = _weighted(s, vis.to(torch.complex128))
    npix, rows = c["nx"] * c["ny"], d.shape[0]
    out = torch.empty(npix, dtype=torch.float64, device="cuda")
    step = max(1, int(1.0e8) // rows)
    for i0 in range(0, npix, step):
        idx = torch.arange(i0, min(npix, i0 + step), device="cuda")
        jx, jy, n, nm1 = _lm(c, s["pix"], idx)
        p, q = _phases(s, slice(0, rows), jx, jy, nm1)
        acc = torch.zeros(idx.numel(), dtype=torch.float64, device="cuda")
        for ch in range(c["chans"]):
            if ch:
                p.mul_(q)
            acc += (d[:, ch].conj() @ p).real      # Re(d conj(p)) = Re(conj(d) p)
        out[idx] = acc / n
    return out.reshape(c["nx"], c["ny"])


def exact(case, seed):
    rows, pix = _rows(case), case["nx"] * case["ny"]
    fwd = rows * 0.01 * pix <= _PAIRS
    adj = rows * float(pix) <= _PAIRS
    call = case["call"]
    if call in ("degrid", "oneshot_degrid"):
        if not fwd:
            return None
        s = _inputs(case, seed)
        return _direct_degrid(s, s["img"])
    if call in ("grid", "oneshot_grid"):
        if not adj:
            return None
        s = _inputs(case, seed)
        return _direct_grid(s, s["vis"])
    if not fwd:
        return None
    s = _inputs(case, seed)
    v = _direct_degrid(s, s["img"])
    if call == "residual":
        r = s["vis"].to(torch.complex128) - v
        return [_direct_grid(s, r) if adj else None, r]
    r = v - s["vis"].to(torch.complex128)
    loss = 0.5 * torch.view_as_real(r).square().sum()
    return [_direct_grid(s, r) if adj else None, r, loss]
