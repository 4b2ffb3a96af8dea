"""Workloads of the library as programs call it, through the Python entry points.

Each case is one pass of a program over data that is already on the GPU: a frame
through the catalog path, a batch of frames, forced photometry, PSF fits, the
differentiable PSF model, alignment, image subtraction, refinement of a catalog
and display maps.  `listed()` gives the fixed cases, `draw()` more of the same
ranges; `exact()` gives the results in 64-bit arithmetic, written here from the
definitions.  Inputs are synthetic star fields drawn with a seeded generator on
the device; sums of stars are formed in integers, so the same seed gives the
same frame everywhere.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2502_10783_gb300 as ipp

SIGMA = 1.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))   # sigma of a Gaussian of FWHM 1
F64 = torch.float64


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # a small ragged cut-out around a target, as an alert pipeline sends it: launches and latency
        dict(name="catalog_cutout", kind="catalog", W=517, H=389, stars=120, mesh=64, interp="keys", filter=0,
             survey=False),
        # one frame of a small camera, 64 px meshes, 500 stars
        dict(name="catalog_1k", kind="catalog", W=1024, H=1024, stars=500, mesh=64, interp="keys", filter=0,
             survey=False),
        # one survey frame: 20,000 stars, varying sky and seeing, hot pixels, cosmic rays, 128 px meshes
        dict(name="catalog_survey_4k", kind="catalog", W=4096, H=4096, stars=20000, mesh=128, interp="keys", filter=0,
             survey=True),
        # a raw camera frame: calibration, catalog, stamps at the detections and a PSF fit of each
        dict(name="raw_u16_4k", kind="raw", W=4096, H=4096, stars=8000, mesh=128, bias_map=False),
        # a night's frames of several cameras, replayed as one captured graph
        dict(name="batch_mixed", kind="batch", frames=9, scale=1.0, mesh=128, mode="streams"),
        # forced photometry: positions of a reference catalogue re-centred and measured on a new frame
        dict(name="measure_20k", kind="measure", W=4096, H=4096, sources=20000, r_ap=5.0, r_in=8.0, r_out=12.0),
        # PSF fit of every stamp of a night's reference stars
        dict(name="psf_fit_200k", kind="psf_fit", stamps=200000, S=15, model="moffat", weights=False),
        # forward and backward of the PSF model, as a training step of an image model calls it
        dict(name="psf_grad_50k", kind="psf_grad", stamps=50000, S=15, model="moffat"),
        # an exposure brought onto the pixel grid of another
        dict(name="align_4k", kind="align", W=4096, H=4096, step=32),
        # image subtraction: kernel fit on the stamps of a 10 x 10 grid, then the difference image
        dict(name="difference_4k", kind="difference", W=4096, H=4096, regions=10),
        # the catalog refined: deblending, cleaning and Kron photometry of the detections
        dict(name="refine_4k", kind="refine", W=4096, H=4096, stars=20000),
        # display maps of a large mosaic: limits, log stretch and histogram equalisation
        dict(name="display_8k", kind="display", W=8192, H=8192, nbins=4096, gray="log"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["catalog", "catalog", "raw", "batch", "measure", "psf_fit", "psf_grad", "align", "difference",
                       "refine", "display"])
    W, H = _log_int(rng, 300, 4096), _log_int(rng, 300, 4096)
    stars = max(20, int(W * H * math.exp(rng.uniform(math.log(3e-4), math.log(1.5e-3)))))
    if kind == "catalog":
        interp = rng.choice(["keys", "keys", "keys", "spline"])
        return dict(kind=kind, W=W, H=H, stars=stars, mesh=rng.choice([32, 48, 64, 128]), interp=interp,
                    filter=0 if interp == "spline" else rng.choice([0, 0, 1]), survey=rng.random() < 0.5)
    if kind == "raw":
        return dict(kind=kind, W=W, H=H, stars=min(stars, 8000), mesh=rng.choice([64, 128]),
                    bias_map=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, frames=rng.randint(2, 9), scale=round(rng.uniform(0.25, 1.0), 3),
                    mesh=rng.choice([64, 128]), mode=rng.choice(["streams", "table"]))
    if kind == "measure":
        r_ap = round(rng.uniform(2.0, 6.5), 2)
        return dict(kind=kind, W=W, H=H, sources=min(_log_int(rng, 50, 20000), W * H // 400), r_ap=r_ap, r_in=r_ap + 3.0, r_out=r_ap + 7.0)
    if kind == "psf_fit":
        return dict(kind=kind, stamps=_log_int(rng, 100, 200000), S=rng.choice([11, 13, 15, 17]),
                    model=rng.choice(["moffat", "gauss"]), weights=rng.random() < 0.3)
    if kind == "psf_grad":
        return dict(kind=kind, stamps=_log_int(rng, 64, 50000), S=rng.choice([9, 11, 15, 21, 24]),
                    model=rng.choice(["moffat", "gauss"]))
    if kind == "align":
        return dict(kind=kind, W=W, H=H, step=rng.choice([16, 32, 64]))
    if kind == "difference":
        return dict(kind=kind, W=max(W, 700), H=max(H, 700), regions=rng.randint(4, 10))
    if kind == "refine":
        return dict(kind=kind, W=W, H=H, stars=stars)
    return dict(kind="display", W=_log_int(rng, 300, 8192), H=_log_int(rng, 300, 8192),
                nbins=rng.choice([256, 1000, 4096, 16384]), gray=rng.choice(["linear", "log", "power", "exp"]))


# ------------------------------------------------------------------ the inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=F64)


def _phi(t):
    return 0.5 * (1.0 + torch.special.erf(t * math.sqrt(0.5)))


def _render(W, H, x, y, flux, sigma):
    """Pixel-integrated circular Gaussians, truncated at 6 sigma; float64 H x W."""
    img = torch.zeros(H * W, dtype=torch.int64, device="cuda")
    R = int(math.ceil(6.0 * float(sigma.max()))) + 1
    k = torch.arange(-R, R + 1, device="cuda")
    for s in range(0, x.numel(), 16384):
        xs, ys, fs, sg = (t[s:s + 16384, None] for t in (x, y, flux, sigma))
        jj, ii = torch.round(xs).long() + k, torch.round(ys).long() + k
        ex = _phi((jj + 0.5 - xs) / sg) - _phi((jj - 0.5 - xs) / sg)
        ey = _phi((ii + 0.5 - ys) / sg) - _phi((ii - 0.5 - ys) / sg)
        ex = ex * (((jj - xs).abs() <= 6 * sg) & (jj >= 0) & (jj < W))
        ey = ey * (((ii - ys).abs() <= 6 * sg) & (ii >= 0) & (ii < H)) * fs
        val = torch.round(ey[:, :, None] * ex[:, None, :] * 2.0 ** 24).long()
        at = ii.clamp(0, H - 1)[:, :, None] * W + jj.clamp(0, W - 1)[:, None, :]
        img.index_add_(0, at.reshape(-1), val.reshape(-1))
    return (img.to(F64) / 2.0 ** 24).reshape(H, W)


def _coords(W, H):
    xh = 2.0 * torch.arange(W, device="cuda", dtype=F64) / max(W - 1, 1) - 1.0
    yh = 2.0 * torch.arange(H, device="cuda", dtype=F64) / max(H - 1, 1) - 1.0
    return xh[None, :], yh[:, None]


def _noisy(g, expected):
    """Poisson counts (gain 1) plus read noise of 5 ADU."""
    n = torch.randn(expected.shape, generator=g, device="cuda", dtype=torch.float32)
    return torch.poisson(expected.clamp_min(0.0).float(), generator=g) + 5.0 * n


def _field(W, H, stars, seed, survey, sky=1000.0):
    """A frame and the stars in it.  survey: quadratic sky, FWHM 2.5 to 4 px along
    x, fluxes dN/dF ~ F^-1.5 on [1e2, 1e6], hot pixels and cosmic rays; else a
    linear sky, FWHM 3 px and log-uniform fluxes 10^2.5 .. 10^5."""
    g = _gen(seed)
    x, y, u = _rand(g, stars, hi=W), _rand(g, stars, hi=H), _rand(g, stars)
    xh, yh = _coords(W, H)
    if survey:
        flux = (1e-1 - u * (1e-1 - 1e-3)) ** -2.0
        fwhm = 2.5 + 1.5 * x / max(W - 1, 1)
        reach = min(1.0, max(W, H) / 4096.0) ** 2   # a cut-out sees its part of the same sky
        base = sky + 0.2 * sky * reach * (xh ** 2 + yh ** 2 - 1.0)
    else:
        flux = 10.0 ** (2.5 + 2.5 * u)
        fwhm = torch.full_like(x, 3.0)
        base = (sky + 0.05 * sky * min(1.0, W / 1024.0) * xh).expand(H, W)
    img = _noisy(g, base + _render(W, H, x, y, flux, fwhm * SIGMA))
    if survey:
        hot = torch.unique(torch.randint(0, W * H, (max(1, W * H // 10000),), generator=g, device="cuda"))
        img.view(-1)[hot] = (base.reshape(-1)[hot] + 5e4).float()
        cosmic = torch.zeros(H, W, dtype=torch.bool, device="cuda")
        n = max(1, W * H // 84000)
        cx, cy, ang = _rand(g, n, hi=W), _rand(g, n, hi=H), _rand(g, n, hi=2.0 * math.pi)
        length = _rand(g, n, lo=1.0, hi=10.0)
        for t in range(11):
            on = t <= length
            j = torch.round(cx + t * torch.cos(ang)).long().clamp(0, W - 1)[on]
            i = torch.round(cy + t * torch.sin(ang)).long().clamp(0, H - 1)[on]
            cosmic[i, j] = True
        img = img + 1e4 * cosmic
    return img.float().contiguous(), (x, y, flux)


def _raw(case, seed):
    """A raw frame: bias 500 ADU, radial flat 1.1 - 0.2 r^2, rounded to uint16."""
    W, H = case["W"], case["H"]
    img, _ = _field(W, H, case["stars"], seed, False)
    xh, yh = _coords(W, H)
    flat = (1.1 - 0.1 * (xh ** 2 + yh ** 2)).float()
    bias = torch.full((H, W), 500.0, device="cuda")
    if case["bias_map"]:
        bias = bias + 2.0 * torch.randn(H, W, generator=_gen(seed + 1), device="cuda")
    raw = torch.round(bias + flat * img).clamp(0, 65535).int()
    return raw.to(torch.uint16), (1.0 / flat).contiguous(), bias if case["bias_map"] else None


def _batch_sizes(case):
    table = [(1024, 1024), (4096, 4096), (2048, 2048), (6144, 6160)]
    s = case["scale"]
    return [(int(w * s), int(h * s)) for w, h in (table[i % 4] for i in range(case["frames"]))]


def _batch_frames(case, seed):
    out = []
    for i, (W, H) in enumerate(_batch_sizes(case)):
        stars = int(W * H * (5e-4, 1.2e-3, 8e-4)[i % 3])
        out.append(_field(W, H, stars, seed * 64 + i, False, sky=(200.0, 1000.0, 3000.0)[i % 3])[0])
    return out


def _stamps(case, seed):
    """Stamps of elliptical Moffat stars (beta 2.5, widths 1-2 px) averaged over 3 x 3
    samples a pixel, fluxes dN/dF ~ F^-1.5 on [1e2, 1e6], Poisson and read noise."""
    n, S = case["stamps"], case["S"]
    g = _gen(seed)
    c = (S - 1) / 2.0
    x, y = _rand(g, n, lo=c - 0.5, hi=c + 0.5), _rand(g, n, lo=c - 0.5, hi=c + 0.5)
    flux = (1e-1 - _rand(g, n) * (1e-1 - 1e-3)) ** -2.0
    sky, ax, ay = _rand(g, n, lo=800.0, hi=1200.0), _rand(g, n, lo=1.0, hi=2.0), _rand(g, n, lo=1.0, hi=2.0)
    th = _rand(g, n, hi=math.pi)
    out = torch.empty(n, S, S, device="cuda")
    px = torch.arange(S, device="cuda", dtype=torch.float32)
    t = [v.float()[:, None, None] for v in (x, y, flux, sky, ax, ay, torch.cos(th), torch.sin(th))]
    for s in range(0, n, 32768):
        X, Y, F, B, A, D, co, si = (v[s:s + 32768] for v in t)
        m = torch.zeros_like(out[s:s + 32768])
        for oy in (-1 / 3, 0.0, 1 / 3):
            for ox in (-1 / 3, 0.0, 1 / 3):
                dx, dy = px[None, None, :] + ox - X, px[None, :, None] + oy - Y
                u, v = (co * dx + si * dy) / A, (co * dy - si * dx) / D
                m += (1.0 + u * u + v * v) ** -2.5
        out[s:s + 32768] = _noisy(g, B + F * (1.5 / math.pi / 9.0) / (A * D) * m)
    w = None
    if case.get("weights"):
        w = (1.0 / (out.clamp_min(1.0) + 25.0)).contiguous()
        w.view(-1)[torch.randint(0, w.numel(), (n,), generator=g, device="cuda")] = 0.0   # bad pixels
    return out, w


def _psf_params(case, seed):
    n, S = case["stamps"], case["S"]
    g = _gen(seed)
    c = (S - 1) / 2.0
    col = [(c - 1, c + 1), (100.0, 1e5), (-20.0, 20.0), (1.2, 2.5), (0.8, 1.9), (-1.5, 1.5)]
    p = [_rand(g, n, lo=a, hi=b) for a, b in [col[0]] + col]
    grad = torch.randn(n, S, S, generator=g, device="cuda")
    return torch.stack(p, 1).float().contiguous(), grad


def _wcs_pair(W, H, seed):
    """Headers of two exposures of one field: 1.5 arcsec pixels, SIP of order 3 with
    a few pixels at the corners, 0.02-0.05 degrees and up to half a degree apart."""
    rng = np.random.default_rng(seed)
    s, half = 1.5 / 3600.0, max(W, H) / 2.0

    def one(ra, dec, rot, k):
        a, b = np.zeros((6, 6)), np.zeros((6, 6))
        for p in range(4):
            for q in range(4 - p):
                if p + q >= 2:
                    a[p, q], b[p, q] = rng.normal(0.0, 2.0, 2) * half ** float(-p - q)
        c, n = math.cos(rot), math.sin(rot)
        return dict(crpix=[W / 2 + 0.5 + k, H / 2 + 0.5 - k], crval=[ra, dec], cd=[[-s * c, s * n], [s * n, s * c]],
                    a=a, b=b, a_order=3, b_order=3)

    ra, dec = rng.uniform(0.0, 360.0), rng.uniform(-60.0, 60.0)
    shift = min(1.0, half / 2048.0)
    src = one(ra, dec, rng.uniform(-0.01, 0.01), 0.0)
    return src, one(ra + shift * rng.uniform(0.02, 0.05) / math.cos(math.radians(dec)),
                    dec - shift * rng.uniform(0.02, 0.05), math.radians(rng.uniform(0.2, 0.5)), 3.25)


def _blur(img, sigma):
    k = torch.exp(-0.5 * (torch.arange(-8, 9, device="cuda", dtype=F64) / sigma) ** 2)
    k = (k / k.sum()).tolist()
    for d in (0, 1):
        img = sum(w * torch.roll(img, i - 8, d) for i, w in enumerate(k))
    return img


def _pair(case, seed):
    """A template and a frame of the same field: blurred, dimmer, on another sky, with its own noise."""
    W, H = case["W"], case["H"]
    g = _gen(seed)
    n = max(400, int(W * H * 1.2e-3))
    x, y = _rand(g, n, hi=W), _rand(g, n, hi=H)
    stars = _render(W, H, x, y, 10.0 ** _rand(g, n, lo=3.0, hi=5.5), torch.full_like(x, 2.6 * SIGMA))
    noise = torch.randn(2, H, W, generator=g, device="cuda")
    tmpl = (stars + 100.0).float() + 3.0 * noise[0]
    img = (0.9 * _blur(stars + 100.0, 1.1) + 30.0).float() + 3.0 * noise[1]
    return img.contiguous(), tmpl.contiguous()


def _mosaic(case, seed):
    W, H = case["W"], case["H"]
    g = _gen(seed)
    img = torch.exp(0.3 * torch.randn(H, W, generator=g, device="cuda")) * 1000.0
    img += (200.0 * _coords(W, H)[0]).float()
    bright = torch.randint(0, W * H, (W * H // 200 + 1,), generator=g, device="cuda")
    img.view(-1)[bright] = 2e4
    if W > 700 and H > 700:
        img[300:340, 500:600] = float("nan")   # a dead block of the detector
    return img


def _bg(case):
    return ipp.BgConfig(mesh=case.get("mesh", 128), interp=case.get("interp", "keys"))


def _zero(*dicts):
    for d in dicts:
        for t in d.values():
            t.zero_()   # rows beyond the catalog are never written


def prepare(case, seed):
    kind = case["kind"]
    if kind == "catalog":
        img, _ = _field(case["W"], case["H"], case["stars"], seed, case["survey"])
        ex = ipp.Extractor(case["W"], case["H"], _bg(case), filter=case["filter"])
        _zero(ex.out, ex.stats)
        return dict(kind=kind, img=img, ex=ex)
    if kind == "raw":
        raw, inv_flat, bias = _raw(case, seed)
        ex = ipp.Extractor(case["W"], case["H"], _bg(case))
        n = ex.max_src
        fit = dict(params=torch.zeros(n, 7, device="cuda"), chi2=torch.zeros(n, device="cuda"),
                   iters=torch.zeros(n, dtype=torch.int32, device="cuda"),
                   flags=torch.zeros(n, dtype=torch.int32, device="cuda"))
        _zero(ex.out, ex.stats)
        return dict(kind=kind, raw=raw, calib=(inv_flat, 500.0) if bias is None else (inv_flat, 500.0, bias), ex=ex,
                    fit=fit)
    if kind == "batch":
        b = ipp.Batch(_batch_frames(case, seed), lanes=8, cfg=_bg(case), max_src=65536, mode=case["mode"])
        for o, s in zip(b.outs, b.stats):
            _zero(o, s)
        b.run()
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        b.capture(stream)
        torch.cuda.current_stream().wait_stream(stream)
        return dict(kind=kind, batch=b)
    if kind == "measure":
        img, (x, y, flux) = _field(case["W"], case["H"], case["sources"], seed, False)
        g = _gen(seed + 7)
        sub = img - 1000.0
        x0 = (x + 0.3 * torch.randn(x.shape, generator=g, device="cuda", dtype=F64)).float()
        y0 = (y + 0.3 * torch.randn(x.shape, generator=g, device="cuda", dtype=F64)).float()
        return dict(kind=kind, sub=sub, x0=x0, y0=y0,
                    n=torch.tensor([x0.numel()], dtype=torch.int32, device="cuda"),
                    phot=dict(r_ap=case["r_ap"], r_in=case["r_in"], r_out=case["r_out"]))
    if kind == "psf_fit":
        stamps, w = _stamps(case, seed)
        return dict(kind=kind, stamps=stamps, weights=w, model=_model(case))
    if kind == "psf_grad":
        p, grad = _psf_params(case, seed)
        return dict(kind=kind, params=p.requires_grad_(True), grad=grad, S=case["S"], model=_model(case))
    if kind == "align":
        img, _ = _field(case["W"], case["H"], max(50, case["W"] * case["H"] // 1000), seed, False)
        src, tgt = _wcs_pair(case["W"], case["H"], seed)
        return dict(kind=kind, img=img, src=src, tgt=tgt, W=case["W"], H=case["H"], step=case["step"])
    if kind == "difference":
        img, tmpl = _pair(case, seed)
        return dict(kind=kind, img=img, tmpl=tmpl, n=case["regions"])
    if kind == "refine":
        W, H = case["W"], case["H"]
        img, _ = _field(W, H, case["stars"], seed, True)
        cfg = ipp.BgConfig(mesh=128)
        ex = ipp.Extractor(W, H, cfg)
        o = ex(img)
        need = ex.L.ipp_deblend_workspace_size(W, H, ex.max_src)
        return dict(kind=kind, sub=o["sub"], labels=o["labels"], n=o["n_src"], stats=ex.stats, rms=o["mesh_rms"],
                    cfg=cfg, rows=torch.arange(ex.max_src, device="cuda"), max_obj=2 * ex.max_src,
                    ws=torch.empty(need, dtype=torch.uint8, device="cuda"))
    img = _mosaic(case, seed)
    return dict(kind="display", img=img, nbins=case["nbins"], gray=_GRAY[case["gray"]])


_GRAY = {"linear": (ipp.GRAY_LINEAR, 1.0), "log": (ipp.GRAY_LOG, 1000.0), "power": (ipp.GRAY_POWER, 0.5),
         "exp": (ipp.GRAY_EXP, 1000.0)}
_LO, _HI = 400.0, 4000.0   # display limits of the stretch


def _model(case):
    return ipp.PSF_GAUSS if case["model"] == "gauss" else ipp.PSF_MOFFAT


def run(s):
    kind = s["kind"]
    if kind == "catalog":
        return dict(s["ex"](s["img"]), stats=s["ex"].stats)
    if kind == "raw":
        ex = s["ex"]
        o = ex(s["raw"], s["calib"])
        cut = ipp.stamp_cut(o["sub"], o["x"], o["y"], n_src=o["n_src"], S=15)
        fit = ipp.psf_fit(cut["stamps"], weights=cut["weights"], n_src=o["n_src"], out=s["fit"])
        return dict(o, stats=ex.stats, fit=fit)
    if kind == "batch":
        outs, stats = s["batch"].launch(), s["batch"].stats
        return [dict(sub=o["sub"], labels=o["labels"], n=o["n_src"], x=o["x"], y=o["y"], flux=o["flux"], iso=t["flux"])
                for o, t in zip(outs, stats)]
    if kind == "measure":
        x, y, it, fl = ipp.centroid(s["sub"], s["x0"], s["y0"], n_src=s["n"])
        return dict(ipp.aperture_phot(s["sub"], x, y, n_src=s["n"], **s["phot"]), x=x, y=y, iters=it, cen_flags=fl)
    if kind == "psf_fit":
        return ipp.psf_fit(s["stamps"], weights=s["weights"], model=s["model"])
    if kind == "psf_grad":
        m = ipp.psf_model(s["params"], s["S"], s["model"])
        (g,) = torch.autograd.grad(m, s["params"], s["grad"])
        return dict(model=m, grad=g)
    if kind == "align":
        out, M, status = ipp.align(s["img"], s["src"], s["tgt"], s["W"], s["H"], step=s["step"])
        return dict(image=out, M=M, status=status)
    if kind == "difference":
        fit = ipp.sub_fit(s["img"], s["tmpl"], nsx=s["n"], nsy=s["n"])
        d = ipp.sub_apply(s["img"], s["tmpl"], fit["coef"])
        return dict(diff=d, coef64=fit["coef64"], coef=fit["coef"], n=fit["n"], status=fit["status"])
    if kind == "refine":
        deb, n = ipp.deblend(s["sub"], s["labels"], s["n"], s["stats"], ws=s["ws"])
        cleaned, n2 = ipp.clean(s["sub"], deb, n, s["max_obj"], mesh_rms=s["rms"], cfg=s["cfg"])
        auto = ipp.auto_phot(s["sub"], s["labels"], s["n"], s["stats"])
        live = s["rows"] < s["n"]   # the count stays on the device: rows beyond it are cleared
        auto = {k: torch.where(live if v.dim() == 1 else live[:, None], v, 0) for k, v in auto.items()}
        return dict(deblended=deb, n_deblended=n, cleaned=cleaned, n_cleaned=n2, auto=auto)
    z, cnt = ipp.zscale(s["img"])
    kind, a = s["gray"]
    g = ipp.gray_transform(s["img"], kind, _LO, _HI, a)
    eq, _ = ipp.hist_equalize(s["img"], nbins=s["nbins"])
    return dict(z=z, counts=cnt, gray=g, equalized=eq)


def work(case):
    """Each input read once, each output written once; the operations of the definitions."""
    kind = case["kind"]
    px = case.get("W", 0) * case.get("H", 0)
    if kind == "catalog":   # frame in, subtracted frame and label map out; about 40 operations a pixel
        return dict(bytes=12.0 * px + 100.0 * case["stars"], flops=40.0 * px + 6e3 * case["stars"])
    if kind == "raw":
        n = 1.7 * case["stars"]   # noise islands pass the threshold too
        return dict(bytes=(14.0 + 4.0 * case["bias_map"]) * px + 150.0 * n, flops=45.0 * px + n * (6e3 + 10 * 225 * 110))
    if kind == "batch":
        px = sum(w * h for w, h in _batch_sizes(case))
        return dict(bytes=12.0 * px + 0.08 * px, flops=45.0 * px)
    if kind == "measure":   # a 25 x 25 box of each source
        n, b = case["sources"], 2 * case["r_out"] + 1
        return dict(bytes=n * (4.0 * min(b * b, px / n) + 44.0), flops=n * 6e3)
    if kind == "psf_fit":   # about ten evaluations of model and Jacobian a stamp
        n, p = case["stamps"], case["S"] ** 2
        return dict(bytes=n * (4.0 * p * (2 if case["weights"] else 1) + 40.0), flops=n * 10.0 * p * 110)
    if kind == "psf_grad":
        n, p = case["stamps"], case["S"] ** 2
        return dict(bytes=n * (8.0 * p + 84.0), flops=n * 80.0 * p)
    if kind == "align":
        return dict(bytes=8.0 * px, flops=20.0 * px)
    if kind == "difference":   # 441 taps a pixel
        return dict(bytes=12.0 * px, flops=882.0 * px)
    if kind == "refine":
        return dict(bytes=16.0 * px, flops=100.0 * px)
    return dict(bytes=12.0 * px, flops=20.0 * px)


# -------------------------------------------------------- results in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind == "catalog":
        img, _ = _field(case["W"], case["H"], case["stars"], seed, case["survey"])
        return _catalog64(img.to(F64), case)
    if kind == "raw":
        raw, inv_flat, bias = _raw(case, seed)
        f = (raw.int().to(F64) - (500.0 if bias is None else bias.to(F64))) * inv_flat.to(F64)
        return _catalog64(f, case)
    if kind == "batch":
        return [dict(sub=_catalog64(f.to(F64), case)["sub"]) for f in _batch_frames(case, seed)]
    if kind == "measure":
        return _measure64(case, seed)
    if kind == "psf_fit":
        # fits of faint stamps that reach the iteration limit end anywhere in a flat
        # valley: their chi^2 is defined there, their parameters are not
        return dict(_fit64(case, *_stamps(case, seed)), params=None)
    if kind == "psf_grad":
        p, grad = _psf_params(case, seed)
        p = p.to(F64).requires_grad_(True)
        m = _model64(p, case)
        (g,) = torch.autograd.grad(m, p, grad.to(F64))
        return dict(model=m.detach(), grad=g)
    if kind == "align":
        return _align64(case, seed)
    if kind == "difference":
        return dict(diff=_difference64(case, *_pair(case, seed)))
    if kind == "refine":
        s = prepare(case, seed)   # the detections are this case's input
        return dict(auto=_auto64(s))
    return _display64(case, seed)


def _clip64(f, mesh):
    """Mesh background 2.5 median - 1.5 mean and sigma of the 3-sigma clipped set."""
    H, W = f.shape
    ny, nx = -(-H // mesh), -(-W // mesh)
    p = torch.full((ny * mesh, nx * mesh), float("nan"), dtype=F64, device=f.device)
    p[:H, :W] = f
    v = p.reshape(ny, mesh, nx, mesh).permute(0, 2, 1, 3).reshape(ny * nx, mesh * mesh).sort(1).values
    n0 = torch.isfinite(v).sum(1)
    c0 = v.gather(1, (n0.clamp_min(1)[:, None] - 1) // 2)
    d = torch.nan_to_num(v - c0)
    z = torch.zeros_like(c0)
    s1, s2 = torch.cat([z, d.cumsum(1)], 1), torch.cat([z, (d * d).cumsum(1)], 1)
    v = torch.nan_to_num(v, nan=float("inf"))
    lo, hi = torch.zeros_like(n0)[:, None], n0[:, None]

    def stats():
        n = (hi - lo).clamp_min(1)
        med = 0.5 * (v.gather(1, (lo + (n - 1) // 2)) + v.gather(1, (lo + n // 2).clamp_max(v.shape[1] - 1)))
        mean = (s1.gather(1, hi) - s1.gather(1, lo)) / n
        var = (s2.gather(1, hi) - s2.gather(1, lo)) / n - mean * mean
        return med, c0 + mean, var.clamp_min(0.0).sqrt()

    for _ in range(10):
        med, mean, sd = stats()
        a = torch.searchsorted(v, med - 3.0 * sd, right=False).maximum(lo)
        b = torch.searchsorted(v, med + 3.0 * sd, right=True).minimum(hi)
        if bool(((a == lo) & (b == hi)).all()):
            break
        lo, hi = a, b
    med, mean, sd = stats()
    ok = (n0 >= 100).reshape(ny, nx).cpu().numpy()
    bkg, rms = ((t.reshape(ny, nx).cpu().numpy()) for t in (2.5 * med - 1.5 * mean, sd))
    grids = []
    for g in (bkg, rms):
        full = g.copy()
        for i, j in zip(*np.nonzero(~ok)):   # the valid nodes nearest to an invalid one
            for k in range(1, max(nx, ny)):
                w = np.s_[max(i - k, 0):i + k + 1, max(j - k, 0):j + k + 1]
                if ok[w].any():
                    full[i, j] = np.median(g[w][ok[w]])
                    break
        q = np.full((ny + 2, nx + 2), np.nan)
        q[1:-1, 1:-1] = full
        w = np.stack([q[a:a + ny, b:b + nx] for a in range(3) for b in range(3)])
        grids.append(torch.from_numpy(np.nanmedian(w, 0)).to(f.device))
    return grids


def _keys_rows(n_px, n, mesh):
    """[n_px, n]: Keys cubic convolution weights of the nodes, indices clamped."""
    u = (np.arange(n_px) + 0.5) / mesh - 0.5
    q = np.floor(u).astype(int)
    s = u - q
    w = [-0.5 * s ** 3 + s ** 2 - 0.5 * s, 1.5 * s ** 3 - 2.5 * s ** 2 + 1.0, -1.5 * s ** 3 + 2.0 * s ** 2 + 0.5 * s,
         0.5 * s ** 3 - 0.5 * s ** 2]
    A = np.zeros((n_px, n))
    for b in range(4):
        np.add.at(A, (np.arange(n_px), np.clip(q - 1 + b, 0, n - 1)), w[b])
    return torch.from_numpy(A).cuda()


def _spline_rows(n_px, n, mesh):
    """[n_px, n]: natural cubic spline through the nodes, continued as a line."""
    u = (np.arange(n_px) + 0.5) / mesh - 0.5
    if n == 1:
        return torch.ones(n_px, 1, dtype=F64, device="cuda")
    second = np.zeros((n, n))   # node values -> second derivatives
    if n > 2:
        T = 4.0 * np.eye(n - 2) + np.eye(n - 2, k=1) + np.eye(n - 2, k=-1)
        D = np.zeros((n - 2, n))
        for i in range(n - 2):
            D[i, i:i + 3] = 6.0, -12.0, 6.0
        second[1:-1] = np.linalg.solve(T, D)
    q = np.clip(np.floor(u).astype(int), 0, n - 2)
    t = u - q
    E, Q = np.eye(n), second
    b, a = t[:, None], 1.0 - t[:, None]
    inside = a * E[q] + b * E[q + 1] + ((a ** 3 - a) * Q[q] + (b ** 3 - b) * Q[q + 1]) / 6.0
    first = E[0] + u[:, None] * (E[1] - E[0] - (2.0 * Q[0] + Q[1]) / 6.0)
    last = E[n - 1] + (u - (n - 1))[:, None] * (E[n - 1] - E[n - 2] + (Q[n - 2] + 2.0 * Q[n - 1]) / 6.0)
    A = np.where((u < 0)[:, None], first, np.where((u > n - 1)[:, None], last, inside))
    return torch.from_numpy(A).cuda()


def _catalog64(f, case):
    H, W = f.shape
    mesh = case["mesh"]
    bkg, rms = _clip64(f, mesh)
    rows = _spline_rows if case.get("interp") == "spline" else _keys_rows
    ref = bkg[0, 0]
    B = ref + rows(H, bkg.shape[0], mesh) @ (bkg - ref) @ rows(W, bkg.shape[1], mesh).T
    return dict(mesh_bkg=bkg, mesh_rms=rms, sub=f - B)


def _beyond(x, y, r):
    """Area of the disk of radius r about the origin in the quadrant X >= x, Y >= y."""
    def corner(u, v):   # u, v >= 0
        a, b = (r * r - u * u).clamp_min(0.0).sqrt(), (r * r - v * v).clamp_min(0.0).sqrt()
        phi = torch.atan2(a * b - u * v, u * b + a * v)
        k = 0.5 * ((a - v) * (b - u) + r * r * phi - (a * b - u * v))
        return torch.where(u * u + v * v < r * r, k, torch.zeros_like(k))
    z = torch.zeros_like(x)
    ax, ay = x.abs(), y.abs()
    k, hx, hy = corner(ax, ay), 2.0 * corner(ax, z), 2.0 * corner(z, ay)
    out = torch.where(x >= 0, torch.where(y >= 0, k, hx - k), torch.where(y >= 0, hy - k, math.pi * r * r - hx - hy + k))
    return out


def _boxes(img, x, y, R):
    """Offsets, values and in-frame flags of the boxes around rint(x), rint(y)."""
    H, W = img.shape
    k = torch.arange(-R, R + 1, device=img.device)
    jj, ii = torch.round(x).long()[:, None, None] + k[None, None, :], torch.round(y).long()[:, None, None] + k[None, :, None]
    ok = (ii >= 0) & (ii < H) & (jj >= 0) & (jj < W)
    v = img.reshape(-1)[(ii.clamp(0, H - 1) * W + jj.clamp(0, W - 1))]
    return jj - x[:, None, None], ii - y[:, None, None], torch.where(ok, v, torch.zeros_like(v)), ok


def _measure64(case, seed):
    s = prepare(case, seed)
    img = s["sub"].to(F64)
    sw = 3.0 / 2.35482
    rad = 4.0 * sw
    parts = []
    for lo in range(0, s["x0"].numel(), 4096):
        x, y = s["x0"][lo:lo + 4096].to(F64), s["y0"][lo:lo + 4096].to(F64)
        sx, sy = x.clone(), y.clone()
        live = torch.ones_like(x, dtype=torch.bool)
        for _ in range(16):
            dx, dy, v, ok = _boxes(img, x, y, int(rad + 0.5))
            d2 = dx * dx + dy * dy
            w = torch.exp(-d2 / (2.0 * sw * sw)) * (d2 < rad * rad) * ok * v
            s0 = w.sum((1, 2))
            ddx, ddy = 2.0 * (w * dx).sum((1, 2)) / s0, 2.0 * (w * dy).sum((1, 2)) / s0
            bad = live & ~(s0 > 0)
            x, y = torch.where(bad, sx, x), torch.where(bad, sy, y)
            live = live & ~bad
            x, y = torch.where(live, x + ddx, x), torch.where(live, y + ddy, y)
            live = live & ~(ddx * ddx + ddy * ddy < 1e-8)
        r, R = case["r_ap"], int(case["r_out"] + 1.5)
        dx, dy, v, ok = _boxes(img, x, y, R)
        x0, x1, y0, y1 = dx - 0.5, dx + 0.5, dy - 0.5, dy + 0.5
        w = (_beyond(*torch.broadcast_tensors(x0, y0), r) - _beyond(*torch.broadcast_tensors(x1, y0), r)
             - _beyond(*torch.broadcast_tensors(x0, y1), r) + _beyond(*torch.broadcast_tensors(x1, y1), r)) * ok
        d2 = dx * dx + dy * dy
        ring = ok & (d2 >= case["r_in"] ** 2) & (d2 < case["r_out"] ** 2)
        a = torch.where(ring, v, torch.full_like(v, float("inf"))).flatten(1).sort(1).values
        n = ring.flatten(1).sum(1, keepdim=True)
        sky = 0.5 * (a.gather(1, ((n - 1) // 2).clamp_min(0)) + a.gather(1, n // 2))[:, 0]
        sky = torch.where(n[:, 0] >= 10, sky, torch.zeros_like(sky))
        area = w.sum((1, 2))
        parts.append((x, y, (w * v).sum((1, 2)) - sky * area, sky, area))
    x, y, flux, sky, area = (torch.cat(t) for t in zip(*parts))
    return dict(x=x, y=y, flux=flux, sky=sky, area=area)


def _pix64(S, dev="cuda"):
    k = torch.arange(S, dtype=F64, device=dev)
    return k.repeat(S)[None, :], k.repeat_interleave(S)[None, :]


def _model64(p, case):
    S = case["S"]
    j, i = _pix64(S, p.device)
    x0, y0, F, sky, sx, sy, th = (p[:, k:k + 1] for k in range(7))
    dx, dy = j - x0, i - y0
    u, v = torch.cos(th) * dx + torch.sin(th) * dy, torch.cos(th) * dy - torch.sin(th) * dx
    q = (u / sx) ** 2 + (v / sy) ** 2
    if case["model"] == "gauss":
        m = F / (2.0 * math.pi * sx * sy) * torch.exp(-0.5 * q)
    else:
        m = F * 1.5 / (math.pi * sx * sy) * (1.0 + q) ** -2.5
    return (m + sky).reshape(-1, S, S)


def _jac64(p, case):
    """Model and its seven derivatives, [n, pixels] and [n, pixels, 7]."""
    j, i = _pix64(case["S"], p.device)
    x0, y0, F, sky, sx, sy, th = (p[:, k:k + 1] for k in range(7))
    c, s = torch.cos(th), torch.sin(th)
    dx, dy = j - x0, i - y0
    u, v = c * dx + s * dy, c * dy - s * dx
    q = (u / sx) ** 2 + (v / sy) ** 2
    if case["model"] == "gauss":
        A = torch.exp(-0.5 * q) / (2.0 * math.pi * sx * sy)
        D = -0.5 * F * A
    else:
        A = 1.5 / (math.pi * sx * sy) * (1.0 + q) ** -2.5
        D = -2.5 * F * A / (1.0 + q)
    P = F * A
    qu, qv = 2.0 * u / sx ** 2, 2.0 * v / sy ** 2
    J = [D * (-qu * c + qv * s), D * (-qu * s - qv * c), A, torch.ones_like(P), -P / sx - D * 2.0 * u * u / sx ** 3,
         -P / sy - D * 2.0 * v * v / sy ** 3, D * 2.0 * u * v * (1.0 / sx ** 2 - 1.0 / sy ** 2)]
    return P + sky, torch.stack(J, 2), P


def _fit64(case, stamps, weights):
    """The Levenberg-Marquardt fit as documented, in 64 bits."""
    S = case["S"]
    out_p, out_c = [], []
    for lo in range(0, stamps.shape[0], 16384):
        z = stamps[lo:lo + 16384].to(F64)
        n = z.shape[0]
        edge = torch.cat([z[:, 0], z[:, -1], z[:, 1:-1, 0], z[:, 1:-1, -1]], 1).sort(1).values
        m = edge.shape[1]
        sky = 0.5 * (edge[:, (m - 1) // 2] + edge[:, m // 2])
        z = z.reshape(n, -1)
        W = torch.ones_like(z) if weights is None else weights[lo:lo + 16384].to(F64).reshape(n, -1)
        c = torch.full((n,), (S - 1) / 2.0, dtype=F64, device=z.device)
        p = torch.stack([c, c, (z - sky[:, None]).sum(1), sky, 0 * c + 1.6, 0 * c + 1.4, 0 * c], 1)

        def at(p):
            mod, J, P = _jac64(p, case)
            r = z - mod
            JW = J * W[:, :, None]
            return (JW.transpose(1, 2) @ J, (JW.transpose(1, 2) @ r[:, :, None])[:, :, 0], (W * r * r).sum(1),
                    (W * P * P).sum(1))

        def solve(Hm, g, lam):
            d = torch.diagonal(Hm, dim1=1, dim2=2)
            D = torch.maximum(d, 1e-9 * d.max(1, keepdim=True).values)
            L, info = torch.linalg.cholesky_ex(Hm + torch.diag_embed(lam[:, None] * D))
            x = torch.cholesky_solve(g[:, :, None], L)[:, :, 0]
            return torch.where((info == 0)[:, None], x, torch.zeros_like(x)), info == 0

        Hm, g, chi, star = at(p)
        lam = torch.full_like(chi, 1e-3)
        it = torch.zeros(n, dtype=torch.int64, device=z.device)
        live = torch.ones(n, dtype=torch.bool, device=z.device)
        for _ in range(51):
            if not bool(live.any()):
                break
            x, ok = solve(Hm, g, lam)
            gn, ok0 = solve(Hm, g, torch.zeros_like(lam))
            thr = 1e-10 * chi + 1e-12 * star
            done = live & ok & ok0 & ((g * x).sum(1) <= thr) & ((g * gn).sum(1) <= thr)
            live = live & ~done
            t = p + x
            good = ok & (t[:, 4] > 0.05) & (t[:, 5] > 0.05)
            t = torch.where((live & good)[:, None], t, p)
            H2, g2, c2, s2 = at(t)
            take = live & good & (c2 < chi)
            p, Hm, g = torch.where(take[:, None], t, p), torch.where(take[:, None, None], H2, Hm), torch.where(take[:, None], g2, g)
            chi, star = torch.where(take, c2, chi), torch.where(take, s2, star)
            lam = torch.where(live, torch.where(take, lam / 10.0, lam * 10.0), lam)
            it = it + live
            live = live & (lam <= 1e10) & (it < 50)
        swap = p[:, 4] < p[:, 5]
        sx, sy = torch.maximum(p[:, 4], p[:, 5]), torch.minimum(p[:, 4], p[:, 5])
        th = p[:, 6] + 0.5 * math.pi * swap
        th = th - math.pi * torch.floor((th + 0.5 * math.pi) / math.pi)
        out_p.append(torch.stack([p[:, 0], p[:, 1], p[:, 2], p[:, 3], sx, sy, th], 1))
        out_c.append(chi)
    return dict(params=torch.cat(out_p), chi2=torch.cat(out_c))


def _sip(w, u, v):
    f, g = np.zeros_like(u), np.zeros_like(u)
    for p in range(4):
        for q in range(4 - p):
            f, g = f + w["a"][p, q] * u ** p * v ** q, g + w["b"][p, q] * u ** p * v ** q
    return f, g


def _align64(case, seed):
    W, H, step = case["W"], case["H"], case["step"]
    img, _ = _field(W, H, max(50, W * H // 1000), seed, False)
    src, tgt = _wcs_pair(W, H, seed)
    y, x = np.mgrid[0:H:step, 0:W:step].astype(float)
    u, v = x + 1.0 - src["crpix"][0], y + 1.0 - src["crpix"][1]
    f, g = _sip(src, u, v)
    cd = np.radians(np.array(src["cd"]))
    p, q = cd[0, 0] * (u + f) + cd[0, 1] * (v + g), cd[1, 0] * (u + f) + cd[1, 1] * (v + g)
    a0, d0 = np.radians(src["crval"])
    den = np.cos(d0) - q * np.sin(d0)
    ra, dec = a0 + np.arctan2(p, den), np.arctan2(np.sin(d0) + q * np.cos(d0), np.hypot(p, den))
    a1, d1 = np.radians(tgt["crval"])
    c = np.sin(d1) * np.sin(dec) + np.cos(d1) * np.cos(dec) * np.cos(ra - a1)
    xi = np.cos(dec) * np.sin(ra - a1) / c
    eta = (np.cos(d1) * np.sin(dec) - np.sin(d1) * np.cos(dec) * np.cos(ra - a1)) / c
    inv = np.linalg.inv(np.radians(np.array(tgt["cd"])))
    X, Y = inv[0, 0] * xi + inv[0, 1] * eta, inv[1, 0] * xi + inv[1, 1] * eta
    U, V = X.copy(), Y.copy()
    for _ in range(60):   # the distortion is a few pixels: a contraction
        f, g = _sip(tgt, U, V)
        U, V = X - f, Y - g
    xt, yt = (U + tgt["crpix"][0] - 1.0).ravel(), (V + tgt["crpix"][1] - 1.0).ravel()
    xs, ys = x.ravel(), y.ravel()
    mx, my, ux, uy = xs.mean(), ys.mean(), xt.mean(), yt.mean()
    dx, dy, ex, ey = xs - mx, ys - my, xt - ux, yt - uy
    nrm = (dx * dx + dy * dy).sum()
    a, b = (dx * ex + dy * ey).sum() / nrm, (dx * ey - dy * ex).sum() / nrm
    tx, ty = ux - a * mx + b * my, uy - b * mx - a * my
    d = a * a + b * b
    Mi = [a / d, b / d, -(a * tx + b * ty) / d, -b / d, a / d, (b * tx - a * ty) / d]
    M = torch.tensor([a, -b, tx, b, a, ty] + Mi, dtype=F64)
    f = img.to(F64)
    jj, ii = torch.arange(W, device="cuda", dtype=F64)[None, :], torch.arange(H, device="cuda", dtype=F64)[:, None]
    sx, sy = Mi[0] * jj + Mi[1] * ii + Mi[2], Mi[3] * jj + Mi[4] * ii + Mi[5]
    inside = (sx >= 0) & (sx <= W - 1) & (sy >= 0) & (sy <= H - 1)
    j0, i0 = sx.floor().clamp(0, W - 2).long(), sy.floor().clamp(0, H - 2).long()
    wx, wy = sx - j0, sy - i0
    flat, at = f.reshape(-1), i0 * W + j0
    out = ((1 - wy) * ((1 - wx) * flat[at] + wx * flat[at + 1])
           + wy * ((1 - wx) * flat[at + W] + wx * flat[at + W + 1]))
    return dict(image=torch.where(inside, out, torch.zeros_like(out)), M=M)


def _difference64(case, img, tmpl):
    """Difference image of the least-squares kernel on the candidate stamps."""
    H, W, n, hw = img.shape[0], img.shape[1], case["regions"], 10
    I, R = img.to(F64), tmpl.to(F64)
    u = torch.arange(-hw, hw + 1, device="cuda", dtype=F64)
    K = []
    for s, d in ((0.7, 6), (1.5, 4), (3.0, 2)):
        e = torch.exp(-u * u / (2.0 * s * s))
        for i in range(d + 1):
            for j in range(d - i + 1):
                K.append((e * u ** j)[:, None] * (e * u ** i)[None, :])   # [v, u]
    K = torch.stack(K).flatten(1)   # [49, 441]

    def poly(x, y, order):
        xs, ys = 2.0 * x / (W - 1) - 1.0, 2.0 * y / (H - 1) - 1.0
        return torch.stack([xs ** p * ys ** q for p in range(order + 1) for q in range(order + 1 - p)], -1)

    rows, rhs = [], []
    for sy in range(n):
        for sx in range(n):
            y0, y1, x0, x1 = sy * H // n, (sy + 1) * H // n, sx * W // n, (sx + 1) * W // n
            r = R[y0:y1, x0:x1]
            v = r.reshape(-1).sort().values
            m = v.numel()
            med = 0.5 * (v[(m - 1) // 2] + v[m // 2])
            a = (v - med).abs().sort().values
            mad = 0.5 * (a[(m - 1) // 2] + a[m // 2])
            e = r.clone()
            yy, xx = torch.arange(y0, y1, device="cuda")[:, None], torch.arange(x0, x1, device="cuda")[None, :]
            e[~((yy >= 20) & (yy < H - 20) & (xx >= 20) & (xx < W - 20)).expand_as(e)] = -float("inf")
            k = int(e.argmax())
            if not bool(e.reshape(-1)[k] > med + 5.0 * 1.4826 * mad):
                continue
            cy, cx = y0 + k // (x1 - x0), x0 + k % (x1 - x0)
            win = R[cy - 20:cy + 21, cx - 20:cx + 21].unfold(0, 21, 1).unfold(1, 21, 1).flip(2, 3).reshape(441, 441)
            C = win @ K.T   # sum_{u,v} K(u, v) R(x - u, y - v)
            P = poly(torch.tensor(float(cx), dtype=F64), torch.tensor(float(cy), dtype=F64), 2).cuda()
            py, px = torch.meshgrid(torch.arange(cy - 10, cy + 11), torch.arange(cx - 10, cx + 11), indexing="ij")
            B = poly(px.reshape(-1).to("cuda", F64), py.reshape(-1).to("cuda", F64), 1)
            rows.append(torch.cat([(C[:, :, None] * P).flatten(1), -B], 1))
            rhs.append(I[cy - 10:cy + 11, cx - 10:cx + 11].reshape(-1))
    A, b = torch.cat(rows), torch.cat(rhs)
    sol = torch.cholesky_solve((A.T @ b)[:, None], torch.linalg.cholesky(A.T @ A))[:, 0]
    out = torch.full((H, W), float("nan"), dtype=F64, device="cuda")
    ck, cb = sol[:294].reshape(49, 6), sol[294:]
    pad = torch.nn.functional.pad(R[None, None], (10, 31, 10, 31), mode="constant")[0, 0]
    xt = torch.arange(0, W, 21, device="cuda")
    for y0 in range(0, H, 21):
        P = poly((xt + 10).to(F64), torch.full_like(xt, y0 + 10).to(F64), 2)      # [tiles, 6]
        kern = (P @ ck.T) @ K                                                     # [tiles, 441]
        strip = pad[y0:y0 + 41, :xt.numel() * 21 + 20].unfold(1, 41, 21).permute(1, 0, 2)
        win = strip.unfold(1, 21, 1).unfold(2, 21, 1).flip(3, 4).reshape(xt.numel(), 441, 441)
        conv = (win @ kern[:, :, None]).reshape(-1, 21, 21).permute(1, 0, 2).reshape(21, -1)[:H - y0, :W]
        h = conv.shape[0]
        py, px = torch.meshgrid(torch.arange(y0, y0 + h, device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
        out[y0:y0 + h] = I[y0:y0 + h] + poly(px.to(F64), py.to(F64), 1) @ cb - conv
    out[:10], out[H - 10:], out[:, :10], out[:, W - 10:] = (float("nan"),) * 4
    return out


def _auto64(s):
    """Kron photometry of each detection, one after another."""
    f, lab = s["sub"].double().cpu().numpy(), s["labels"].cpu().numpy()
    st = {k: v.cpu().numpy() for k, v in s["stats"].items()}
    H, W = f.shape
    rows, n = st["xbar"].size, int(s["n"])
    out = dict(flux=np.zeros(rows), area=np.zeros(rows), kron=np.zeros(rows), shape=np.zeros((rows, 3)))
    for k in range(n):
        y0, y1, x0, x1 = st["ymin"][k], st["ymax"][k] + 1, st["xmin"][k], st["xmax"][k] + 1
        xb, yb = float(st["xbar"][k]), float(st["ybar"][k])
        v = f[y0:y1, x0:x1] * (lab[y0:y1, x0:x1] == k + 1)
        t = v.sum()
        dx, dy = np.arange(x0, x1)[None, :] - xb, np.arange(y0, y1)[:, None] - yb
        x2, y2, xy = 1 / 12, 1 / 12, 0.0
        if t > 0:
            x2, y2, xy = (v * dx * dx).sum() / t, (v * dy * dy).sum() / t, (v * dx * dy).sum() / t
            if x2 * y2 - xy * xy < 1 / 144:
                x2, y2 = x2 + 1 / 12, y2 + 1 / 12
        det = x2 * y2 - xy * xy

        def box(r):
            a, b = r * math.sqrt(max(x2, 0.0)) + 1, r * math.sqrt(max(y2, 0.0)) + 1
            i0, i1 = max(int(math.floor(yb - b)), 0), min(int(math.ceil(yb + b)) + 1, H)
            j0, j1 = max(int(math.floor(xb - a)), 0), min(int(math.ceil(xb + a)) + 1, W)
            dx, dy = np.arange(j0, j1)[None, :] - xb, np.arange(i0, i1)[:, None] - yb
            return f[i0:i1, j0:j1], (y2 * dx * dx - 2 * xy * dx * dy + x2 * dy * dy) / det

        g, r2 = box(6.0)
        in6 = r2 <= 36.0
        g = g[in6]
        num, den = (np.sqrt(np.maximum(r2[in6], 0.0)) * g).sum(), g.sum()
        r1 = num / den if num > 0 and den > 0 else 0.0
        ra = max(2.5 * r1, 3.5)
        g, r2 = box(ra)
        inside = r2 <= ra * ra
        out["flux"][k], out["area"][k], out["kron"][k], out["shape"][k] = g[inside].sum(), inside.sum(), r1, (x2, y2, xy)
    return out


def _display64(case, seed):
    img = _mosaic(case, seed)
    H, W = img.shape
    flat = img.reshape(-1)
    # zscale: iterated line through the sorted samples
    s = flat[::max(1, W * H // 1000)][:1000].double().cpu().numpy()
    s = np.sort(s[np.isfinite(s)])
    n = s.size
    c = (n - 1) // 2
    xk, good, minpix, last, slope = np.arange(n) - c, np.ones(n, bool), max(5, n // 2), n + 1, 0.0
    grow = max(1, n // 100) // 2
    for _ in range(5):
        ng = int(good.sum())
        if ng >= last or ng < minpix:
            break
        last = ng
        slope, icept = np.polyfit(xk[good], s[good], 1)
        res = s - (icept + slope * xk)
        rej = np.abs(res) > 2.5 * res[good].std()
        good = ~np.convolve(rej, np.ones(2 * grow + 1), "same").astype(bool)
    med = 0.5 * (s[(n - 1) // 2] + s[n // 2])
    z = np.array([s[0], s[-1]])
    if good.sum() >= minpix:
        z = np.array([max(s[0], med - (c - 1) * slope / 0.25), min(s[-1], med + (n - c) * slope / 0.25)])
    # stretch
    fin = torch.isfinite(img)
    a = _GRAY[case["gray"]][1]
    xn = ((torch.nan_to_num(img).double() - _LO) / (_HI - _LO)).clamp(0.0, 1.0)
    g = {"linear": lambda t: t, "log": lambda t: torch.log10(a * t + 1.0) / math.log10(a + 1.0),
         "power": lambda t: t ** a, "exp": lambda t: (a ** t - 1.0) / (a - 1.0)}[case["gray"]](xn) * fin
    # equalisation: the bins are decided in 32 bits, as documented
    nb = case["nbins"]
    v = flat[fin.reshape(-1)]
    lo, hi = v.min(), v.max()
    sc = torch.tensor(float(nb), device="cuda") / (hi - lo)
    b = ((v - lo) * sc).floor().clamp(0, nb - 1).long()
    C = torch.bincount(b, minlength=nb).double().cumsum(0) / v.numel()
    t = ((torch.nan_to_num(img).double() - lo.double()) * sc.double() - 0.5).clamp(0.0, nb - 1.0)
    k = t.floor().clamp(0, nb - 2).long()
    eq = (C[k] + (t - k) * (C[k + 1] - C[k])) * fin
    return dict(z=z, gray=g, equalized=eq)
