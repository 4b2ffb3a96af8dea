"""The kernel variants that a size, type or alignment selects, at the sizes where the
choice changes: each against the oracle, or against another route to the same
result.  Tolerances are those of the kernels' own parity tests (float results to a
few ulp of the quantities summed, whole numbers and selections exact)."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


# blocks per region: 1 (small regions), 2 or 4 (a slice of the next size), 8, and a
# region above eight slices, which is read from memory in every pass
@pytest.mark.parametrize("W,H,nsx,nsy", [(300, 261, 4, 4), (301, 260, 1, 1), (517, 389, 2, 2), (1031, 877, 2, 1),
                                         (1031, 877, 10, 10), (700, 40, 9, 1)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -20, 2.0 ** 40])
def test_stamp_clusters(gpu, orc, W, H, nsx, nsy, scale):
    R, _ = synth.tiny_frame(W, H, 5, n_stars=W * H // 900, sky=300.0, flux=(3.0, 4.5))
    R = (R * np.float32(scale)).astype(np.float32)
    rng = np.random.default_rng(W + nsx)
    R[rng.integers(0, H, 20), rng.integers(0, W, 20)] = np.nan
    I = (R * np.float32(0.75)).astype(np.float32)
    kw = dict(nsx=nsx, nsy=nsy, hw=4, fh=5, nsig=5.0)
    cx, cy, n = gpu.sub_stamps(dev(I), dev(R), **kw)
    ocx, ocy = orc.sub_stamps(I, R, **kw)
    k = int(host(n)[0])
    assert k == len(ocx) and np.array_equal(host(cx)[:k], ocx) and np.array_equal(host(cy)[:k], ocy)


# candidates cut into 6, 4, 3 and 1 blocks: the parts of a fit are the same sums
# whatever the cut, so the normal equations of the first candidates do not depend on
# how many slots follow them
@pytest.mark.parametrize("slots", [4, 30, 100, 140, 400])
def test_fit_parts(gpu, slots):
    R, _ = synth.tiny_frame(517, 389, 7, n_stars=90, sky=300.0, flux=(3.5, 4.5))
    I = dev((0.9 * R + 7.0).astype(np.float32))
    R = dev(R)
    cx, cy, n = gpu.sub_stamps(I, R, nsx=2, nsy=2)
    k = int(host(n)[0])
    A0, b0 = gpu.sub_normal(I, R, cx[:k].clone(), cy[:k].clone(), n)
    pad = torch.zeros(slots, dtype=torch.int32, device="cuda")
    px, py = pad.clone(), pad.clone()
    px[:k], py[:k] = cx[:k], cy[:k]
    A, b = gpu.sub_normal(I, R, px, py, n)
    assert k > 1 and torch.equal(A, A0) and torch.equal(b, b0)


@pytest.mark.parametrize("np_", [1, 2, 31, 32, 33, 64, 65, 97, 300])
def test_cholesky_sizes(gpu, np_):
    rng = np.random.default_rng(np_)
    B = rng.normal(size=(np_ + 20, np_))
    A, x = B.T @ B, rng.normal(size=np_)
    c64, c32, st = gpu.sub_solve(dev(A), dev(A @ x))
    # backward stable: |x - x0| <= c n eps cond |x|, cond of a (n + 20) x n Gaussian's Gram < 1e5
    assert int(host(st)[0]) == 0
    assert np.max(np.abs(host(c64) - x)) <= 1e-16 * np_ * np.linalg.cond(A) * 10 * np.max(np.abs(x)) + 1e-13
    A[np_ // 2, np_ // 2] = -1.0   # not positive definite: reported, nothing solved
    _, _, st = gpu.sub_solve(dev(A), dev(A @ x))
    assert int(host(st)[0]) == 1


# tiles of every half width on frames of one tile, one group of tiles and a ragged rest
@pytest.mark.parametrize("hw", [4, 6, 8, 10, 12])
@pytest.mark.parametrize("extra", [(1, 1), (2, 7), (70, 3)])
def test_apply_shapes(gpu, orc, hw, extra):
    W, H = 2 * hw + extra[0] + 2 * hw, 2 * hw + extra[1]
    rng = np.random.default_rng(hw + extra[0])
    R = rng.normal(300.0, 20.0, (H, W)).astype(np.float32)
    I = rng.normal(300.0, 20.0, (H, W)).astype(np.float32)
    sig, deg, sord, bord = (1.0, 2.5), (2, 1), 1, 2
    coef = rng.normal(0, 0.05, 9 * 3 + 6)
    g = host(gpu.sub_apply(dev(I), dev(R), coef, hw=hw, sig=sig, deg=deg, sord=sord, bord=bord))
    o = orc.sub_apply(I, R, coef, hw=hw, sig=sig, deg=deg, sord=sord, bord=bord, tile=2 * hw + 1)
    assert np.array_equal(np.isnan(g), np.isnan(o))
    B = np.abs(orc.sub_basis(hw, sig, deg)).reshape(9, -1).sum(1)
    bound = (np.abs(coef[:27]).reshape(9, 3).sum(1) * B).sum() * 400.0 + 400.0 + np.abs(coef[27:]).sum()
    assert np.nanmax(np.abs(g - o)) <= 1e-5 * bound


# eight lanes a stamp up to 5 x 5 pixels, a warp above
@pytest.mark.parametrize("S", [3, 5, 6, 7, 32])
@pytest.mark.parametrize("model", [0, 1])
def test_psf_model_sizes(gpu, orc, S, model):
    rng = np.random.default_rng(S)
    n, c = 37, (S - 1) / 2
    P = np.stack([c + rng.uniform(-0.6, 0.6, n), c + rng.uniform(-0.6, 0.6, n), rng.uniform(500, 5e4, n),
                  rng.uniform(50, 1000, n), rng.uniform(1.0, 2.0, n), rng.uniform(1.0, 2.0, n),
                  rng.uniform(-1.5, 1.5, n)], 1).astype(np.float32)
    G = rng.normal(size=(n, S, S)).astype(np.float32)
    p = dev(P).requires_grad_(True)
    m = gpu.psf_model(p, S, model, 2.5)
    m.backward(dev(G))
    m, ga = host(m.detach()), host(p.grad)
    for k in range(n):
        om, J = orc.psf_model(P[k].astype(np.float64), S, model, 2.5)
        assert np.max(np.abs(m[k] - om)) <= 2e-5 * np.max(np.abs(om))
        sc = np.abs(J).max(axis=0) * np.abs(G[k]).sum()
        assert np.all(np.abs(ga[k] - J.T @ G[k].ravel().astype(np.float64)) <= 1e-5 * sc + 1e-6)


# a fit does not depend on the stamps around it: not on its slot, its warp, or when its
# convergence test is taken
@pytest.mark.parametrize("S,n", [(11, 41000), (15, 30001), (15, 9000)])
def test_fit_order_independent(gpu, S, n):
    g = torch.Generator(device="cuda").manual_seed(S)
    c = (S - 1) / 2
    p = torch.rand(n, 7, generator=g, device="cuda")
    lo = torch.tensor([c - 0.5, c - 0.5, 100.0, 900.0, 1.1, 0.9, -1.5], device="cuda")
    hi = torch.tensor([c + 0.5, c + 0.5, 2e4, 1100.0, 2.0, 1.8, 1.5], device="cuda")
    st = gpu.psf_model(lo + p * (hi - lo), S)
    st = st + torch.randn(st.shape, generator=g, device="cuda") * st.clamp_min(1.0).sqrt()
    perm = torch.randperm(n, generator=g, device="cuda")
    a, b = gpu.psf_fit(st), gpu.psf_fit(st[perm].contiguous())
    for k in ("params", "chi2", "iters", "flags"):
        assert torch.equal(a[k][perm], b[k]), k


@pytest.mark.parametrize("ns", [1, 31, 32, 33, 1000, 1024, 1025, 2048, 4096])
def test_zscale_sample_sizes(gpu, orc, ns):
    img, _ = synth.tiny_frame(131, 97, 3, n_stars=30, sky=500.0, flux=(3.0, 4.5))
    img[5:9, 7:30] = np.nan
    z, cnt = gpu.zscale(dev(img), n_samples=ns)
    z1, z2, oc = orc.zscale(img, n_samples=ns)
    assert tuple(int(v) for v in host(cnt)) == oc
    assert np.allclose(host(z), [z1, z2], rtol=1e-9, atol=0.0)


# two warps a block up to 8 x 152 x 64 points, eight above
@pytest.mark.parametrize("n", [2, 77824, 77825])
def test_affine_fit_sizes(gpu, n):
    rng = np.random.default_rng(n)
    x, y = rng.uniform(0, 4096, n), rng.uniform(0, 4096, n)
    a, b, tx, ty = 0.9993, 0.0121, 13.5, -7.25
    M, st = gpu.affine_fit(dev(a * x - b * y + tx), dev(b * x + a * y + ty), x=dev(x), y=dev(y))
    assert int(host(st)[0]) == 0
    assert np.max(np.abs(host(M)[:6] - [a, -b, tx, b, a, ty])) <= 1e-9


# groups of eight segments of 128 columns: an integer shift is exact for any width
@pytest.mark.parametrize("W,H", [(1, 1), (127, 3), (128, 8), (129, 5), (1030, 3)])
def test_reproject_segments(gpu, W, H):
    img = np.random.default_rng(W).normal(size=(H, W)).astype(np.float32)
    out = host(gpu.reproject_affine(dev(img), dev(np.array([1.0, 0.0, 1.0, 0.0, 1.0, 0.0])), W, H, fill=-5.0))
    assert np.array_equal(out[:, :-1], img[:, 1:]) and np.all(out[:, -1] == -5.0)


# rows of raw frames read in fours where the frame and its maps allow, else one by one
@pytest.mark.parametrize("W,H,mesh", [(256, 128, 64), (260, 131, 64), (257, 96, 32), (300, 100, 48)])
@pytest.mark.parametrize("maps", [False, True])
@pytest.mark.parametrize("shift", [0, 1])
def test_raw_mesh_reads(gpu, W, H, mesh, maps, shift):
    g = torch.Generator(device="cuda").manual_seed(W + H)
    buf = torch.randint(900, 1100, (W * H + 8,), generator=g, device="cuda", dtype=torch.int32).to(torch.uint16)
    raw = buf[shift:shift + W * H].view(H, W)   # a shift of one value leaves rows unaligned
    inv = 0.9 + 0.2 * torch.rand(H, W, generator=g, device="cuda")
    bias = torch.full((H, W), 500.0, device="cuda")
    if maps:
        bias = bias + torch.randn(H, W, generator=g, device="cuda")
    cal = (inv, 500.0, bias) if maps else (inv, 500.0)
    got = gpu.bg_estimate(raw, mesh=mesh, calib=cal)
    ref = gpu.bg_estimate((raw.int().float() - bias) * inv, mesh=mesh)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])


# windows of up to 11 columns and of up to 15
@pytest.mark.parametrize("fwhm", [1.0, 3.0, 3.05, 3.3, 4.0, 4.4])
def test_centroid_windows(gpu, orc, fwhm):
    img, _ = synth.tiny_frame(160, 120, 9, n_stars=40, sky=0.0, flux=(3.5, 4.5))
    rng = np.random.default_rng(2)
    y0, x0 = (np.asarray(v, np.float32) for v in np.unravel_index(np.argsort(img.ravel())[-60:], img.shape))
    x0, y0 = x0 + rng.uniform(-0.5, 0.5, 60).astype(np.float32), y0 + rng.uniform(-0.5, 0.5, 60).astype(np.float32)
    ox, oy, _, ofl = orc.centroid(img, x0, y0, fwhm_win=fwhm)
    gx, gy, _, gfl = (host(t) for t in gpu.centroid(dev(img), dev(x0), dev(y0), fwhm_win=fwhm))
    ok = ((ofl & 2) == 0) & ((gfl & 2) == 0)
    assert np.array_equal(gfl & 1, ofl & 1) and ok.sum() >= 20
    assert np.all(np.abs(gx - ox)[ok] <= 1e-3) and np.all(np.abs(gy - oy)[ok] <= 1e-3)


# corner tables (r_ap < 7), per-pixel overlaps above, annuli from one pixel to the widest,
# centres inside the frame, at its edges and beyond
@pytest.mark.parametrize("r_ap,r_in,r_out", [(0.7, 1.0, 3.0), (5.0, 8.0, 12.0), (6.9, 0.0, 7.5), (7.5, 9.0, 16.0),
                                             (16.0, 15.0, 16.0), (3.0, 12.0, 12.4)])
def test_aperture_radii(gpu, orc, r_ap, r_in, r_out):
    rng = np.random.default_rng(int(10 * r_ap))
    sub = rng.normal(5.0, 30, (90, 110)).astype(np.float32)
    x, y = rng.uniform(-3, 113, 700).astype(np.float32), rng.uniform(-3, 93, 700).astype(np.float32)
    x[:60], y[:60] = np.round(2 * x[:60]) / 2, np.round(2 * y[:60]) / 2
    kw = dict(r_ap=r_ap, r_in=r_in, r_out=r_out)
    ph = orc.aperture(sub, x, y, **kw)
    g = {k: host(v) for k, v in gpu.aperture_phot(dev(sub), dev(x), dev(y), **kw).items()}
    assert np.array_equal(g["n_ann"], ph["n_ann"]) and np.array_equal(g["flags"], ph["flags"])
    assert np.array_equal(g["sky"], ph["sky"].astype(np.float32))
    scale = np.abs(ph["flux"]) + ph["area"] * (np.abs(ph["sky"]) + 30.0)
    assert np.all(np.abs(g["flux"] - ph["flux"]) <= 1e-5 * scale + 1e-5)


# the chain of dependent launches on small and larger grids, back to back on one stream and
# on two: every pass gives the first one's catalog
@pytest.mark.parametrize("W,H,mesh", [(200, 150, 32), (1000, 900, 64), (2100, 1500, 64)])
def test_extract_repeats(gpu, W, H, mesh):
    img, _ = synth.tiny_frame(W, H, 4, n_stars=W * H // 2000, sky=500.0, flux=(3.0, 4.5))
    d = dev(img)
    cfg = gpu.BgConfig(mesh=mesh)
    ref = gpu.extract(d, cfg)
    torch.cuda.synchronize()
    n = int(host(ref["n_src"])[0])
    exs = [gpu.Extractor(W, H, cfg) for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    for s in streams:
        s.wait_stream(torch.cuda.current_stream())
    for _ in range(20):
        for ex, s in zip(exs, streams):
            with torch.cuda.stream(s):
                ex(d)
    torch.cuda.synchronize()
    for ex in exs:
        assert int(host(ex.out["n_src"])[0]) == n
        assert torch.equal(ex.out["labels"], ref["labels"]) and torch.equal(ex.out["sub"], ref["sub"])
        for k in ("x", "y", "flux", "sky"):
            assert torch.equal(ex.out[k][:n], ref[k][:n])


# Kron apertures whose box gives a thread 16 pixels a row and more (rows told apart by two
# bounds) and narrower ones, for footprints above and below the block form's 128
# pixels, inside and beyond the frame.
# The moments are FP32 sums (1e-4 relative), so the ellipse's area may differ by 1e-3 of
# itself; one that holds the frame holds every pixel.
@pytest.mark.parametrize("k_kron", [12.0, 25.0, 60.0, 1e4])
def test_wide_kron_apertures(gpu, orc, k_kron):
    H, W = 120, 4203
    rng = np.random.default_rng(3)
    yy, xx = np.mgrid[:H, :W]
    sub = rng.normal(0.0, 1.0, (H, W))
    lab = np.zeros((H, W), np.int32)
    stats = {k: [] for k in ("xmin", "xmax", "ymin", "ymax", "xbar", "ybar")}
    for n, (cx, cy, a, b, th) in enumerate([(2000, 50, 2.0, 1.6, 0.0), (900, 60, 5.0, 1.5, 0.1), (3300, 70, 9.0, 2.0, -0.05),
                                            (8, 100, 3.0, 2.5, 0.3)]):
        u = (xx - cx) * np.cos(th) + (yy - cy) * np.sin(th)
        v = (yy - cy) * np.cos(th) - (xx - cx) * np.sin(th)
        q = (u / a) ** 2 + (v / b) ** 2
        sub += 200.0 * np.exp(-0.5 * q)
        foot = (q < 5.0) & (lab == 0)
        lab[foot] = n + 1
        for k, m in (("xmin", xx[foot].min()), ("xmax", xx[foot].max()), ("ymin", yy[foot].min()), ("ymax", yy[foot].max()),
                     ("xbar", cx + 0.25), ("ybar", cy - 0.125)):
            stats[k].append(m)
    sub = sub.astype(np.float32)
    st = {k: np.asarray(v, np.float32 if k[1:] == "bar" else np.int32) for k, v in stats.items()}
    o = orc.auto_phot(sub, lab, st, k_kron=k_kron)
    full = gpu._alloc_stats(4, torch.device("cuda"))
    for k, v in st.items():
        full[k].copy_(dev(v))
    g = gpu.auto_phot(dev(sub), dev(lab), torch.tensor([4], dtype=torch.int32, device="cuda"), full, k_kron=k_kron)
    g = {k: host(v) for k, v in g.items()}
    assert np.array_equal(g["flags"], o["flags"])
    edge = np.where(o["area"] == W * H, 0.0, 1e-3 * o["area"] + 4.0)
    assert np.all(np.abs(g["area"] - o["area"]) <= edge)
    assert np.all(np.abs(g["flux"] - o["flux"]) <= 1e-5 * np.abs(sub).sum() + 6.0 * edge)
