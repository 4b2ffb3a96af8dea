"""Chains of dependent launches, back to back, in ways that change what a kernel's
predecessor writes from one pass to the next: a pass that read a value of the pass before
would differ from the same pass run alone."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _frames(W, H):
    return [dev(synth.tiny_frame(W, H, s, n_stars=W * H // 2000, sky=500.0 + 40 * s, flux=(3.0, 4.5))[0]) for s in (4, 5)]


# the filtered catalog path (thresholded again on the subtracted frame that the kernel
# before has just written), two frames in turn through one workspace
@pytest.mark.parametrize("W,H,mesh", [(200, 150, 32), (517, 389, 12), (2100, 1500, 64)])
def test_filtered_extract_repeats(gpu, W, H, mesh):
    fr = _frames(W, H)
    cfg = gpu.BgConfig(mesh=mesh)
    ref = [gpu.Extractor(W, H, cfg, filter=1)(f) for f in fr]
    torch.cuda.synchronize()
    n = [int(host(r["n_src"])[0]) for r in ref]
    assert min(n) > 5
    ex = gpu.Extractor(W, H, cfg, filter=1)
    keys = ("n_src", "labels", "sub", "x", "y", "flux", "sky")
    got = [{q: v.clone() for q, v in ex(fr[it & 1]).items() if q in keys} for it in range(20)]
    for it, out in enumerate(got):
        for q in keys:
            m = n[it & 1] if q in ("x", "y", "flux", "sky") else None
            assert torch.equal(out[q][:m], ref[it & 1][q][:m]), q


# alignment (the reprojection reads the transform that the kernel before has just solved)
# and the catalog of its output, two exposures in turn, nothing waited for in between
@pytest.mark.parametrize("W,H", [(300, 260), (1500, 1100)])
def test_align_then_extract_repeats(gpu, W, H):
    fr = _frames(W, H)
    wcs = [synth.wcs_pair(W, H, seed=s) for s in (7001, 7002)]
    cfg = gpu.BgConfig(mesh=32)

    def one(i, ex, out):
        img, M, _ = gpu.align(fr[i], *wcs[i], W, H, out=out)
        return M, img.clone(), {q: ex(img)[q].clone() for q in ("sub", "labels", "n_src")}

    ref = []
    for i in (0, 1):
        ref.append(one(i, gpu.Extractor(W, H, cfg), torch.empty(H, W, device="cuda")))
        torch.cuda.synchronize()
    assert not torch.equal(ref[0][0], ref[1][0])
    ex, buf = gpu.Extractor(W, H, cfg), torch.empty(H, W, device="cuda")
    got = [one(it & 1, ex, buf) for it in range(20)]
    for it, (M, img, cat) in enumerate(got):
        r = ref[it & 1]
        assert torch.equal(M, r[0]) and torch.equal(img, r[1])
        assert all(torch.equal(cat[q], r[2][q]) for q in cat)


# under capture, after a copy and after a fork from another stream: the first kernel's
# predecessor in the graph is not a kernel
def test_captured_after_copy_and_fork(gpu):
    W, H = 517, 389
    fr = _frames(W, H)
    cfg = gpu.BgConfig(mesh=32)
    ref = [gpu.Extractor(W, H, cfg)(f) for f in fr]
    ex = [gpu.Extractor(W, H, cfg) for _ in range(2)]
    d = torch.empty(H, W, device="cuda")
    ex[0](fr[0]), ex[1](fr[0])
    torch.cuda.synchronize()
    s, t, g = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    h = host(fr[0])
    pin = torch.from_numpy(h.copy()).pin_memory()
    with torch.cuda.graph(g, stream=s):
        d.copy_(pin, non_blocking=True)
        ex[0](d)
        t.wait_stream(s)
        with torch.cuda.stream(t):
            ex[1](d)
        s.wait_stream(t)
    for it in range(6):
        pin.copy_(fr[it & 1].cpu())
        g.replay()
        torch.cuda.synchronize()
        for e in ex:
            assert all(torch.equal(e.out[q], ref[it & 1][q]) for q in ("sub", "labels", "n_src"))
