"""Cleaning in other units: objects of one pixel (whose shape does not depend on the scale
of the frame), peaks, threshold and frame scaled by a power of two."""
import numpy as np
import pytest
import torch

from gpu_util import dev, host

pytestmark = pytest.mark.gpu


# a faint object among 3600 bright ones 20 px apart: their wings at it are ~1e-5 of a peak
# each and decide together; at 2^-112 every one of them is below 2^-126
@pytest.mark.parametrize("k", [0, -60, -112])
def test_clean_scaled(gpu, orc, k):
    n, step = 61, 20
    W = H = n * step
    sub, lab = np.zeros((H, W), np.float64), np.zeros((H, W), np.int32)
    yy, xx = (v.ravel() * step + step // 2 for v in np.mgrid[:n, :n])
    rng = np.random.default_rng(1)
    sub[yy, xx] = 1.0 + rng.random(n * n)
    lab[yy, xx] = np.arange(1, n * n + 1)
    m = n * n
    fx, fy = 30 * step, 30 * step        # ten pixels from the nearest
    sub[fy, fx], lab[fy, fx] = 0.06, m + 1
    # its wings sum: sum over the others of peak / (1 + q), q = r^2 det^-1/2 scale of a pixel
    inv_a2 = 1.0 / (2.0 * np.log(2.0))
    q = ((yy - fy) ** 2 + (xx - fx) ** 2) * 12.0 * inv_a2
    wings = (sub[yy, xx] / (1.0 + q)).sum()
    for frac, merged in ((1.05, True), (0.95, False)):
        thr = 0.06 - wings / frac        # kept when peak - wings >= threshold
        assert thr > 0.0
        s = 2.0 ** k
        a = dev((sub * s).astype(np.float32))
        out, cnt = gpu.clean(a, dev(lab), torch.tensor([m + 1], dtype=torch.int32, device="cuda"), m + 1,
                             thr_map=torch.full((H, W), thr * s, dtype=torch.float32, device="cuda"), beta=1.0)
        kept = int(host(out)[fy, fx]) not in set(host(out)[yy, xx].tolist())
        assert kept != merged, (frac, wings, int(host(cnt)[0]))
