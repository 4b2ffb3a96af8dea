"""Cuts of the work that follow from sizes: results that may not depend on the cut, at the
sizes where it changes."""
import numpy as np
import pytest

from gpu_util import dev, host

pytestmark = pytest.mark.gpu


# segments of the reprojection in groups of 1, 2, 4 and 8 a warp: an integer shift is exact
@pytest.mark.parametrize("W,H", [(128, 4800), (128, 4870), (127, 9733), (257, 6490), (1000, 2437)])
def test_reproject_groups(gpu, W, H):
    img = np.random.default_rng(H).normal(size=(H, W)).astype(np.float32)
    out = host(gpu.reproject_affine(dev(img), dev(np.array([1.0, 0.0, -1.0, 0.0, 1.0, 2.0])), W, H, fill=-5.0))
    assert np.array_equal(out[:-2, 1:], img[2:, :-1]) and np.all(out[:, 0] == -5.0) and np.all(out[-2:] == -5.0)
