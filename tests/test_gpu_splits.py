"""Cuts of the work that follow from sizes: results that may not depend on the cut, at the
sizes where it changes, and the quotients of the row solves bit for bit."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


# candidates cut into 4 and 2 blocks (152 SMs; 4, 30, 100, 140 and 400 slots give 6, 5, 3, 1
# and 3): the parts of a fit are the same sums whatever the cut
@pytest.mark.parametrize("slots", [38, 76])
def test_fit_parts_even(gpu, slots):
    R, _ = synth.tiny_frame(517, 389, 7, n_stars=90, sky=300.0, flux=(3.5, 4.5))
    I, R = dev((0.9 * R + 7.0).astype(np.float32)), dev(R)
    cx, cy, n = gpu.sub_stamps(I, R, nsx=2, nsy=2)
    k = int(host(n)[0])
    A0, b0 = gpu.sub_normal(I, R, cx[:k].clone(), cy[:k].clone(), n)
    px, py = (torch.zeros(slots, dtype=torch.int32, device="cuda") for _ in range(2))
    px[:k], py[:k] = cx[:k], cy[:k]
    A, b = gpu.sub_normal(I, R, px, py, n)
    assert k > 1 and torch.equal(A, A0) and torch.equal(b, b0)


# the row solves' quotients against IEEE division: the leading 32 x 32 block is diagonal
# with the squares of b, so the first panel leaves a / b in every row below it.  Divisors
# and dividends on both sides of the range that is divided by reciprocals (2^-250 to 2^250
# and 2^-600 to 2^600), all-ones mantissas, zeros, subnormals, both signs.
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_row_solve_quotients(gpu, seed):
    rng = np.random.default_rng(seed)
    rows = 1500
    ones = np.nextafter(2.0, 1.0)
    b = rng.uniform(1.0, 2.0, 32)
    b[:6] = [1.0, ones, np.nextafter(1.0, 2.0), 1.5, ones, np.nextafter(1.0, 2.0)]
    eb = np.r_[np.zeros(16, int), rng.integers(-240, 240, 4), -250, -251, 249, 250, -250, -251, 249, 250, -300, 300, -255, 255]
    b = np.ldexp(rng.permutation(b), eb)
    a = rng.uniform(1.0, 2.0, (rows, 32)) * rng.choice([-1.0, 1.0], (rows, 32))
    a[:200] = rng.choice([1.0, ones, -ones, np.nextafter(1.0, 2.0), 0.0, 1.25], (200, 32))
    ea = np.zeros((rows, 32), int)
    ea[400:900] = rng.choice([-600, -601, 599, 600, -599, 598], (500, 32))
    ea[900:1300] = rng.integers(-590, 590, (400, 32))
    ea[1300:1400] = rng.integers(-1074, -1000, (100, 32))
    a = np.ldexp(a, ea)
    n = 32 + rows
    A = np.zeros((n, n))
    A[np.arange(32), np.arange(32)] = b * b
    A[32:, :32] = a
    assert np.array_equal(np.sqrt(b * b), b)
    t = dev(A)
    gpu.sub_solve(t, dev(np.zeros(n)))   # fails at the next panel, whose rows are of rank 32
    with np.errstate(under="ignore"):
        assert np.array_equal(host(t)[32:, :32], a / b)


# segments of the reprojection in groups of 1, 2, 4 and 8 a warp: an integer shift is exact
@pytest.mark.parametrize("W,H", [(128, 4800), (128, 4870), (127, 9733), (257, 6490), (1000, 2437)])
def test_reproject_groups(gpu, W, H):
    img = np.random.default_rng(H).normal(size=(H, W)).astype(np.float32)
    out = host(gpu.reproject_affine(dev(img), dev(np.array([1.0, 0.0, -1.0, 0.0, 1.0, 2.0])), W, H, fill=-5.0))
    assert np.array_equal(out[:-2, 1:], img[2:, :-1]) and np.all(out[:, 0] == -5.0) and np.all(out[-2:] == -5.0)
