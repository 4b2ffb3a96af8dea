"""Error of the PSF model's adjoint against the formula's own rounding in 32 bits."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _terms(p, G, S, gauss, beta=2.5):
    """g dm/dp of every pixel and parameter, in the type of p: [7][n, S, S]."""
    x0, y0, F, _, sx, sy, th = [v.view(-1, 1, 1) for v in p.unbind(1)]
    jj = torch.arange(S, device=p.device, dtype=p.dtype).view(1, 1, S)
    dx, dy, c, s = jj - x0, jj.view(1, S, 1) - y0, torch.cos(th), torch.sin(th)
    u, v, ix, iy = c * dx + s * dy, c * dy - s * dx, 1 / (sx * sx), 1 / (sy * sy)
    q = u * u * ix + v * v * iy
    if gauss:
        A = torch.exp(-0.5 * q) / (2 * math.pi * sx * sy)
        d = -0.5 * F * A
    else:
        A = (beta - 1) / (math.pi * sx * sy) * torch.exp2(-beta * torch.log2(1 + q))
        d = -beta * F * A / (1 + q)
    P = F * A
    J = [d * (2 * v * iy * s - 2 * u * ix * c), -d * (2 * u * ix * s + 2 * v * iy * c), A, torch.ones_like(A),
         -P / sx - d * 2 * u * u * ix / sx, -P / sy - d * 2 * v * v * iy / sy,
         d * 2 * u * v * (sy - sx) * (sy + sx) * ix * iy]
    return [G * j for j in J]


# the derivatives evaluated plainly in 32 bits, pixel by pixel, and summed without error
# set the mean error of the formula itself.  The kernel's sums add the rounding of a tree
# of additions, each of 2.5e-8 rms of its result: the partial sums of a level have together
# the spread of the whole sum, so seven levels of terms that a few pixels carry give 2.6
# times that, a mean of at most 2^-24 of the sum
@pytest.mark.parametrize("S", [5, 6, 15, 24])
@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("positive", [False, True])
def test_adjoint_error(gpu, S, model, positive):
    g = torch.Generator(device="cuda").manual_seed(10 * S + model)
    n, c = 20000, (S - 1) / 2
    lo = torch.tensor([c - 0.5, c - 0.5, 100.0, 50.0, 0.9, 0.9, -1.5], device="cuda")
    hi = torch.tensor([c + 0.5, c + 0.5, 5e4, 1000.0, 2.5, 2.5, 1.5], device="cuda")
    p = lo + torch.rand(n, 7, generator=g, device="cuda") * (hi - lo)
    G = torch.randn(n, S, S, generator=g, device="cuda")
    G = G.abs() if positive else G
    t = p.clone().requires_grad_(True)
    gpu.psf_model(t, S, model).backward(G)
    t64, t32 = _terms(p.double(), G.double(), S, model == gpu.PSF_GAUSS), _terms(p, G, S, model == gpu.PSF_GAUSS)
    for k in (0, 1, 2, 4, 5, 6):   # the sky's is a sum of g alone
        ref, mag = t64[k].sum((1, 2)), t64[k].abs().sum((1, 2))
        plain = ((t32[k].double().sum((1, 2)) - ref).abs() / mag).mean().item()
        err = ((t.grad[:, k].double() - ref).abs() / mag).mean().item()
        assert err <= plain + 2.0 ** -24 * (ref.abs() / mag).mean().item(), (k, err, plain)
