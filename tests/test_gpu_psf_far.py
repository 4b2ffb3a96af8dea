"""PSF fits that start with the star so far off its stamp that the profile there is below
2^-126: the model's values count all the same when the flux is large."""
import math

import pytest
import torch

from gpu_util import host

pytestmark = pytest.mark.gpu


# (model, centre beyond the stamp, width, flux): profiles of 2^-133 and 2^-127 at the
# nearest pixels.  The stamp is the model at the start, so its chi^2 is that of the rounding
# (1e-4 of each value at most, the profile keeping 12 bits or more), and a fit only lowers it
@pytest.mark.parametrize("model,far,width,flux", [("gauss", 13.6, 1.0, 1e38), ("moffat", 2.53e6, 0.06, 1e38)])
@pytest.mark.parametrize("n", [3, 40000])
def test_far_start(gpu, model, far, width, flux, n):
    S, gauss = 5, model == "gauss"
    x0 = torch.tensor(S - 1 + far, dtype=torch.float32).item()
    jj = torch.arange(S, dtype=torch.float64)
    q = ((jj.view(1, S) - x0) ** 2 + (jj.view(S, 1) - 2.0) ** 2) / float(torch.tensor(width)) ** 2
    if gauss:
        st = flux / (2 * math.pi * width * width) * torch.exp(-0.5 * q)
    else:
        st = flux * 1.5 / (math.pi * width * width) * (1 + q) ** -2.5
    st = st.float().cuda().expand(n, S, S).contiguous()
    init = torch.tensor([x0, 2.0, flux, 0.0, width, width, 0.0], device="cuda").expand(n, 7).contiguous()
    o = gpu.psf_fit(st, init=init, model=gpu.PSF_GAUSS if gauss else gpu.PSF_MOFFAT, max_iter=1)
    assert (host(o["chi2"]).astype(float) <= 1e-4 * float((st[0].double() ** 2).sum())).all()
