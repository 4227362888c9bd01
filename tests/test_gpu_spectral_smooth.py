"""The spectral analysis for channel counts without an FFT, on smooth spectra,
whose coefficients are small differences of large sums: it must not be further
from 64-bit arithmetic than float32 multiply-adds channel by channel are, whatever
it adds up first."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


# at least 2^18 values: the register-tiled product
@pytest.mark.parametrize("n,L", [(512, 3), (256, 5), (256, 6), (256, 12), (256, 15), (128, 17), (128, 21), (128, 37), (64, 96), (64, 200), (64, 201)])
@pytest.mark.parametrize("noise", [0.0, 0.05])
def test_coefficients_of_smooth_spectra(lib, n, L, noise):
    g = torch.Generator(device="cuda").manual_seed(100 * n + L)
    nu = torch.linspace(1.0, 1.5, L, device="cuda")[:, None, None]
    amp = 0.5 + 1.5 * torch.rand(n, n, device="cuda", generator=g)
    slope = 0.5 + 0.5 * torch.rand(n, n, device="cuda", generator=g)
    y = amp * nu ** -slope + noise * torch.randn(L, n, n, device="cuda", generator=g)
    psf = torch.zeros(L, n, n, device="cuda")
    psf[:, n // 2, n // 2] = 1.0                       # H = I: from X = V = 0 the step is X = tau y, D = 2 X
    k = 2.0 ** -8                                      # no coefficient reaches its bound
    m = lib.Muffin(y, psf, nscales=1, mu_s=0.0, mu_l=k, tau=0.25, power_iters=1)
    zero = torch.zeros_like(y)
    m.set_state(zero, torch.zeros(L, 2, n, n, device="cuda"), zero, 0)
    m.iterate(1)
    x, _, v, _ = m.get_state()
    torch.cuda.synchronize()
    m.close()
    D = 2 * x.reshape(L, -1)
    kk = torch.arange(L, dtype=torch.float64, device="cuda")
    C = torch.cos(math.pi * (2 * kk[None] + 1) * kk[:, None] / (2 * L)) * math.sqrt(2.0 / L)
    C[0] = math.sqrt(1.0 / L)
    Cf, c = C.float().double(), torch.zeros(L, n * n, device="cuda")
    for l in range(L):                                 # float32 multiply-adds, channel by channel
        c = torch.addcmul(c.double(), Cf[:, l:l + 1], D[l:l + 1].double()).float()
    exact = C @ D.double()
    got = v.reshape(L, -1).double() / k
    err = lambda t: float((t.double() - exact)[1:].square().mean().sqrt())  # noqa: E731
    # one in a hundred for the chance in either error, of at least 6000 pixels
    assert err(got) <= 1.01 * err(c)
