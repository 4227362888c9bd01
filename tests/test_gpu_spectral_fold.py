"""The folded DCT product (channel counts without an FFT), each product against
64-bit arithmetic on the values the kernel itself read: channel counts at the
edges of its register tiles (8 even and 8 odd rows), of its subtile widths (100
and 200 channels) and of its range, odd and even, and images of one subtile up
to several blocks of several subtiles."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


# at least 2^18 values, but for the last three (the plain product)
@pytest.mark.parametrize("n,L", [(512, 1), (512, 2), (512, 3), (256, 5), (256, 7), (256, 8), (128, 17), (128, 31),
                                 (128, 33), (128, 48), (64, 99), (64, 100), (64, 101), (64, 130), (64, 199), (64, 200),
                                 (64, 201), (64, 255), (32, 257), (32, 511), (32, 512), (16, 3), (64, 8), (16, 300)])
def test_folded_spectral_step(lib, n, L):
    mu_l, sigma, tau = 0.7, 1.5, 0.25
    rho = 1.3 if L % 2 else 1.0
    g = torch.Generator(device="cuda").manual_seed(1000 * n + L)
    y = torch.randn(L, n, n, device="cuda", generator=g) + 1.0
    psf = torch.zeros(L, n, n, device="cuda")
    psf[:, n // 2, n // 2] = 1.0                      # H = I: the gradient is x - y
    m = lib.Muffin(y, psf, nscales=1, mu_s=0.0, mu_l=mu_l, tau=tau, sigma=sigma, rho=rho, power_iters=1)
    x0, v0 = torch.zeros_like(y), (0.8 * torch.randn(L, n, n, device="cuda", generator=g)).clamp(-1, 1)
    m.set_state(x0, torch.zeros(L, 2, n, n, device="cuda"), v0, 0)
    states = [(x0, v0)]
    for _ in range(2):
        m.iterate(1)
        x, _, v, _ = m.get_state()
        states.append((x, v))
    torch.cuda.synchronize()
    m.close()
    k = torch.arange(L, dtype=torch.float64, device="cuda")
    C = torch.cos(math.pi * (2 * k[None] + 1) * k[:, None] / (2 * L)) * math.sqrt(2.0 / L)
    C[0] = math.sqrt(1.0 / L)
    flat = lambda M, t: (M @ t.double().reshape(L, -1)).reshape(t.shape)  # noqa: E731
    kk, terms = sigma * mu_l, (L + 1) // 2 + 6        # roundings of one folded sum: table, fold, products, epilogue
    for (xa, va), (xb, vb) in zip(states, states[1:]):
        # adjoint: x_b = x_a + rho (max(x_a - tau (x_a - y + mu_l T), 0) - x_a), T = C^T v_a
        T = flat(C.T, va)
        xt = (xa.double() - tau * (xa.double() - y.double() + mu_l * T)).clamp_min(0)
        ref = rho * xt + (1 - rho) * xa.double()
        fft = 64 * EPS * (xa.abs().max() + y.abs().max())       # forward and inverse FFT of x and of y, at most 6 passes each way
        bound = rho * tau * (mu_l * terms * EPS * flat(C.abs().T, va.abs()) + fft) + 8 * EPS * (1 + xa.abs().max() + xt.abs().max())
        assert bool(((xb.double() - ref).abs() <= bound).all())
        # analysis and dual step, from the x_b that the pass wrote: D = 2 x~ - x_a with x_b = rho x~ + (1 - rho) x_a
        xtb = (xb.double() - (1 - rho) * xa.double()) / rho
        D = 2 * xtb - xa.double()
        sat = (va.double() + kk * flat(C, D)).clamp(-1, 1)
        ref = rho * sat + (1 - rho) * va.double()
        dD = 8 * EPS * (xb.abs().max() + xa.abs().max())        # D is rounded, and here recovered from a rounded x_b
        bound = rho * kk * (terms * EPS * flat(C.abs(), D.abs()) + dD * C.abs().sum(1)[:, None, None]) + 8 * EPS
        assert bool(((vb.double() - ref).abs() <= bound).all())
