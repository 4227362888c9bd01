"""The row march of the fine wavelet levels (large cubes) and of the coarse
levels on 128 x 128 sub-images (512 of them at least) against the general
kernels, which the same cube runs on when MUFFIN_IUWT_GENERAL is set: every
width, split and level count the march takes, the coarse plane's dual in its
epilogue (J = j1), relaxation, strips that end inside a channel, and channel
counts on both sides of its thresholds (2^21 and 2^22 pixels)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# (n, L, J, j1): at least 2^22 pixels unless noted
CASES = [(128, 257, 3, 1), (128, 256, 3, 2), (128, 259, 3, 3), (128, 258, 4, 3), (256, 67, 1, 1), (256, 65, 4, 2),
         (256, 64, 3, 3), (512, 17, 2, 2), (512, 33, 5, 3), (1024, 4, 3, 3), (1024, 5, 4, 3),
         (1024, 8, 4, 3), (1024, 9, 5, 3),       # coarse march too
         (1024, 7, 5, 3),                       # too few sub-images for it
         (64, 9, 3, 0), (32, 5, 2, 0), (64, 64, 1, 0),      # the whole image as one resident sub-image
         (256, 33, 4, 2),                       # march adjoint, tile analysis
         (256, 31, 4, 2), (512, 7, 4, 3)]       # below both thresholds


def _passes(n, L, J, j1, rho, state, dirty, psf):
    from paper_1602_08847_gb300.muffin import Muffin

    m = Muffin(dirty, psf, nscales=J, tau=0.02, rho=rho, fine_levels=j1, power_iters=1)
    m.set_state(*state, 0)
    m.iterate(2)              # the second pass reads the adjoint that the first one left
    out = m.get_state()[:3]
    torch.cuda.synchronize()
    m.close()
    return out


@pytest.mark.parametrize("n,L,J,j1", CASES)
def test_march_equals_general_kernels(n, L, J, j1, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(7 * n + L)
    dirty = torch.randn(L, n, n, device="cuda", generator=g)
    psf = torch.zeros(L, n, n, device="cuda")
    psf[:, n // 2, n // 2] = 1.0
    psf[:, n // 2, n // 2 + 1] = 0.25
    state = [torch.rand(L, n, n, device="cuda", generator=g)]
    state += [(1.5 * torch.randn(*s, device="cuda", generator=g)).clamp(-1, 1) for s in ((L, J + 1, n, n), (L, n, n))]
    rho = 1.3 if L % 2 else 1.0
    monkeypatch.delenv("MUFFIN_IUWT_GENERAL", raising=False)
    a = _passes(n, L, J, j1, rho, state, dirty, psf)
    monkeypatch.setenv("MUFFIN_IUWT_GENERAL", "1")
    b = _passes(n, L, J, j1, rho, state, dirty, psf)
    # every filtered value is a sum of at most 25 terms per level with weights that add up to 1, so each of the at
    # most 5 levels rounds by less than 12 units of 2^-24 of the largest value (below 8); two passes
    tol = 2 * 5 * 12 * 2.0 ** -24 * 8
    for x, y in zip(a, b):
        assert torch.isfinite(x).all()
        assert float((x - y).abs().max()) <= tol
