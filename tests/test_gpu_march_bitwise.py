"""The row march of the fine wavelet levels and the march of the coarse ones give
bitwise the results of the halo-tile and block kernels: a cube that is taken in
groups of channels too small for the march (muffin_set_plan) runs on those, the
same cube in one group on the march.  The library's own rules say which kernels
a group of that size takes."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


class Geom(ctypes.Structure):                # muffin::Geom (internal.h)
    _fields_ = [(k, ctypes.c_int) for k in ("n", "L", "J", "gen", "j1", "cs", "dict", "vec", "fnt", "cnt")]


def rule(lib, name, n, L, J, j1):
    f = getattr(lib.lib, "_ZN6muffin%d%sERKNS_4GeomE" % (len(name), name))
    f.argtypes, f.restype = [ctypes.POINTER(Geom)], ctypes.c_bool
    return f(ctypes.byref(Geom(n, L, J, 1, j1, 0, 0, 1, 256, 256)))


# n, channels, J, fine levels, channels of a group, whether the coarse levels march too
@pytest.mark.parametrize("n,L,J,j1,group,coarse", [(128, 260, 3, 1, 100, False), (128, 257, 3, 3, 100, False),
                                                   (128, 258, 4, 2, 127, False), (256, 65, 4, 2, 31, False),
                                                   (256, 67, 3, 3, 29, False), (512, 17, 5, 3, 7, False),
                                                   (512, 19, 2, 2, 5, False), (1024, 5, 3, 3, 1, False),
                                                   (1024, 9, 4, 3, 1, True), (1024, 9, 5, 3, 1, True)])
@pytest.mark.parametrize("rho", [1.0, 1.3])
def test_march_is_bitwise_the_tile_kernels(lib, n, L, J, j1, group, coarse, rho, monkeypatch):
    monkeypatch.delenv("MUFFIN_IUWT_GENERAL", raising=False)
    for name in ("iuwt_march_analysis", "iuwt_march_adjoint"):
        assert rule(lib, name, n, L, J, j1) and not rule(lib, name, n, group, J, j1)
    assert rule(lib, "coarse_march_ok", n, L, J, j1) == coarse and not rule(lib, "coarse_march_ok", n, group, J, j1)
    g = torch.Generator(device="cuda").manual_seed(n + L)
    dirty = torch.randn(L, n, n, device="cuda", generator=g)
    psf = torch.zeros(L, n, n, device="cuda")
    psf[:, n // 2, n // 2] = 1.0
    psf[:, n // 2, n // 2 + 1] = 0.25
    state = [torch.rand(L, n, n, device="cuda", generator=g)]
    state += [(1.5 * torch.randn(*s, device="cuda", generator=g)).clamp(-1, 1) for s in ((L, J + 1, n, n), (L, n, n))]
    out = []
    for plan in (L, group):
        m = lib.Muffin(dirty, psf, nscales=J, tau=0.02, rho=rho, fine_levels=j1, power_iters=1)
        m.set_plan(plan, 1)
        m.set_state(*state, 0)
        m.iterate(3)
        out.append(m.get_state()[:3])
        torch.cuda.synchronize()
        m.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
