"""The long sums and the scaling of the power method (k_misc.cu), called through the library's
internal launchers: on integers a double holds every partial sum exactly, and
so must the sums in floats between two additions to a double."""
import ctypes
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

_P, _S = ctypes.c_void_p, ctypes.c_size_t


def stream():
    return torch.cuda.current_stream().cuda_stream


def dot(lib, a, b):
    """The partial sums of k_dot, added on the host (without rounding where they are finite)."""
    f = lib.lib._ZN6muffin10launch_dotEPKfS1_mPdPiP11CUstream_st     # muffin::launch_dot
    f.argtypes, f.restype = [_P, _P, _S, _P, ctypes.POINTER(ctypes.c_int), _P], ctypes.c_int
    parts, np = torch.zeros(1024, dtype=torch.float64, device="cuda"), ctypes.c_int()
    assert f(a.data_ptr(), b.data_ptr(), a.numel(), parts.data_ptr(), ctypes.byref(np), stream()) == 0
    parts = parts[:np.value].tolist()
    return math.fsum(parts) if all(map(math.isfinite, parts)) else sum(parts)


def place(t, offset):
    """t on the GPU, `offset` floats past a 16-byte boundary."""
    buf = torch.zeros(t.numel() + 8, device="cuda")
    out = buf[offset:offset + t.numel()]
    out.copy_(t)
    return out


@pytest.mark.parametrize("n", [1, 3, 4, 16, 17, 115, 1027, 4096, 4099])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("lo", [-1, 0])          # both signs, and one
def test_dot_is_exact_where_doubles_are(lib, n, offset, lo):
    g = torch.Generator().manual_seed(100 * n + offset)
    # at most 115 products that are not zero, so every partial sum is below 115 * 2^46 < 2^53; in the long ones they
    # are the 16 products of each of the first threads: float4 t + 256 e of a block of 256 threads
    keep = torch.arange(n) if n <= 115 else torch.tensor([4 * (t + 256 * e) + c for t in range(7) for e in range(4)
                                                          for c in range(4) if 4 * (t + 256 * e) + c < n])
    for _ in range(20):
        a, b = torch.zeros(n, dtype=torch.int64), torch.zeros(n, dtype=torch.int64)
        a[keep] = torch.randint(lo * 2 ** 23 + 1, 2 ** 23, (len(keep),), generator=g)
        b[keep] = torch.randint(lo * 2 ** 23 + 1, 2 ** 23, (len(keep),), generator=g)
        exact = sum(x * y for x, y in zip(a.tolist(), b.tolist()))
        assert dot(lib, place(a.float(), offset), place(b.float(), offset)) == exact


@pytest.mark.parametrize("offset", [0, 3])
def test_dot_long_and_out_of_range(lib, offset):
    g = torch.Generator().manual_seed(7)
    n = (1 << 20) + 5
    a, b = torch.randn(n, generator=g), torch.randn(n, generator=g)
    scale = torch.ones(n)
    scale[1000:3000] = 2.0 ** -80            # products below the range in which their errors are floats
    scale[5000:5100] = 2.0 ** 50             # and sums near its end
    a *= scale
    b *= scale
    terms = (a.double() * b.double()).tolist()
    exact = math.fsum(terms)
    got = dot(lib, place(a, offset), place(b, offset))
    # at most ceil(n / 2^18) = 5 values or groups a thread (one a group in the unaligned case), three additions a group,
    # five levels of a warp and five of a block, each rounding to 2^-53 of a sum of at most the magnitudes
    assert abs(got - exact) <= 32 * 2.0 ** -53 * math.fsum(abs(t) for t in terms)
    for bad, check in ((float("inf"), math.isinf), (float("nan"), math.isnan)):
        a[777] = bad
        b[777] = 1.0
        assert check(dot(lib, place(a, offset), place(b, offset)))


@pytest.mark.parametrize("offset", [0, 1])
def test_scale_rounds_the_double_product(lib, offset):
    """x <- (float)((double)x * f) to the bit, for every significand and both paths of the kernel."""
    fn = lib.lib._ZN6muffin12launch_scaleEPfmPKdS2_P11CUstream_st    # muffin::launch_scale
    fn.argtypes, fn.restype = [_P, _S, _P, _P, _P], ctypes.c_int
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    ordinary = (torch.arange(2 ** 23, dtype=torch.int32, device="cuda") + 0x3F800000).view(torch.float32)   # [1, 2)
    g = torch.Generator(device="cuda").manual_seed(5)
    wild = torch.randint(-2 ** 31, 2 ** 31, (2 ** 20 + 3,), device="cuda", generator=g).int().view(torch.float32)
    wild[:4] = torch.tensor([0.0, -0.0, float("inf"), float("-inf")])    # any bits: every exponent, NaNs among them
    factors = [(0.5 + k / 23.0) ** 0.5 for k in range(12)] + [1.0, 0.25, 3.1e-5, 7.7e8]
    factors += [1e-31, 3e-38, 1e-44, 1e31, 1e300, 0.0, float("inf"), float("nan")]   # factors without two floats
    for x in (ordinary, wild):
        for f in factors if x is wild else factors[:16]:
            num = torch.tensor([f], dtype=torch.float64, device="cuda")
            got = place(x, offset)
            assert fn(got.data_ptr(), got.numel(), num.data_ptr(), one.data_ptr(), stream()) == 0
            want = (x.double() * f).float()
            same = (got.view(torch.int32) == want.view(torch.int32)) | (got.isnan() & want.isnan())
            assert bool(same.all()), (f, x[~same][:3], got[~same][:3], want[~same][:3])


def cancelling(g, groups, small):
    """8 * groups + 3 integers of at most 24 significant bits, one large in eight and small odd ones behind it, that add
    up to `small`; every partial sum is below 2^53."""
    v = 2 * torch.randint(2 ** 22, 2 ** 23, (8 * groups,), generator=g) + 1
    v[::8] <<= 23
    v = v.tolist()
    rest = small - sum(v)
    for _ in range(3):
        step = max(abs(rest).bit_length() - 24, 0)
        v.append((abs(rest) >> step << step) * (1 if rest > 0 else -1))
        rest -= v[-1]
    assert rest == 0
    return v


@pytest.mark.parametrize("groups", [1, 2, 5, 19])
def test_reduction_of_partial_sums_keeps_the_bits_of_doubles(lib, groups):
    """Weight and bias gradients from their blocks' partial sums (k_net.cu), through mnet::launch_reduce."""
    f = lib.lib._ZN4mnet13launch_reduceEPKfiiPfiiS1_S2_P11CUstream_st
    f.argtypes, f.restype = [_P, ctypes.c_int, ctypes.c_int, _P, ctypes.c_int, ctypes.c_int, _P, _P, _P], None
    g = torch.Generator().manual_seed(groups)
    n, P, want = 64, 8 * groups + 3, list(range(-48, 48))
    v = torch.tensor([cancelling(g, groups, s) for s in want], dtype=torch.float64).T.contiguous()     # [P][n + 32]
    assert torch.equal(v.float().double(), v)
    part, bpart = v[:, :n].float().cuda(), v[:, n:].float().cuda()
    out, bout = torch.zeros(27 * 1024, device="cuda"), torch.zeros(32, device="cuda")
    for bad in (None, float("inf"), float("nan")):
        if bad is not None:
            part[1, 5] = bad
            want[5] = bad
        f(part.contiguous().data_ptr(), P, n, out.data_ptr(), 1, 1, bpart.contiguous().data_ptr(), bout.data_ptr(), stream())
        # output i = (tap 0, co i / 32, ci i % 32) goes to (co 32 + ci) 27
        got = torch.cat([out[:27 * n:27], bout]).cpu()
        assert torch.equal(torch.nan_to_num(got, nan=1e30), torch.nan_to_num(torch.tensor(want, dtype=torch.float32), nan=1e30))
