"""The marching tensor-core kernels of the network (k_net.cu): waits that run
out part of the way, at poll bounds between none and enough; and the kernels'
steady state (many tiles a block: full rings, every barrier phase, runs that
cross columns) on integers, where every result is exact."""
import pytest
import torch

from paper_1602_08847_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def netmod(lib):
    from paper_1602_08847_gb300 import net
    return net


@pytest.mark.parametrize("polls", [1, 2, 3, 5, 8, 13, 30, 100, 1000])
def test_waits_that_run_out_midway(netmod, polls):
    """With a small poll bound some warps give up and others do not, at any of
    the waits.  Every call returns, either with the result of an undisturbed
    run or with a give-up on record, and the next undisturbed run is right."""
    shape, K = (9, 70, 90), 2                 # 540 tiles: several a block, runs that cross columns
    theta = torch.from_numpy(synth.net_init(31, K).astype("float32")).cuda()
    y = torch.from_numpy(synth.random_field(shape, 32, -0.3, 1.0).astype("float32")).cuda()
    ta = torch.zeros((shape[0], K - 1, shape[1], shape[2]), dtype=torch.bfloat16, device="cuda")
    a = torch.relu(torch.from_numpy(synth.random_field(shape + (32,), 33).astype("float32"))).cuda().bfloat16()
    w = torch.from_numpy(synth.random_field((32, 32, 3, 3, 3), 34, -0.1, 0.1).astype("float32")).cuda()
    n = netmod.WarmStartNet(shape, training=True, theta=theta, n_out=K)

    def calls():
        yield lambda: (netmod.conv3d_forward(a, w, None, True),)
        yield lambda: (netmod.conv3d_backward_data(a, w, None),)
        yield lambda: netmod.conv3d_backward_weights(a, a)
        yield lambda: (n.loss_grad(y, torch.relu(y), ta)[1],)

    def guarded(f):
        try:
            out = f()
        except netmod._m.MuffinError as e:
            assert "TIMEOUT" in str(e)        # loss_grad reports (and clears) the give-ups itself
            return None
        torch.cuda.synchronize()
        return None if netmod.wait_timeouts() else out

    refs = [f() for f in calls()]
    assert netmod.wait_timeouts() == 0
    for f, ref in zip(calls(), refs):
        try:
            netmod.set_wait_limit(polls)
            got = guarded(f)
        finally:
            netmod.set_wait_limit(None)
        assert got is None or all(torch.equal(p, q) for p, q in zip(got, ref))
        assert all(torch.equal(p, q) for p, q in zip(f(), ref))
        assert netmod.wait_timeouts() == 0
    n.close()


# ---------------------------------------------------------------- exact references
#
# Small integers throughout: every product and every sum of the kernels is an
# integer (times a power of two) below 2^24, exact in float32 whatever the order
# and the rounding of the additions, so results are compared for equality.  The
# one rounding left, of a map to bfloat16, is to nearest even on both sides.

SHAPES = [(40, 20, 20),        # few tall columns: one tile a block
          (31, 120, 100),      # 3224 tiles of the layers: eleven a block (21 in the weight gradient), ragged edges
          (64, 200, 136),      # 14144: runs of 46 (93), whole columns and parts of two
          (3, 264, 520)]       # 3315, columns shorter than the rings


def ints(shape, seed, lo, hi, keep=1.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randint(lo, hi + 1, shape, device="cuda", generator=g).double()
    return v if keep == 1.0 else v * (torch.rand(shape, device="cuda", generator=g) < keep)


def windows(a):
    """The 27 zero-padded shifts of a [z][y][x][f] map, each as a matrix."""
    z, y, x, f = a.shape
    ap = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        kz, ky, kx = t // 9, t // 3 % 3, t % 3
        yield t, ap[kz:kz + z, ky:ky + y, kx:kx + x].reshape(-1, f)


def conv(a, w, b=None):
    w = w.reshape(*w.shape[:2], 27)
    out = torch.zeros(a[..., 0].numel(), w.shape[0], dtype=torch.float64, device="cuda")
    for t, m in windows(a):
        out.addmm_(m, w[:, :, t].T)
    out = out.reshape(*a.shape[:3], -1)
    return out if b is None else out + b


def conv_back(dz, w):
    return conv(dz, w.transpose(0, 1).flip(2, 3, 4))


def conv_weights(a, dz):
    d = dz.reshape(-1, dz.shape[-1])
    dw = torch.stack([d.T @ m for _, m in windows(a)], dim=2)
    return dw.reshape(*dw.shape[:2], 3, 3, 3), d.sum(0)


@pytest.mark.parametrize("shape", SHAPES)
def test_layers_exact(netmod, shape):
    a, dz = ints(shape + (32,), 1, 0, 2), ints(shape + (32,), 2, -2, 2)
    w, b = ints((32, 32, 3, 3, 3), 3, -3, 3), ints((32,), 4, -9, 9)
    assert 2 * 2 * a[..., 0].numel() < 2 ** 24
    A, D, W, B = a.bfloat16(), dz.bfloat16(), w.float(), b.float()
    z = conv(a, w, b)
    assert torch.equal(netmod.conv3d_forward(A, W, B, True), z.clamp(min=0).bfloat16())
    assert torch.equal(netmod.conv3d_forward(A, W, None, False), (z - b).bfloat16())
    da = conv_back(dz, w)
    assert torch.equal(netmod.conv3d_backward_data(D, W, None), da.bfloat16())
    assert torch.equal(netmod.conv3d_backward_data(D, W, A), (da * (a > 0)).bfloat16())
    dw, db = conv_weights(a, dz)
    got_w, got_b = netmod.conv3d_backward_weights(A, D)
    assert torch.equal(got_w, dw.float()) and torch.equal(got_b, db.float())
    assert netmod.wait_timeouts() == 0


def sparse_weights(co, ci, seed, per_row=3):
    """+-1 at per_row places of each output's 27 ci weights."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.zeros(co, ci * 27, dtype=torch.float64, device="cuda")
    at = torch.rand(co, ci * 27, device="cuda", generator=g).argsort(dim=1)[:, :per_row]
    sign = 2.0 * torch.randint(0, 2, at.shape, device="cuda", generator=g).double() - 1.0
    return w.scatter_(1, at, sign).reshape(co, ci, 3, 3, 3)


@pytest.mark.parametrize("shape,K", [((64, 100, 64), 1), ((64, 100, 64), 6), ((31, 120, 100), 8), ((7, 264, 264), 3)])
def test_network_exact(netmod, shape, K):
    """Prediction, loss and gradient: maps of integers of at most 3^5, from a sparse cube of zeros and ones and three
    weights of +-1 an output; loss weights that make the factor of the loss gradient a power of two."""
    V = shape[0] * shape[1] * shape[2]
    layers = [(sparse_weights(co, ci, 50 + i), torch.zeros(co, dtype=torch.float64, device="cuda"))
              for i, (ci, co) in enumerate([(1, 32)] + [(32, 32)] * 4 + [(32, K)])]
    theta = torch.cat([t.reshape(-1) for wb in layers for t in wb]).float()
    lam = [V / 2.0 ** (2 + k % 3) for k in range(K)]       # 2 / V lam = 2^-1, 2^-2, 2^-3
    y = ints(shape, 60, 1, 1, keep=0.03)
    tx = ints(shape, 61, 0, 3, keep=0.03)
    ta = ints((shape[0], K - 1) + shape[1:], 62, -1, 1, keep=0.03) if K > 1 else None
    assert float(y.max()) == 1.0
    acts = [y[..., None]]
    for i, (w, b) in enumerate(layers):
        z = conv(acts[-1], w, b)
        acts.append(z.clamp(min=0).bfloat16().double() if i < 5 else z)
    net = netmod.WarmStartNet(shape, theta=theta, n_out=K, out_weight=lam)
    x, aux = net.predict(y.float())
    assert torch.equal(x, acts[-1][..., 0].clamp(min=0).float())
    if K > 1:
        assert torch.equal(aux, acts[-1][..., 1:].clamp(-1, 1).permute(0, 3, 1, 2).float())
    net.close()
    target = tx[..., None] if ta is None else torch.cat([tx[..., None], ta.permute(0, 2, 3, 1)], dim=-1)
    r = acts[-1] - target
    L = torch.tensor(lam, dtype=torch.float64, device="cuda")
    loss = float((L * r * r).sum()) / V
    dz, grads = torch.tensor([2.0 * v / V for v in lam], dtype=torch.float64, device="cuda") * r, []   # powers of two
    for i in range(5, -1, -1):
        dw, db = conv_weights(acts[i], dz)
        # the premise: every sum of magnitudes stays below 2^24 units of 2^-3 (one unit of the loss gradient)
        mw, mb = conv_weights(acts[i].abs(), dz.abs())
        assert max(float(mw.max()), float(mb.max())) * 8 < 2 ** 24
        grads = [dw.reshape(-1), db] + grads
        if i:
            dz = (conv_back(dz, layers[i][0]) * (acts[i] > 0)).bfloat16().double()
    net = netmod.WarmStartNet(shape, training=True, theta=theta, n_out=K, out_weight=lam)
    got, g = net.loss_grad(y.float(), tx.float(), None if ta is None else ta.bfloat16().contiguous())
    assert got == loss
    want = torch.cat(grads).float()
    assert float(want.abs().max()) > 0 and torch.equal(g, want)
    net.close()
    assert netmod.wait_timeouts() == 0


def test_weight_gradient_accumulators_are_flushed(netmod):
    """One full column of tiles after another, 1024 of 152 runs of six or seven.  The first tile of every run adds 2^21
    to the centre tap, after which the tensor core truncates the others' steps of 2^-4 away (a unit is 2^-2); a flush
    after five planes, which reach at most the first five tiles, lets those of the tiles behind it through."""
    shape = (64, 32, 64)
    tiles, P = 1024, torch.cuda.get_device_properties(0).multi_processor_count
    if P != 152:
        pytest.skip("runs laid out for 152 blocks")
    dz = torch.full(shape + (32,), 2.0 ** -8, device="cuda")
    for b in range(P):
        t = tiles * b // P                       # column t / 64 (8 columns across, 16 rows), channel t % 64
        col, z = t // 64, t % 64
        y0, x0 = col // 8 * 16, col % 8 * 8
        dz[z, y0:y0 + 16, x0:x0 + 8] = 2.0 ** 14
    a = torch.ones(shape + (32,), device="cuda").bfloat16()
    dw, _ = netmod.conv3d_backward_weights(a, dz.bfloat16())
    large, small = P * 2.0 ** 21, (tiles - P) * 0.5
    # of the five or six small tiles of a run at least one comes through, and none is counted twice
    got = dw[:, :, 1, 1, 1].double() - large
    assert float(got.min()) >= small / 6 - 16 and float(got.max()) <= small + 16      # the result is rounded to 32


def bare_net(netmod, shape, K, b5, w6, lam):
    """A training net whose weights are zero but for the last layer's: its feature map is max(b5, 0) at every voxel."""
    theta = torch.zeros(netmod.n_params(K), dtype=torch.float64, device="cuda")
    last = netmod.n_params(K) - K * (32 * 27 + 1)
    theta[last - 32:last] = b5
    theta[last:last + K * 32 * 27] = w6
    return netmod.WarmStartNet(shape, training=True, theta=theta.float(), n_out=K, out_weight=lam), last


@pytest.mark.parametrize("shape,K", [((31, 120, 100), 1), ((31, 120, 100), 6), ((64, 200, 136), 3), ((7, 33, 41), 8)])
def test_last_weight_gradient_rounds_to_nearest(netmod, shape, K):
    """Terms of one sign and of many exponents, so that truncated additions would show as a bias (4e-7 over 32 of them).
    float32 sums rounded to nearest: a chain of n terms has an rms error of 0.289 2^-23 sqrt(n / 3) of its sum, P
    independent ones a sqrt(P)-th of that; four times it, and the rounding of the result.  That holds for map 0, whose
    targets are float32 values; the fields' are bfloat16, whose sums leave few different remainders."""
    nz, ny, nx = shape
    V = nz * ny * nx
    b5 = 1 + (4 * torch.arange(32, device="cuda").double() + 1) / 128
    net, last = bare_net(netmod, shape, K, b5, 0.0, [V / 2.0] * K)      # factor of the loss gradient: 1
    g = torch.Generator(device="cuda").manual_seed(3)
    y = torch.ones(shape, device="cuda")
    tx = torch.exp2(-6 * torch.rand(shape, device="cuda", generator=g))
    ta = torch.exp2(-6 * torch.rand((nz, K - 1, ny, nx), device="cuda", generator=g)).bfloat16() if K > 1 else None
    _, grad = net.loss_grad(y, tx, ta)
    d6 = -tx.double()[..., None] if ta is None else -torch.cat([tx[:, None].double(), ta.double()], 1).permute(0, 2, 3, 1)
    dw, _ = conv_weights(b5.expand(*shape, 32), d6)
    got = grad[last:last + K * 32 * 27].view(K, 32, 3, 3, 3).double()
    tiles = ((nx + 15) // 16) * ((ny + 7) // 8) * ((nz + 1) // 2)
    P = min(tiles, 304)
    n = 256 * -(-tiles // P)
    bound = 4 * 0.289 * 2.0 ** -23 * (n / 3 / P) ** 0.5 + 2.0 ** -24
    err = ((got - dw) / dw)[0]
    assert float(err.abs().max()) <= bound
    assert abs(float(err.mean())) <= bound / 32 ** 0.5        # and no bias: the features' errors are independent
    net.close()


def test_last_input_gradient_rounds_to_nearest(netmod):
    """One map, weights 1, a loss gradient of v everywhere: the last layer's input gradient is the sum of v over the
    taps inside the cube.  v is chosen so that 27 additions rounded to nearest end two to four units above a tie of the
    rounding to bfloat16, and truncated ones more than four below it.  Seen through the bias gradient of the layer
    before, the sum of the map over the cube."""
    import numpy as np

    def chain(v, n, nearest):
        s = np.zeros_like(v)
        for _ in range(n):
            exact = s.astype(np.float64) + v                  # exact in double
            t = exact.astype(np.float32)
            s = t if nearest else np.where(t > exact, np.nextafter(t, np.float32(0)), t)
        return s

    def above_tie(s):                                         # units of the last place above a tie of bfloat16
        return (s.view(np.uint32) & 0xFFFF).astype(int) - 0x8000

    vs = np.arange(0x3F800001, 0x40000000, 7, dtype=np.uint32).view(np.float32)
    up, down = above_tie(chain(vs, 27, True)), above_tie(chain(vs, 27, False))
    v = vs[(up >= 2) & (up <= 4) & (down < -4) & (down > -1000)][:1]
    shape = (6, 40, 40)
    V = 6 * 40 * 40
    net, last = bare_net(netmod, shape, 1, 2.0 ** -100, 1.0, [V / 2.0])
    _, grad = net.loss_grad(torch.ones(shape, device="cuda"), torch.full(shape, -float(v[0]), device="cuda"))
    want = 0.0
    for inner, count in ((4 * 38 * 38, 27), (2 * 38 * 38 + 2 * 4 * 38 * 2, 18), (2 * 38 * 4 + 4 * 4, 12), (2 * 4, 8)):
        want += inner * float(torch.from_numpy(chain(v, count, True)).bfloat16()[0])
    # a bfloat16 unit at the interior voxels is at least 2^-8 of most of the sum
    assert abs(grad[last - 32:last].double() / want - 1).max() <= 1e-4
    net.close()


def test_loss_sums_keep_the_bits_of_doubles(netmod):
    """Residuals that are integers at the voxels of four columns along the channel axis, where one thread sums a
    stretch of them, and zero elsewhere: one large value in eight and small odd ones behind it, which a sum in float
    pairs cannot hold.  The sums of lam r^2, and of r, stay below 2^53, so doubles hold every partial sum; those of r
    cancel to a small integer."""
    shape = (64, 200, 136)
    V = 64 * 200 * 136
    y = torch.ones(shape, device="cuda")
    g = torch.Generator().manual_seed(11)
    columns = [(5, 7), (77, 30), (150, 99), (199, 135)]
    lam = 2 ** 18 - 1
    net, last = bare_net(netmod, shape, 1, 0.0, 0.0, [float(lam)])
    tx = torch.zeros(shape)
    for r, c in columns:
        v = 2 * torch.randint(2, 5, (64,), generator=g) + 1                  # lam r^2 of 23 to 25 bits
        v[::8] = 2 * torch.randint(10000, 11000, (8,), generator=g) + 1      # of 47
        tx[:, r, c] = -v.float()
    total = lam * int((tx.double() ** 2).sum())
    loss, _ = net.loss_grad(y, tx.cuda())
    assert total < 2 ** 53 and loss == total / V
    net.close()
    net, last = bare_net(netmod, shape, 1, 0.0, 0.0, [1.0])
    for small in (3, -1001):
        tx = torch.zeros(shape)
        for r, c in columns:
            v = 2 * torch.randint(2 ** 22, 2 ** 23, (56,), generator=g) + 1  # odd, 24 bits
            v[::8] <<= 23
            v = v.tolist()
            rest = small - sum(v)                          # in three floats of at most 24 bits
            for _ in range(3):
                step = max(abs(rest).bit_length() - 24, 0)
                part = (abs(rest) >> step << step) * (1 if rest > 0 else -1)
                v.append(part)
                rest -= part
            assert rest == 0
            tx[:len(v), r, c] = -torch.tensor(v, dtype=torch.float64).float()
        _, grad = net.loss_grad(y, tx.cuda())
        assert float(grad[-1]) == float(torch.tensor(2.0 * len(columns) * small / V, dtype=torch.float64).float())
    net.close()
