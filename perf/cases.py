"""What the performance of this library is measured on.

Each case is one call, or a short run of calls, that a program makes through
the public Python binding: passes of Algorithm 1 on cubes of the sizes this
repository is configured, tested and benchmarked with, the objective, a whole
solve, a batch of uneven cubes, and the warm-start network (prediction,
gradient, single layers).  Inputs are synthetic cubes made on the GPU from a
seed, with the recipe of ``paper_1602_08847_gb300.synth``: Gaussian sources with
power-law spectra, a PSF from a uv mask of random antennas, noise at 20 dB.
Step sizes are pinned from the closed-form norms, so that a 64-bit evaluation
needs nothing of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1602_08847_gb300.muffin import Batch, Muffin, solve
from paper_1602_08847_gb300.net import (WarmStartNet, conv3d_backward_data, conv3d_backward_weights,
                                        conv3d_forward)

DEV = "cuda"
MU_S, MU_L = 0.25, 3.0
LARGEST_VOXELS = 512 * 512 * 256


def _pass(name, n, L, J, **more):
    return {"name": name, "kind": "pass", "n": n, "L": L, "J": J, "gen": 1, "dict": "iuwt", "mu_l": MU_L,
            "rho": 1.0, "weights": False, "passes": 10, **more}


def listed() -> list[dict]:
    return [
        # the smallest configuration: ten passes between two looks at the state (the stopping test is
        # made every ten passes); launches and latency count
        _pass("pass 64x64x8", 64, 8, 3),
        # the ordinary cube, the size the warm-start network is trained on
        _pass("pass 256x256x64", 256, 64, 4),
        # the benchmark's cube, the largest
        _pass("pass 512x512x256", 512, 256, 5),
        # few channels of large images (a member of the uneven batch, run alone)
        _pass("pass 1024x1024x8", 1024, 8, 4),
        # second-generation wavelets, over-relaxed, noise-weighted channels whose number is no power of two
        _pass("pass 128x128x37 gen2", 128, 37, 4, gen=2, rho=1.3, weights=True),
        # the union of eight Daubechies bases, the dictionary the paper compares with
        _pass("pass 256x256x64 union", 256, 64, 4, dict="union"),
        # four cubes of uneven sizes advanced together
        {"name": "batch of four", "kind": "batch", "cubes": "128x16,256x32,512x64,1024x8", "J": 4, "passes": 10},
        # the stopping test: objective in double precision
        {"name": "objective 256x256x64", "kind": "objective", "n": 256, "L": 64, "J": 4, "gen": 1},
        # a whole call on a new cube: set-up, norms, fifty passes (what the network takes as its input)
        {"name": "solve 256x256x64", "kind": "solve", "n": 256, "L": 64, "J": 4, "gen": 1, "passes": 50},
        # the network's prediction of a starting state (cube and five dual planes)
        {"name": "predict 64x256x256", "kind": "predict", "nz": 64, "ny": 256, "nx": 256, "K": 6},
        # one training gradient on such a cube
        {"name": "gradient 64x256x256", "kind": "gradient", "nz": 64, "ny": 256, "nx": 256, "K": 6},
        # one 32 -> 32 layer on a ragged cube, forward and backward, as a program that composes its own network calls it
        {"name": "layer 31x120x100", "kind": "layer", "nz": 31, "ny": 120, "nx": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["pass", "pass", "pass", "pass", "union", "batch", "objective", "solve", "predict", "gradient",
                       "layer", "layer"])
    if kind in ("pass", "union", "objective", "solve"):
        n = rng.choice([64, 128, 256, 512, 1024])
        # the union costs about four times, second-generation wavelets about twice an ordinary pass
        gen = 1 if kind == "union" else rng.choice([1, 1, 1, 2])
        most = LARGEST_VOXELS // (8 if kind == "union" else 4 if gen == 2 or kind != "pass" else 1)
        L = _log_int(rng, 5, max(6, min(256, most // (n * n))))
        if rng.random() < 0.5:                     # powers of two have a fast spectral transform
            L = 1 << (L.bit_length() - 1)
        elif L > 96:                               # the others a matrix product
            L = 96 - L % 7
        J = rng.randint(2, 4 if n <= 64 else 5)
        if kind == "objective":
            return {"kind": "objective", "n": n, "L": L, "J": J, "gen": gen}
        if kind == "solve":
            return {"kind": "solve", "n": n, "L": L, "J": J, "gen": gen, "passes": rng.randint(10, 60)}
        c = _pass("", n, L, J, gen=gen, mu_l=rng.choice([MU_L, MU_L, 0.0]), rho=rng.choice([1.0, 1.0, 1.3]),
                  weights=rng.random() < 0.3, dict="union" if kind == "union" else "iuwt", passes=rng.randint(2, 10))
        del c["name"]
        return c
    if kind == "batch":
        cubes = []
        for _ in range(rng.randint(2, 4)):
            n = rng.choice([64, 128, 256, 512])
            cubes.append("%dx%d" % (n, _log_int(rng, 5, min(64, (1 << 22) * 4 // (n * n)))))
        return {"kind": "batch", "cubes": ",".join(cubes), "J": rng.randint(2, 4), "passes": rng.randint(2, 10)}
    nz, ny, nx = _log_int(rng, 5, 64), _log_int(rng, 24, 256), _log_int(rng, 24, 256)
    c = {"kind": kind, "nz": nz, "ny": ny, "nx": nx}
    return c if kind == "layer" else {**c, "K": rng.randint(1, 8)}


# ---------------------------------------------------------------- inputs

def _gen(seed: int, salt: int = 0) -> torch.Generator:
    return torch.Generator(device=DEV).manual_seed(1000003 * salt + seed)


def _cube(n: int, L: int, seed: int):
    """(dirty, psf, sky): float32 [L][n][n] on the GPU."""
    g = _gen(seed)
    big = n >= 512 and L >= 128
    n_src, n_ant = (200, 128) if big else (40, 60) if n >= 128 else (5, 20)
    u = lambda k, lo, hi: torch.rand(k, device=DEV, generator=g) * (hi - lo) + lo  # noqa: E731
    freqs = torch.linspace(1.0, 1.5, L, device=DEV)
    cy, cx, width, peak, alpha = u(n_src, 0, n), u(n_src, 0, n), u(n_src, 1, 4), u(n_src, 0.5, 2), u(n_src, 0.5, 1)
    pix = torch.arange(n, device=DEV, dtype=torch.float32)
    gy = torch.exp(-((pix[None] - cy[:, None]) ** 2) / (2 * width[:, None] ** 2))
    gx = torch.exp(-((pix[None] - cx[:, None]) ** 2) / (2 * width[:, None] ** 2))
    spectra = peak[None] * (freqs[:, None] / 1.25) ** (-alpha[None])               # [L][n_src]
    sky = torch.matmul((spectra[:, :, None] * gy[None]).transpose(1, 2), gx)       # [L][n][n]
    ant = torch.rand(n_ant, 2, device=DEV, generator=g) * 2 - 1
    base = (ant[:, None] - ant[None]).reshape(-1, 2)                               # both signs and (0, 0)
    cells = torch.round(base[None] * (freqs[:, None, None] / 1.5) * (n / 5.0)).long() % n
    mask = torch.zeros(L, n * n, device=DEV)
    mask.scatter_(1, cells[..., 0] * n + cells[..., 1], 1.0)
    mask = mask.view(L, n, n)
    psf = torch.fft.ifft2(mask).real
    psf = psf / psf[:, :1, :1]
    h = torch.fft.rfft2(psf)
    clean = torch.fft.irfft2(h * torch.fft.rfft2(sky), s=(n, n))
    noise = clean.square().mean(dim=(1, 2), keepdim=True).sqrt() * 0.1             # 20 dB
    dirty = clean + noise * torch.randn(L, n, n, device=DEV, generator=g)
    return dirty.contiguous(), torch.fft.fftshift(psf, dim=(1, 2)).contiguous(), sky


def _state(sky, planes: int, seed: int):
    """A state from inside a run: a non-negative cube, duals in [-1, 1], some at their bounds."""
    g = _gen(seed, 1)
    L, n, _ = sky.shape
    x = (sky + 0.05 * torch.randn(L, n, n, device=DEV, generator=g)).clamp_(min=0)
    u = (0.6 * torch.randn(L, planes, n, n, device=DEV, generator=g)).clamp_(-1, 1)
    v = (0.6 * torch.randn(L, n, n, device=DEV, generator=g)).clamp_(-1, 1)
    return x, u, v


def _weights(L: int, on: bool) -> list[float]:
    return [1.0 + 0.5 * math.sin(1.7 * l) for l in range(L)] if on else [1.0] * L


def _ws_norm2(n: int, J: int, gen: int, dictionary: str) -> float:
    """||W_s||^2 from the transfer functions (the union of bases is a tight frame)."""
    if dictionary == "union" or J == 0:
        return 1.0
    t = 2 * np.pi * np.arange(n) / n
    a, total = np.ones((n, n)), np.zeros((n, n))
    for j in range(J):
        r = (6 + 8 * np.cos(2 ** j * t) + 2 * np.cos(2 ** (j + 1) * t)) / 16
        h = r[:, None] * r[None]
        total += ((1 - (h if gen == 1 else h * h)) * a) ** 2
        a = a * h
    return float((total + a ** 2).max())


def _tau(psf, w, J, gen, dictionary, mu_l) -> float:
    """Primal step by Condat's rule from the exact norms."""
    n = psf.shape[-1]
    top = torch.fft.rfft2(psf.double()).abs().square().amax(dim=(1, 2))
    beta = float((top * torch.tensor(w, dtype=torch.float64, device=DEV)).max())
    return 0.99 / (beta / 2 + MU_S ** 2 * _ws_norm2(n, J, gen, dictionary) + mu_l ** 2)


def _planes(c) -> int:
    return 8 if c.get("dict") == "union" else c["J"] + 1


def _problem_of(c, n, L, seed):
    """What one cube's problem is made of (the same for the library and for the 64-bit evaluation)."""
    dirty, psf, sky = _cube(n, L, seed)
    w = _weights(L, c.get("weights", False))
    tau = _tau(psf, w, c["J"], c.get("gen", 1), c.get("dict", "iuwt"), c.get("mu_l", MU_L))
    return dirty, psf, sky, w, tau


def _muffin(c, n, L, seed):
    dirty, psf, sky, w, tau = _problem_of(c, n, L, seed)
    m = Muffin(dirty, psf, nscales=c["J"], gen=c.get("gen", 1), mu_s=MU_S, mu_l=c.get("mu_l", MU_L), tau=tau,
               rho=c.get("rho", 1.0), weights=w if c.get("weights") else None, dictionary=c.get("dict", "iuwt"))
    m.set_state(*_state(sky, _planes(c), seed), 0)
    return m


def _sizes(c):
    return [tuple(int(v) for v in s.split("x")) for s in c["cubes"].split(",")]


def _theta(K: int, seed: int):
    """He-normal weights on the bfloat16 grid, small biases, packed as the library takes them."""
    g = _gen(seed, 2)
    parts = []
    for k, (ci, co) in enumerate([(1, 32)] + [(32, 32)] * 4 + [(32, K)]):
        w = torch.randn(co * ci * 27, device=DEV, generator=g) * math.sqrt(2.0 / (27 * ci)) * (0.3 if k == 5 else 1.0)
        parts += [w.bfloat16().float(), 0.05 * torch.randn(co, device=DEV, generator=g)]
    return torch.cat(parts)


def _lam(K: int) -> list[float]:
    return [1000.0, 4.0][:K] + [1.0] * max(0, K - 2)


def _net_inputs(c, seed):
    """(cube, target cube, target fields): a blurred noisy sky, the sky, duals in [-1, 1]."""
    g = _gen(seed, 3)
    shape = (c["nz"], c["ny"], c["nx"])
    t = torch.randn(shape, device=DEV, generator=g).clamp_(min=0) * 2
    y = torch.nn.functional.avg_pool3d(t[None, None], 3, 1, 1)[0, 0] + 0.1 * torch.randn(shape, device=DEV, generator=g)
    aux = None
    if c["K"] > 1:
        aux = (0.6 * torch.randn((c["nz"], c["K"] - 1, c["ny"], c["nx"]), device=DEV, generator=g)).clamp_(-1, 1)
        aux = aux.bfloat16()
    return y.contiguous(), t.contiguous(), aux


def _layer_inputs(c, seed):
    g = _gen(seed, 4)
    shape = (c["nz"], c["ny"], c["nx"], 32)
    a = torch.randn(shape, device=DEV, generator=g).clamp_(min=0).bfloat16()
    dz = (0.01 * torch.randn(shape, device=DEV, generator=g)).bfloat16()
    w = (torch.randn((32, 32, 3, 3, 3), device=DEV, generator=g) * math.sqrt(2.0 / 864)).bfloat16().float()
    return a, dz, w, 0.05 * torch.randn(32, device=DEV, generator=g)


def prepare(case: dict, seed: int):
    k = case["kind"]
    if k in ("pass", "objective"):
        return {"case": case, "m": _muffin(case, case["n"], case["L"], seed)}
    if k == "batch":
        ms = [_muffin(case, n, L, seed + 101 * i) for i, (n, L) in enumerate(_sizes(case))]
        return {"case": case, "ms": ms, "b": Batch(ms)}
    if k == "solve":
        dirty, psf, _, _, tau = _problem_of(case, case["n"], case["L"], seed)
        return {"case": case, "dirty": dirty, "psf": psf, "tau": tau}
    if k in ("predict", "gradient"):
        y, t, aux = _net_inputs(case, seed)
        net = WarmStartNet((case["nz"], case["ny"], case["nx"]), training=k == "gradient",
                           theta=_theta(case["K"], seed), n_out=case["K"], out_weight=_lam(case["K"]))
        return {"case": case, "net": net, "y": y, "t": t, "aux": aux}
    return {"case": case, "in": _layer_inputs(case, seed)}


# ---------------------------------------------------------------- the calls

def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "pass":
        state["m"].iterate(c["passes"])
        x, u, v, _ = state["m"].get_state()
        return {"x": x, "u": u, "v": v}
    if k == "batch":
        state["b"].iterate(c["passes"])
        out = []
        for m in state["ms"]:
            x, u, v, _ = m.get_state()
            out.append({"x": x, "u": u, "v": v})
        return out
    if k == "objective":
        total, terms = state["m"].objective()
        return {"total": total, "terms": list(terms)}
    if k == "solve":
        return solve(state["dirty"], state["psf"], c["passes"], nscales=c["J"], gen=c["gen"], mu_s=MU_S, mu_l=MU_L,
                     tau=state["tau"])
    if k == "predict":
        x, aux = state["net"].predict(state["y"])
        return {"x": x, "aux": aux}
    if k == "gradient":
        value, g = state["net"].loss_grad(state["y"], state["t"], state["aux"])
        return {"loss": value, "gradient": g}
    a, dz, w, b = state["in"]
    dw, db = conv3d_backward_weights(a, dz)
    return {"z": conv3d_forward(a, w, b, True), "da": conv3d_backward_data(dz, w, a), "dw": dw, "db": db}


# ---------------------------------------------------------------- what a pass cannot do without

def _pass_work(n, L, J, dictionary, mu_l, passes, state=True):
    v = n * n * L
    planes = 8 if dictionary == "union" else J + 1
    # X, U, V read and written once, b and the Fourier multiplier (half of the plane) read once
    per = 8 + 8 * planes + (8 if mu_l else 0) + 4 + 2
    flops = 10 * math.log2(n) * 2 + 6 * planes + 12
    flops += 8 * 27 * 4 if dictionary == "union" else J * 2 * 18
    flops += 2 * 5 * math.log2(max(L, 2)) + 6 if mu_l else 0
    copy = 2 * 4 * (planes + 2) if state else 0
    return v * (per * passes + copy), v * flops * passes


def work(case: dict) -> dict:
    k = case["kind"]
    if k == "pass":
        b, f = _pass_work(case["n"], case["L"], case["J"], case["dict"], case["mu_l"], case["passes"])
    elif k == "batch":
        got = [_pass_work(n, L, case["J"], "iuwt", MU_L, case["passes"]) for n, L in _sizes(case)]
        b, f = sum(x for x, _ in got), sum(y for _, y in got)
    elif k == "objective":
        v = case["n"] ** 2 * case["L"]
        # X, and the complex double transforms of PSF and dirty cube
        b, f = v * (4 + 32), v * (10 * math.log2(case["n"]) + case["J"] * 18 + 5 * math.log2(max(case["L"], 2)) + 20)
    elif k == "solve":
        b, f = _pass_work(case["n"], case["L"], case["J"], "iuwt", MU_L, case["passes"], state=False)
        b += case["n"] ** 2 * case["L"] * 12
    else:
        v = case["nz"] * case["ny"] * case["nx"]
        if k == "layer":
            b, f = v * 64 * 6, v * 2 * 27648 * 3
        else:
            K = case["K"]
            fwd = 2 * 27 * (32 + 4 * 1024 + 32 * K)
            b, f = v * (4 + 4 * K), v * fwd
            if k == "gradient":
                b, f = v * (8 + 2 * (K - 1)), v * (3 * fwd - 2 * 27 * 32)
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch

def _smooth(c, d):
    for axis in (-1, -2):
        c = (6 * c + 4 * (torch.roll(c, d, axis) + torch.roll(c, -d, axis))
             + torch.roll(c, 2 * d, axis) + torch.roll(c, -2 * d, axis)) / 16
    return c


def _daubechies(p):
    q = np.array([1.0 + 0j])
    if p > 1:
        for y in np.roots([math.comb(p - 1 + k, k) for k in range(p)][::-1]):
            a = 1 - 2 * y
            r = np.sqrt(a * a - 1 + 0j)
            z = a + r if abs(a + r) < 1 else a - r
            q = np.convolve(q, [1, -z]) / (1 - z)
    binom = np.array([math.comb(p, t) for t in range(p + 1)]) / 2.0 ** p
    return np.sqrt(2.0) * np.real(np.convolve(binom, q))


def _dwt_matrix(p, M):
    """One periodic analysis step on vectors of length M: [low | high]."""
    h = _daubechies(p)
    g = (-1.0) ** np.arange(2 * p) * h[::-1]
    A = np.zeros((M, M))
    for k in range(M // 2):
        for t in range(2 * p):
            A[k, (2 * k + t) % M] += h[t]
            A[M // 2 + k, (2 * k + t) % M] += g[t]
    return torch.from_numpy(A).to(DEV)


class _Spatial:
    """W_s and its adjoint."""

    def __init__(self, c, n):
        self.J, self.gen, self.union = c["J"], c.get("gen", 1), c.get("dict") == "union"
        if self.union:
            self.A = [[_dwt_matrix(p, n >> j) for j in range(self.J)] for p in range(1, 9)]

    def analysis(self, x):
        out = []
        if self.union:
            for A in self.A:
                c = x.clone()
                for a in A:
                    M = a.shape[0]
                    c[..., :M, :M] = a @ c[..., :M, :M] @ a.T
                out.append(c / math.sqrt(8))
        else:
            c = x
            for j in range(self.J):
                nxt = _smooth(c, 2 ** j)
                out.append(c - (nxt if self.gen == 1 else _smooth(nxt, 2 ** j)))
                c = nxt
            out.append(c)
        return torch.stack(out, dim=1)

    def adjoint(self, u):
        if self.union:
            total = 0
            for i, A in enumerate(self.A):
                c = u[:, i].clone()
                for a in reversed(A):
                    M = a.shape[0]
                    c[..., :M, :M] = a.T @ c[..., :M, :M] @ a
                total = total + c / math.sqrt(8)
            return total
        r = u[:, self.J]
        for j in range(self.J - 1, -1, -1):
            uj = u[:, j]
            r = uj + _smooth(r - (uj if self.gen == 1 else _smooth(uj, 2 ** j)), 2 ** j)
        return r


def _dct(L):
    k = torch.arange(L, dtype=torch.float64, device=DEV)
    C = torch.cos(math.pi * (2 * k[None] + 1) * k[:, None] / (2 * L)) * math.sqrt(2.0 / L)
    C[0] = math.sqrt(1.0 / L)
    return C


def _exact_passes(c, n, L, seed, passes, start=True):
    dirty, psf, sky, w, tau = _problem_of(c, n, L, seed)
    if start:
        x, u, v = (t.double() for t in _state(sky, _planes(c), seed))
    else:
        x, v = (torch.zeros(L, n, n, dtype=torch.float64, device=DEV) for _ in range(2))
        u = torch.zeros(L, _planes(c), n, n, dtype=torch.float64, device=DEV)
    h = torch.fft.rfft2(torch.fft.ifftshift(psf.double(), dim=(1, 2)))
    w = torch.tensor(w, dtype=torch.float64, device=DEV)[:, None, None]
    K = w * h.abs().square()
    b = w * torch.fft.irfft2(h.conj() * torch.fft.rfft2(dirty.double()), s=(n, n))
    del h, dirty, psf, sky
    W, C = _Spatial(c, n), _dct(L)
    rho, mu_l = c.get("rho", 1.0), c.get("mu_l", MU_L)
    flat = lambda M, t: (M @ t.reshape(L, -1)).reshape(t.shape)  # noqa: E731
    for _ in range(passes):
        g = torch.fft.irfft2(K * torch.fft.rfft2(x), s=(n, n)) - b + MU_S * W.adjoint(u)
        if mu_l:
            g += mu_l * flat(C.T, v)
        xt = (x - tau * g).clamp_(min=0)
        del g
        d = 2 * xt - x
        ut = W.analysis(d).mul_(MU_S).add_(u).clamp_(-1, 1)
        u = ut if rho == 1 else rho * ut + (1 - rho) * u
        if mu_l:
            vt = (v + mu_l * flat(C, d)).clamp_(-1, 1)
            v = vt if rho == 1 else rho * vt + (1 - rho) * v
        x = xt if rho == 1 else rho * xt + (1 - rho) * x
    return {"x": x, "u": u, "v": v}


def _windows(a):
    """The 27 zero-padded shifts of a [z][y][x][f] map, in the order of the taps, each as a matrix."""
    z, y, x, f = a.shape
    ap = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        kz, ky, kx = t // 9, t // 3 % 3, t % 3
        yield t, ap[kz:kz + z, ky:ky + y, kx:kx + x].reshape(-1, f)


def _conv(a, w, b=None):
    """[z][y][x][ci] by [co][ci][3][3][3], zero padding."""
    co, w = w.shape[0], w.reshape(*w.shape[:2], 27)
    out = torch.zeros(a[..., 0].numel(), co, dtype=torch.float64, device=DEV)
    for t, m in _windows(a):
        out.addmm_(m, w[:, :, t].T)
    out = out.reshape(*a.shape[:3], co)
    return out if b is None else out + b


def _conv_back(dz, w):
    return _conv(dz, w.transpose(0, 1).flip(2, 3, 4))


def _conv_weights(a, dz):
    d = dz.reshape(-1, dz.shape[-1])
    dw = torch.empty(dz.shape[-1], a.shape[-1], 27, dtype=torch.float64, device=DEV)
    for t, m in _windows(a):
        dw[:, :, t] = d.T @ m
    return dw.reshape(*dw.shape[:2], 3, 3, 3), d.sum(0)


def _exact_net(c, seed):
    y, t, aux = _net_inputs(c, seed)
    K, theta = c["K"], _theta(c["K"], seed).double()
    layers, at = [], 0
    for ci, co in [(1, 32)] + [(32, 32)] * 4 + [(32, K)]:
        w = theta[at:at + co * ci * 27].reshape(co, ci, 3, 3, 3)
        layers.append((w, theta[at + co * ci * 27:at + co * (ci * 27 + 1)]))
        at += co * (ci * 27 + 1)
    y, s = y.double(), y.double().abs().max()
    acts = [(y / s)[..., None]]
    for i, (w, b) in enumerate(layers):
        z = _conv(acts[-1], w, b)
        acts.append(z.clamp_(min=0) if i < 5 else z)
    z = acts[-1]
    if c["kind"] == "predict":
        return {"x": (s * z[..., 0]).clamp(min=0), "aux": z[..., 1:].clamp(-1, 1).permute(0, 3, 1, 2) if K > 1 else None}
    target = (t.double() / s)[..., None]
    if aux is not None:
        target = torch.cat([target, aux.double().permute(0, 2, 3, 1)], dim=-1)
    lam = torch.tensor(_lam(K), dtype=torch.float64, device=DEV)
    r, v = z - target, y.numel()
    value = float((lam * r * r).sum() / v)
    dz, grads = 2 / v * lam * r, []
    for i in range(5, -1, -1):
        dw, db = _conv_weights(acts[i], dz)
        grads = [dw.reshape(-1), db] + grads
        if i:
            dz = _conv_back(dz, layers[i][0]) * (acts[i] > 0)
    return {"loss": value, "gradient": torch.cat(grads)}


def exact(case: dict, seed: int):
    k = case["kind"]
    if k == "pass":
        return _exact_passes(case, case["n"], case["L"], seed, case["passes"])
    if k == "batch":
        return [_exact_passes(case, n, L, seed + 101 * i, case["passes"]) for i, (n, L) in enumerate(_sizes(case))]
    if k == "solve":
        return _exact_passes(case, case["n"], case["L"], seed, case["passes"], start=False)["x"]
    if k == "objective":
        n, L = case["n"], case["L"]
        dirty, psf, sky, _, _ = _problem_of(case, n, L, seed)
        x = _state(sky, case["J"] + 1, seed)[0].double()
        h = torch.fft.rfft2(torch.fft.ifftshift(psf.double(), dim=(1, 2)))
        r = dirty.double() - torch.fft.irfft2(h * torch.fft.rfft2(x), s=(n, n))
        terms = [0.5 * float(r.square().sum()), MU_S * float(_Spatial(case, n).analysis(x).abs().sum()),
                 MU_L * float((_dct(L) @ x.reshape(L, -1)).abs().sum())]
        return {"total": sum(terms), "terms": terms}
    if k in ("predict", "gradient"):
        return _exact_net(case, seed)
    a, dz, w, b = (t.double() for t in _layer_inputs(case, seed))
    dw, db = _conv_weights(a, dz)
    return {"z": _conv(a, w, b).clamp_(min=0), "da": _conv_back(dz, w) * (a > 0), "dw": dw, "db": db}
