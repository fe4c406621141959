"""What users of this framework have it compute, as measurable cases.

A case is one call pattern of the public Python API on inputs of one size: engine iterations of a
plan (`Reconstruction`, `ReconstructionBatch`), a monochromatisation call (`monochromatise`), a
warm-start estimate or training steps (`WarmStart`). Inputs are simulated measurements made on the
GPU from a seed (a smooth random object seen through a probe, partially coherent by a Gaussian
blur, Poisson counts), in the sizes of this repository's configurations and benchmark workloads.

`listed()` are fixed cases, `draw(rng)` gives others of the same ranges, `prepare(case, seed)` is
what a program holds before the call, `run(state)` one pass, `work(case)` the bytes and operations
a pass cannot do without, `exact(case, seed)` the first pass's result in 64 bits (plain torch).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_06640_gb300.engine import Reconstruction, ReconstructionBatch, monochromatise
from paper_2406_06640_gb300.warmstart import LatticeSpec, WarmStart, WarmStartConfig

EVERY_ITERATION = [(1, 1 << 30)]  # complex-constraint window over a whole run
FRESNEL_F = 10.0
DEV = "cuda"


def _engine_case(name, M, K, N, obj, scan, step, **kw):
    c = dict(kind="engine", name=name, M=M, K=K, N=N, obj=obj, scan=scan, step=step, geometry="far", blur="amplitude",
             sigma=1.5, taps=11, dose=1e6, corr=8.0, phase=3.14, rule="normalised", engine="pie", minibatch=0,
             constraint=True, monitor=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest reconstruction (64^2, one mode, 100 positions), the error read after every
        # iteration as an interactive run does: latency, launches and synchronisation count
        _engine_case("small64", 64, 1, 100, 192, "raster", 12, sigma=1.0, dose=1e5, monitor=True),
        # the headline workload: 900 far-field patterns of 128^2 on a Fermat spiral, four modes
        _engine_case("far128x4", 128, 4, 900, 640, "spiral", 6.0),
        # electron data: 4096 overlapping patterns, one mode, the intensity model with a wide kernel
        _engine_case("electron128", 128, 1, 4096, 256, "raster", 2, blur="intensity", sigma=2.0, taps=21, dose=2e4,
                     corr=1.5, phase=1.0, constraint=False),
        # the difference-map engine on the headline data (exit-wave state in device memory)
        _engine_case("dm128x4", 128, 4, 900, 640, "spiral", 6.0, engine="dm", constraint=False),
        # the sequential engine as mini-batches of 32 positions with rPIE steps
        _engine_case("minibatch128x4", 128, 4, 900, 640, "spiral", 6.0, rule="rpie", minibatch=32),
        # visible-light near field: 256^2, eight modes
        _engine_case("near256x8", 256, 8, 256, 1024, "raster", 20, geometry="near", sigma=2.0, dose=1e5, phase=0.5),
        # the largest tile, few positions, an object side that is no multiple of the tiles
        _engine_case("far512x2", 512, 2, 49, 805, "raster", 40, sigma=2.0, dose=1e6),
        # twelve reconstructions of uneven sizes in one plan, as a beamline queue submits them
        dict(kind="batch", name="batch12", members=12, mix=3, n_lo=100, n_hi=400),
        # broadband far-field data made monochromatic: 5 % bandwidth, every pattern of a scan
        dict(kind="mono", name="mono128", M=128, N=900, J=5, span=0.05, k=25),
        # white light on the large detector
        dict(kind="mono", name="mono256white", M=256, N=192, J=32, span=0.75, k=25),
        # the learned start: object and blur width from 64 sampled patterns
        dict(kind="estimate", name="estimate128", S=128, C=32, batch=64, N=64, step=16),
        # training that network on generated patterns, a few optimiser steps and the weights read back
        dict(kind="train", name="train128", S=128, C=32, batch=64, steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["engine"] * 5 + ["batch", "mono", "mono", "estimate", "train"])
    if kind == "engine":
        M = rng.choice([64, 128, 128, 256, 512])
        K = rng.choice([1, 2, 3, 4, 6, 8])
        # no more pattern-mode pixels than the headline workload (M <= 128) or the near-field one
        most = (3600 if M == 128 else 8192 if M == 64 else 1500 if M == 256 else 98) // K
        N = _log_int(rng, 30 if M < 512 else 9, max(31 if M < 512 else 10, most))
        side = math.ceil(math.sqrt(N))
        scan = rng.choice(["raster", "spiral"])
        step = rng.randint(2, max(3, M // 8))
        reach = (side - 1) * step if scan == "raster" else 2 * math.ceil(step / math.sqrt(math.pi) * math.sqrt(N))
        obj = M + reach + rng.randint(3, 60)
        engine = rng.choice(["pie", "pie", "pie", "dm"])
        batches = engine == "pie" and rng.random() < 0.25
        blur, geometry = rng.choice(["amplitude", "amplitude", "intensity"]), rng.choice(["far", "near"])
        return dict(kind="engine", M=M, K=K, N=N, obj=obj, scan=scan, step=step, geometry=geometry,
                    blur=blur, sigma=round(rng.uniform(0.5, 3.0), 3), taps=rng.choice([11, 11, 7, 21, 31]),
                    dose=math.exp(rng.uniform(math.log(1e5), math.log(1e6))), corr=round(rng.uniform(3.0, 8.0), 2),
                    phase=3.14 if geometry == "far" else 0.5, rule="rpie" if batches or rng.random() < 0.3 else "normalised", engine=engine,
                    minibatch=_log_int(rng, 8, 64) if batches else 0, constraint=engine == "pie" and rng.random() < 0.7,
                    monitor=rng.random() < 0.2)
    if kind == "batch":
        lo = rng.randint(40, 150)
        return dict(kind="batch", members=rng.randint(2, 12), mix=rng.randrange(1 << 20), n_lo=lo,
                    n_hi=lo + rng.randint(1, 250))
    if kind == "mono":
        M = rng.choice([64, 128, 128, 256])
        J = _log_int(rng, 3, 32)
        most = {64: 4000, 128: 28800, 256: 6144}[M]
        return dict(kind="mono", M=M, N=_log_int(rng, 20, max(21, min(1000, most // J))), J=J,
                    span=round(rng.uniform(0.02, 0.8), 3), k=rng.randint(5, 25))
    S = rng.choice([64, 128])
    batch = 2 * rng.randint(4, 32)
    if kind == "estimate":
        return dict(kind="estimate", S=S, C=rng.choice([16, 32]), batch=batch, N=rng.randint(3, 150),
                    step=rng.randint(5, S // 4))
    return dict(kind="train", S=S, C=rng.choice([16, 32]), batch=batch, steps=rng.randint(2, 4))


# ----------------------------------------------------------------------------- simulated measurements


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _smooth(gen, shape, corr):
    """White noise low-passed by a Gaussian of `corr` pixels (periodic), scaled to [0, 1]."""
    f = torch.fft.rfft2(torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64))
    ky = torch.fft.fftfreq(shape[0], device=DEV, dtype=torch.float64)[:, None]
    kx = torch.fft.rfftfreq(shape[1], device=DEV, dtype=torch.float64)[None]
    f = torch.fft.irfft2(f * torch.exp(-2 * (math.pi * corr) ** 2 * (ky ** 2 + kx ** 2)), s=shape)
    return (f - f.min()) / (f.max() - f.min())


def _positions(N, M, obj, scan, step, rng):
    if scan == "spiral":
        i = np.arange(N)
        r, a = step / math.sqrt(math.pi) * np.sqrt(i), i * math.pi * (3.0 - math.sqrt(5.0))
        pos = np.stack([r * np.sin(a), r * np.cos(a)], 1) + (obj - M) / 2
    else:
        cols = math.ceil(math.sqrt(N))
        pos = np.stack(np.divmod(np.arange(N), cols), 1) * float(step) + max(0, obj - M - (cols - 1) * step) // 2
        if step > 4:
            pos = pos + rng.integers(-1, 2, pos.shape)
    return np.clip(np.rint(pos), 0, obj - M).astype(np.int32)


def _radius(M):
    y = torch.arange(M, device=DEV, dtype=torch.float64) - (M - 1) / 2
    return torch.hypot(y[:, None], y[None])


def _fresnel(M):
    u = torch.fft.fftfreq(M, 1.0 / M, device=DEV, dtype=torch.float64)
    return torch.exp(-1j * math.pi * (u[:, None] ** 2 + u[None] ** 2) / (M * FRESNEL_F))


def _taps(sigma, half):
    d = torch.arange(-half, half + 1, device=DEV, dtype=torch.float64)
    g = torch.exp(-d * d / (2 * sigma * sigma)) if sigma > 0 else (d == 0).double()
    return g / g.sum()


def _blur(a, g):
    """Zero-padded separable correlation of (..., M, M) with the taps g on both axes."""
    h = len(g) // 2
    for dim in (-1, -2):
        p = torch.nn.functional.pad(a, (h, h, 0, 0) if dim == -1 else (0, 0, h, h))
        a = sum(w * p.narrow(dim, i, a.shape[dim]) for i, w in enumerate(g.tolist()))
    return a


def _boxes(field, pos, M):
    """(N, M, M) boxes of a 2-D field at the (row, col) corners pos (a device tensor)."""
    i = torch.arange(M, device=DEV)
    return field[pos[:, 0, None, None] + i[:, None], pos[:, 1, None, None] + i[None]]


def _simulate(c, seed):
    """Measured patterns, positions and first guess of one reconstruction."""
    gen, rng = _generator(seed), np.random.default_rng(seed)
    M, K, N, obj = c["M"], c["K"], c["N"], c["obj"]
    amp = 0.8 + 0.2 * _smooth(gen, (obj, obj), c["corr"])
    O = amp * torch.exp(1j * c["phase"] * _smooth(gen, (obj, obj), c["corr"]))
    r, far = _radius(M), c["geometry"] == "far"
    if far:  # a defocused disc
        rad = 0.3 * M
        P = (r <= rad) * torch.exp(4j * math.pi * (r / rad) ** 2)
    else:  # a diffuser in the beam
        P = torch.exp(-(r / (0.4 * M)) ** 8) * torch.exp(2j * math.pi * _smooth(gen, (M, M), 3.0))
    pos = _positions(N, M, obj, c["scan"], c["step"], rng)
    dpos, g = torch.from_numpy(pos.astype(np.int64)).to(DEV), _taps(c["sigma"], math.ceil(5 * c["sigma"]))
    I = torch.empty(N, M, M, device=DEV)
    for a in range(0, N, 128):
        psi = (P * _boxes(O, dpos[a:a + 128], M)).to(torch.complex64)
        if far:
            psi = torch.fft.fftshift(torch.fft.fft2(psi), dim=(-2, -1))
        else:
            psi = torch.fft.ifft2(torch.fft.fft2(psi) * _fresnel(M).to(torch.complex64))
        I[a:a + 128] = _blur(psi.abs().square(), g)
    I *= c["dose"] / I.sum(dim=(1, 2)).mean()
    I = torch.poisson(I, generator=gen)
    energy = float(I.sum(dtype=torch.float64)) / N / (M * M if far else 1)
    if not far:
        P = torch.complex(*(torch.nn.functional.avg_pool2d(x[None, None], 5, 1, 2)[0, 0] for x in (P.real, P.imag)))
    P0 = P * math.sqrt(energy / float(P.abs().square().sum()))
    turn = torch.exp(2j * math.pi * torch.rand((K, M, M), generator=gen, device=DEV, dtype=torch.float64))
    turn = torch.where(torch.arange(K, device=DEV)[:, None, None] == 0, torch.ones_like(turn), 0.1 * turn)
    return I, pos, torch.ones(obj, obj, device=DEV, dtype=torch.complex64), (P0 * turn).to(torch.complex64)


def _params(c):
    p = dict(M=c["M"], K=c["K"], N=c["N"], obj_h=c["obj"], obj_w=c["obj"], geometry=c["geometry"],
             blur_domain=c["blur"], fresnel_F=FRESNEL_F if c["geometry"] == "near" else 0.0, sigma1=c["sigma"],
             sigma2=c["sigma"], kernel_size=c["taps"], windows=EVERY_ITERATION if c["constraint"] else [])
    if c["rule"] == "rpie":
        p.update(step_rule="rpie", rpie_alpha_obj=0.2, rpie_alpha_probe=0.5)
    if c["minibatch"]:
        p.update(minibatch=c["minibatch"], order_seed=11)
    if c["engine"] == "dm":
        p.update(engine="dm")
    return p


def _members(c):
    """Sizes of a batch's problems (64 to 256 pixels, uneven position counts, both geometries)."""
    rng = np.random.default_rng(c["mix"])
    out = []
    for _ in range(c["members"]):
        M, K = int(rng.choice([64, 128, 256])), int(rng.choice([1, 2, 4]))
        N = int(rng.integers(c["n_lo"], c["n_hi"] + 1))
        step = math.ceil(0.15 * M)
        obj = M + (math.ceil(math.sqrt(N)) - 1) * step + 2
        far = rng.random() < 0.5
        out.append(_engine_case(None, M, K, N, obj, "raster", step, geometry="far" if far else "near",
                                sigma=float(rng.uniform(0.5, 3.0)), dose=1e5, phase=3.14 if far else 0.5,
                                constraint=False))
    return out


def _spectrum(c):
    a = [1.0 + c["span"] * j / max(c["J"] - 1, 1) for j in range(c["J"])]
    m = 1.0 + 0.4 * c["span"]
    w = [math.exp(-0.5 * ((x - m) / (0.3 * c["span"])) ** 2) for x in a]
    return a, [x / sum(w) for x in w]


def _broadband(c, seed):
    """Patterns with a bright centre and speckle, as counts."""
    gen = _generator(seed)
    r = _radius(c["M"]) / c["M"]
    out = torch.empty(c["N"], c["M"], c["M"], device=DEV)
    for n in range(0, c["N"], 64):
        z = torch.randn((min(64, c["N"] - n), c["M"], c["M"], 2), generator=gen, device=DEV)
        out[n:n + 64] = 200.0 * z.square().sum(-1) * torch.exp(-(r / 0.2) ** 2).float() + 0.5
    return torch.poisson(out, generator=gen)


def _estimate_inputs(c, seed):
    gen = _generator(seed)
    S, N = c["S"], c["N"]
    cols = math.ceil(math.sqrt(N))
    pos = (np.stack(np.divmod(np.arange(N), cols), 1) * c["step"]).astype(np.int32)
    I = 200.0 * torch.rand((N, S, S), generator=gen, device=DEV) * torch.exp(-(_radius(S) / (0.3 * S)) ** 4).float()
    C = c["C"]
    ci, co = [1, C, 2 * C, 4 * C, 12 * C, 6 * C, 2 * C], [C, 2 * C, 4 * C, 8 * C, 4 * C, 2 * C, 2]
    layers = []  # He-scaled weights as a trained network's magnitudes, (Cout, 3, 3, Cin), and biases
    for i, o in zip(ci, co):
        w = torch.randn((o, 3, 3, i), generator=gen, device=DEV) * math.sqrt(2.0 / (9 * i))
        layers.append((w, 0.01 * torch.randn(o, generator=gen, device=DEV)))
    head = torch.randn(8 * C, generator=gen, device=DEV) * math.sqrt(1.0 / (8 * C))
    flat = torch.cat([t.reshape(-1) for wb in layers for t in wb] + [head, torch.full((1,), 1.5, device=DEV)])
    return torch.poisson(I, generator=gen), pos, (cols - 1) * c["step"] + S, layers, head, flat


def _network(c, seed, **kw):
    probe = torch.exp(-(_radius(c["S"]) / (0.3 * c["S"])) ** 8).to(torch.complex64)
    return WarmStart(probe, WarmStartConfig(S=c["S"], C=c["C"], batch=c["batch"], dose=2e4, target_scale=1.0,
                                            lattice=LatticeSpec(peak=1.0), seed=int(seed) % (1 << 31), **kw),
                     stream_ptr=torch.cuda.current_stream().cuda_stream)


def prepare(case, seed):
    c = case
    if c["kind"] == "engine":
        I, pos, O, P = _simulate(c, seed)
        return dict(kind="engine", rec=Reconstruction(_params(c), I, pos), O=O, P=P, monitor=c["monitor"])
    if c["kind"] == "batch":
        sims = [(_params(m), _simulate(m, seed * 1000 + i)) for i, m in enumerate(_members(c))]
        batch = ReconstructionBatch([(p, s[0], s[1]) for p, s in sims])
        return dict(kind="batch", rec=batch, O=[s[2] for _, s in sims], P=[s[3] for _, s in sims])
    if c["kind"] == "mono":
        a, w = _spectrum(c)
        return dict(kind="mono", b=_broadband(c, seed), a=a, w=w, k=c["k"])
    if c["kind"] == "estimate":
        I, pos, obj, _, _, flat = _estimate_inputs(c, seed)
        ws = _network(c, seed)
        ws.net.set_params(flat.cpu().numpy())
        return dict(kind="estimate", ws=ws, I=I, pos=pos, obj=obj)
    ws = _network(c, seed)
    return dict(kind="train", ws=ws, patterns=c["steps"] * c["batch"],
                weights=np.empty(ws.net.param_count(), np.float32))


def run(state):
    s = state
    if s["kind"] == "engine":  # the next iteration of a running reconstruction
        s["rec"].iterate(s["O"], s["P"], 1)
        out = dict(object=s["O"], probe=s["P"])
        if s["monitor"]:
            out["error"] = s["rec"].error()
        return out
    if s["kind"] == "batch":
        s["rec"].iterate(s["O"], s["P"], 1)
        return dict(objects=s["O"], probes=s["P"])
    if s["kind"] == "mono":
        return monochromatise(s["b"], s["a"], s["w"], s["k"])
    if s["kind"] == "estimate":
        O, sigma = s["ws"].estimate(s["I"], s["pos"], s["obj"], s["obj"])
        return dict(object=O, sigma=sigma)
    s["ws"].train(s["patterns"])
    return dict(weights=s["ws"].net.get_params(s["weights"]))


# ----------------------------------------------------------------------------- necessary work


def _engine_work(c):
    M, K, N = c["M"], c["K"], c["N"]
    px, fft = M * M, 5.0 * M * M * math.log2(M * M)
    near, dm = c["geometry"] == "near", c["engine"] == "dm"
    flops = N * K * ((6 if near else 3) if dm else (4 if near else 2)) * fft
    flops += N * px * (K * (38 if dm else 26) + 2 * 2 * c["taps"] * (2 if dm else 1) + 11)
    bytes_ = 4 * N * px + 2 * 8 * (c["obj"] ** 2 + K * px) + 8 * N
    if dm:
        bytes_ += 2 * 8 * N * K * px
    return bytes_, flops


def _conv_flops(S, C):
    layers = [(S, 1, C), (S // 2, C, 2 * C), (S // 4, 2 * C, 4 * C), (S // 8, 4 * C, 8 * C), (S // 4, 12 * C, 4 * C),
              (S // 2, 6 * C, 2 * C), (S // 2, 2 * C, 2)]
    return [2.0 * h * h * 9 * i * o for h, i, o in layers]


def work(case):
    c = case
    if c["kind"] == "engine":
        b, f = _engine_work(c)
    elif c["kind"] == "batch":
        each = [_engine_work(m) for m in _members(c)]
        b, f = sum(x for x, _ in each), sum(x for _, x in each)
    elif c["kind"] == "mono":
        px = c["M"] ** 2
        b, f = 8 * c["N"] * px, c["N"] * px * ((2 * c["k"] + 1) * 8 * c["J"] + 10 * c["k"])
    else:
        weights = sum(x / (2 * h * h) for x, h in zip(_conv_flops(c["S"], c["C"]), [c["S"] // d for d in
                                                                                    (1, 2, 4, 8, 4, 2, 2)]))
        fwd = sum(_conv_flops(c["S"], c["C"]))
        if c["kind"] == "estimate":
            side = (math.ceil(math.sqrt(c["N"])) - 1) * c["step"] + c["S"]
            b, f = 4 * c["N"] * c["S"] ** 2 + 4 * weights + 8 * side * side, c["N"] * fwd
        else:
            n = c["steps"] * c["batch"]
            b = c["steps"] * 4 * 6 * weights + 4 * n * c["S"] ** 2 + 4 * weights
            f = n * (3 * fwd - _conv_flops(c["S"], c["C"])[0])
    return {"bytes": float(b), "flops": float(f)}


# ----------------------------------------------------------------------------- the same in 64 bits


def _philox_order(n, seed, stream, t):
    """The Philox4x32-10 Fisher-Yates order that mini-batches are drawn in (see ptycho.h)."""
    a = list(range(n))
    for i in range(n - 1, 0, -1):
        x, k0, k1 = [i, t, stream, 5], seed & 0xFFFFFFFF, seed >> 32
        for _ in range(10):
            p, q = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
            x = [(q >> 32) ^ x[1] ^ k0, q & 0xFFFFFFFF, (p >> 32) ^ x[3] ^ k1, p & 0xFFFFFFFF]
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        j = (x[0] * (i + 1)) >> 32
        a[i], a[j] = a[j], a[i]
    return a


class _Engine64:
    """One engine iteration in complex128."""

    def __init__(self, c, I, pos, O, P):
        self.c, self.I, self.pos = c, I, torch.from_numpy(pos.astype(np.int64)).to(DEV)
        self.O, self.P = O.to(torch.complex128), P.to(torch.complex128)
        self.eps = 1e-6 * math.sqrt(float(I.sum(dtype=torch.float64)) / I.numel())
        self.g = _taps(c["sigma"], c["taps"] // 2)
        self.H = _fresnel(c["M"])
        self.err = 0.0

    def forward(self, psi):
        if self.c["geometry"] == "far":
            return torch.fft.fftshift(torch.fft.fft2(psi), dim=(-2, -1))
        return torch.fft.ifft2(torch.fft.fft2(psi) * self.H)

    def backward(self, psi):
        if self.c["geometry"] == "far":
            return torch.fft.ifft2(torch.fft.ifftshift(psi, dim=(-2, -1)))
        return torch.fft.ifft2(torch.fft.fft2(psi) * self.H.conj())

    def ratio(self, psi, I):
        """Modulus ratio and model intensity of detector waves (n, K, M, M)."""
        S = psi.abs().square().sum(1)
        if self.c["blur"] == "amplitude":
            A = _blur(S.sqrt(), self.g)
            return I.sqrt() / (A + self.eps), A * A
        A = _blur(S, self.g)
        return I.sqrt() / (A + self.eps ** 2).sqrt(), A

    def at(self, idx):
        i = torch.arange(self.c["M"], device=DEV)
        p = self.pos[idx]
        return (p[:, 0, None, None] + i[:, None]) * self.c["obj"] + p[:, 1, None, None] + i[None]

    def step(self, num, den, kind):
        c_den, c_max = (1.0, 1e-3)
        if self.c["rule"] == "rpie":
            a = 0.2 if kind == "object" else 0.5
            c_den, c_max = 1 - a, a
        return torch.where(den > 0, num / (c_den * den + c_max * den.max()).clamp_min(1e-300), 0)

    def sweep(self, idx, per=64):
        """Simultaneous step over the positions idx (the pc-DM one with a fresh exit-wave state)."""
        c, O, P = self.c, self.O, self.P
        M, K, dm = c["M"], c["K"], c["engine"] == "dm"
        per = max(1, per * 4 * 128 * 128 // (K * M * M))
        NO, DO = torch.zeros_like(O).reshape(-1), torch.zeros(O.numel(), device=DEV, dtype=torch.float64)
        NP, DP = torch.zeros_like(P), torch.zeros((M, M), device=DEV, dtype=torch.float64)
        P2, states = P.abs().square().sum(0), []
        for a in range(0, len(idx), per):
            at, I = self.at(idx[a:a + per]), self.I[idx[a:a + per]].double()
            o = O.reshape(-1)[at]
            psi = P * o[:, None]
            wave = self.forward(psi)  # with a fresh state pc-DM's reflected wave is the estimate itself
            R, Ihat = self.ratio(wave, I)
            self.err += float((Ihat - I).square().sum())
            d = self.backward(R[:, None] * wave) - psi
            NO.index_add_(0, at.reshape(-1), (P.conj() * d).sum(1).reshape(-1))
            DO.index_add_(0, at.reshape(-1), P2.expand(len(at), M, M).reshape(-1))
            if dm:
                states.append(psi + d)
            else:
                NP += (o.conj()[:, None] * d).sum(0)
                DP += o.abs().square().sum(0)
        self.O = O + self.step(NO, DO, "object").reshape(O.shape)
        if dm:
            for a, st in zip(range(0, len(idx), per), states):
                o = self.O.reshape(-1)[self.at(idx[a:a + per])]
                NP += (o.conj()[:, None] * (st - P * o[:, None])).sum(0)
                DP += o.abs().square().sum(0)
        self.P = P + self.step(NP, DP, "probe")

    def constrain(self):
        a, phi = self.O.abs().clamp_min(1e-6), self.O.angle()
        ln = a.log()
        at = [self.at(slice(n, n + 256)) for n in range(0, len(self.pos), 256)]
        num, den = (torch.cat([x.abs().reshape(-1)[i].sum((1, 2)) for i in at]) for x in (ln, phi))
        cb = (num / den.clamp_min(1e-30)).clamp(0.01, 10.0)
        tot, cnt = torch.zeros_like(ln).reshape(-1), torch.zeros_like(ln).reshape(-1)
        for n, i in zip(range(0, len(self.pos), 256), at):
            tot.index_add_(0, i.reshape(-1), cb[n:n + 256, None, None].expand(i.shape).reshape(-1))
            cnt.index_add_(0, i.reshape(-1), torch.ones(i.numel(), device=DEV, dtype=torch.float64))
        C = (tot / cnt.clamp_min(1.0)).reshape(ln.shape)
        self.O = torch.where(cnt.reshape(ln.shape) > 0, torch.exp(C * phi + 1j * phi), self.O)

    def iteration(self):
        c = self.c
        parts = [list(range(c["N"]))]
        if 0 < c["minibatch"] < c["N"]:
            order = _philox_order(c["N"], 11, 3, 0)
            parts = [order[i:i + c["minibatch"]] for i in range(0, c["N"], c["minibatch"])]
            parts = [parts[i] for i in _philox_order(len(parts), 11, 4, 1)]
        for idx in parts:
            self.sweep(torch.tensor(idx, device=DEV))
        if c["constraint"]:
            self.constrain()
        E = math.sqrt(self.err / sum(float(self.I[a:a + 64].double().square().sum()) for a in range(0, c["N"], 64)))
        return self.O, self.P, E


def _cgls64(b, a, w, k):
    """k CGLS steps of min ||C x - b|| per pattern, C the spectrum's linear interpolation."""
    M = b.shape[-1]
    i = torch.arange(M, device=DEV, dtype=torch.float64)
    S = []
    for s in a:
        t = M / 2 + (i - M / 2) / s
        i0 = t.floor().long()
        f = t - i0
        m = torch.zeros(M + 2, M, device=DEV, dtype=torch.float64)  # [source + 1, output]
        inside = (i0 >= -1) & (i0 <= M - 1)
        col = torch.arange(M, device=DEV)
        m[i0.clamp(-1, M - 1) + 1, col] += torch.where(inside, 1 - f, 0.0)
        m[i0.clamp(-1, M - 1) + 2, col] += torch.where(inside, f, 0.0)
        S.append(m[1:-1].T.contiguous())
    def taps(m):  # a banded matrix as gathers: for each row, up to `width` source indices and weights
        width = int((m != 0).sum(1).max())
        wt, ix = m.abs().topk(max(width, 1), dim=1)
        return [(ix[:, q].contiguous(), wt[:, q].contiguous()) for q in range(max(width, 1))]
    fwd, adj = [taps(m) for m in S], [taps(m.T.contiguous()) for m in S]
    def apply(x, ops):
        out = torch.zeros_like(x)
        for op, s, wt in zip(ops, a, w):
            y = sum(x[:, :, ix] * g for ix, g in op)
            out += wt / (s * s) * sum(y[:, ix, :] * g[:, None] for ix, g in op)
        return out
    x, r = torch.zeros_like(b), b.clone()
    s = apply(r, adj)
    p, gamma = s.clone(), s.square().sum((1, 2), keepdim=True)
    for _ in range(k):
        q = apply(p, fwd)
        alpha = gamma / q.square().sum((1, 2), keepdim=True).clamp_min(1e-300)
        x += alpha * p
        r -= alpha * q
        s = apply(r, adj)
        new = s.square().sum((1, 2), keepdim=True)
        p = s + new / gamma.clamp_min(1e-300) * p
        gamma = new
    return x


def _estimate64(c, seed):
    I, pos, obj, layers, head, _ = _estimate_inputs(c, seed)
    f = torch.nn.functional
    conv = lambda x, n: f.conv2d(x, layers[n][0].double().permute(0, 3, 1, 2), layers[n][1].double(), padding=1)  # noqa: E731
    up = lambda x: x.repeat_interleave(2, -1).repeat_interleave(2, -2)  # noqa: E731
    S, N = c["S"], c["N"]
    Q = S // 2
    win = torch.sin(math.pi * (torch.arange(Q, device=DEV, dtype=torch.float64) + 0.5) / Q).square()
    win = win[:, None] * win[None]
    num = torch.zeros(obj, obj, device=DEV, dtype=torch.complex128)
    den = torch.zeros(obj, obj, device=DEV, dtype=torch.float64)
    sig = []
    for a in range(0, N, 16):
        x = torch.log1p(I[a:a + 16].double())[:, None] / 4
        a0 = conv(x, 0).relu()
        a1 = conv(f.avg_pool2d(a0, 2), 1).relu()
        a2 = conv(f.avg_pool2d(a1, 2), 2).relu()
        a3 = conv(f.avg_pool2d(a2, 2), 3).relu()
        a4 = conv(torch.cat([up(a3), a2], 1), 4).relu()
        a5 = conv(torch.cat([up(a4), a1], 1), 5).relu()
        out = conv(a5, 6)
        sig += (a3.mean((2, 3)) @ head.double() + 1.5).tolist()
        for n in range(len(out)):
            y, x0 = (int(v) + S // 4 for v in pos[a + n])
            num[y:y + Q, x0:x0 + Q] += win * torch.exp(torch.complex(out[n, 0], out[n, 1]))
            den[y:y + Q, x0:x0 + Q] += win
    O = torch.where(den > 0, num / den.clamp_min(1e-300), torch.ones_like(num))
    return dict(object=O, sigma=float(np.median(sig)))


def exact(case, seed):
    c = case
    if c["kind"] == "engine":
        O, P, E = _Engine64(c, *_simulate(c, seed)).iteration()
        return dict(object=O, probe=P, error=E) if c["monitor"] else dict(object=O, probe=P)
    if c["kind"] == "batch":
        got = [_Engine64(m, *_simulate(m, seed * 1000 + i)).iteration() for i, m in enumerate(_members(c))]
        return dict(objects=[g[0] for g in got], probes=[g[1] for g in got])
    if c["kind"] == "mono":
        a, w = _spectrum(c)
        b = _broadband(c, seed).double()
        return torch.cat([_cgls64(b[n:n + 128], a, w, c["k"]) for n in range(0, c["N"], 128)])
    if c["kind"] == "estimate":
        return _estimate64(c, seed)
    return None  # training draws its patterns with the framework's own counter-based generator
