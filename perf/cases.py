"""The framework's work, as a user's program calls it: the cases that its speed is judged by.

Every case goes through the package's public entry points (`Plan` and its
methods, `prop_apply`, `prop_reconstruct_batch`) on complex64 data, the only
type they take.  Sizes are those of the repository's workloads (`synth`), its
tests and its benchmark, or lie between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_13177_gb300 import Plan, ProjParams, ReconParams, prop_apply, prop_reconstruct_batch

DEV = "cuda"
GOLDEN = math.pi * (math.sqrt(5.0) - 1.0) / 2.0
SIZES = [16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512]  # image sizes N the plans take

# Adam's epsilon of the cases that run Adam.  The data gradients are of order
# 1 to 100, so this is a small fraction of most of them, but it makes a step a
# smooth function of the gradient: at 1e-8 the first step is the gradient's
# sign, and a component that rounding moves across zero jumps by 2 lr.
ADAM_EPS = 1e-1


def _case(name, kind, N, Nf, B, L, R, T=1, width=0, chunk=0, iters=0, **more):
    return dict(name=name, kind=kind, N=N, Nf=Nf, B=B, L=L, R=R, T=T, width=width, chunk=chunk, iters=iters, **more)


def listed():
    return [
        # One forward pass of the smallest test problem: a call inside a
        # user's own loop, where launches and latency are all of it.
        _case("forward_tiny", "forward", 32, 8, 5, 8, 32),
        # Loss and gradient of the small reference problem for an optimiser
        # of the caller's; the default (width 6) operator.
        _case("grad_small64", "grad", 64, 8, 8, 16, 64),
        # The same for odd counts of bins, blades, lines and samples, several
        # frames and a grid length with a factor 3.
        _case("grad_odd", "grad", 96, 5, 7, 11, 97, T=3, width=8),
        # The two directions of the operator at the benchmark's static
        # configuration, kernel width 8: simulation, and gridding of a scan.
        _case("forward_static", "forward", 256, 32, 16, 24, 256, width=8),
        _case("adjoint_static", "adjoint", 256, 32, 16, 24, 256, width=8),
        # The benchmark's reconstruction of a static scan, and its render.
        _case("recon_static", "recon", 256, 32, 16, 24, 256, width=8, iters=10),
        # The dynamic configuration: 32 frames of two golden-angle blades each
        # with TV in time.
        _case("recon_dynamic", "recon", 192, 16, 64, 16, 192, T=32, width=8, iters=4),
        # The operator inside a differentiable program, forward and backward,
        # at the largest configuration (the default width).
        _case("autograd_diff", "autograd", 384, 64, 32, 32, 384),
        # Loss and gradient at the largest image, in 16-bin chunks (the option
        # that holds the workspace down), the last chunk ragged.
        _case("grad_chunked", "grad", 512, 24, 12, 32, 512, chunk=16),
        # Requests of different blade counts and frames advanced together, as
        # the request server batches them.
        _case("batch_mixed", "batch", 192, 16, 8, 24, 192, T=1, iters=4, B2=16, T2=1, B3=24, T3=4, B4=32, T4=16),
        # One pass over the blades with the paper's own forward model.
        _case("proj_static", "proj", 256, 32, 16, 24, 256, iters=16),
        # One training step of the K-Planes model with the caller's own
        # optimiser: render, loss and volume gradient, parameter gradients.
        _case("kplanes_dynamic", "kplanes", 192, 16, 64, 16, 192, T=32, width=8, F=8, S=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["forward", "adjoint", "autograd", "grad", "recon", "recon", "batch", "proj", "kplanes"])
        N = rng.choice(SIZES)
        # bins: the strides with kernels of their own, and anything between
        Nf = rng.choice([8, 16, 32, 64]) if rng.random() < 0.5 else _log_int(rng, 1, 64)
        T = 1 if rng.random() < 0.5 else _log_int(rng, 2, 32)
        B = max(T, _log_int(rng, 4, 64))
        L = max(1, N // 8 + rng.randint(-3, 3)) if rng.random() < 0.5 else _log_int(rng, 4, 32)
        R = N if rng.random() < 0.6 else max(8, N + rng.randint(-N // 4, N // 8))
        width = rng.choice([0, 8])
        chunk = rng.choice([8, 16, 32]) if kind in ("forward", "adjoint", "autograd", "grad") and rng.random() < 0.2 else 0
        iters = {"recon": rng.randint(2, 10), "batch": rng.randint(2, 6), "proj": rng.randint(2, 24)}.get(kind, 0)
        c = dict(kind=kind, N=N, Nf=Nf, B=B, L=L, R=R, T=T, width=width, chunk=chunk, iters=iters)
        if kind == "batch":
            c |= dict(B2=_log_int(rng, 4, 32), T2=1, B3=_log_int(rng, 4, 32), T3=rng.randint(1, 4),
                      B4=_log_int(rng, 8, 32), T4=rng.randint(1, 8))
        if kind == "kplanes":
            c |= dict(F=rng.choice([2, 4, 8, 16]), S=rng.choice([1, 2]))
        if kind == "proj" and T * B > 512:
            continue
        samples = sum(g["B"] for g in _members(c)) * L * R
        if samples <= 400_000 and _cost(c) <= top:
            return c


# --- sizes ---------------------------------------------------------------------


def _members(c):
    """The geometries of a case: one, or those of a batch."""
    got = [dict(c, B=c["B"], T=c["T"])]
    if c["kind"] == "batch":
        got += [dict(c, B=max(c["B%d" % i], c["T%d" % i]), T=c["T%d" % i]) for i in (2, 3, 4)]
    return got


def _kp_params(c):
    N, Nf, T, F = c["N"], c["Nf"], c["T"], c["F"]
    n = 0
    for s in range(c["S"]):
        m = N >> s
        n += (m * m + 2 * Nf * m + 2 * T * m + T * Nf + 1) * F
    return n


def work(c):
    """Bytes of one pass: its inputs read and its outputs written once (the
    state of each Adam step read and written once a step); flops: the
    transforms on the 2N grid (5 n log2 n each), the taps, the updates."""
    by = fl = 0.0
    for g in _members(c):
        N, Nf, T = g["N"], g["Nf"], g["T"]
        W = g["width"] or 6
        vol, y = 8.0 * T * N * N * Nf, 8.0 * g["B"] * g["L"] * g["R"]
        n = 2 * N
        fft = Nf * T * (n + N) * 5.0 * n * math.log2(n)           # zero rows skipped
        taps = y / 8 * Nf * (W * W * 4.0 + 8)
        one = fft + taps                                          # one direction of the operator
        vox = vol / 8
        k = g["kind"]
        if k in ("forward", "adjoint"):
            by, fl = by + vol + y, fl + one
        elif k == "autograd":
            by, fl = by + 2 * vol + 2 * y, fl + 2 * one
        elif k == "grad":
            by, fl = by + 2 * vol + y, fl + 2 * one + 60 * vox
        elif k in ("recon", "batch"):
            by, fl = by + g["iters"] * (6 * vol + y), fl + g["iters"] * (2 * one + 100 * vox)
        elif k == "proj":
            img = 8.0 * N * N
            by += g["iters"] * (6 * vol + img)
            fl += g["iters"] * (16 * vox / T + 2 * 10.0 * N * N * math.log2(N) + 130 * vox)
        else:
            p = 8.0 * _kp_params(g)
            by += 3 * p + 3 * vol + y
            fl += 2 * one + 60 * vox + vox * g["F"] * g["S"] * (16 + 3 * 16)
    return {"bytes": by, "flops": fl}


def _cost(c):
    w = work(c)
    # the oversampled grid and the volume's own buffers bound what a state holds
    return max(w["bytes"], w["flops"] / 50)


# --- inputs ----------------------------------------------------------------------


def _geometry(c):
    b = np.arange(c["B"], dtype=np.float64)
    theta = math.pi * b / c["B"] if c["T"] == 1 else np.mod(b * GOLDEN, math.pi)
    delta = np.linspace(-4.0, 4.0, c["Nf"]) if c["Nf"] > 1 else np.array([1.7])
    frames = (np.arange(c["B"]) * c["T"] // c["B"]).astype(np.int32)
    return theta, delta, frames


def _plan(c):
    theta, delta, frames = _geometry(c)
    return Plan(c["N"], c["L"], c["R"], theta, delta, frames, c["T"], c["chunk"], None, c["width"])


def _blobs(gen, N, count=12):
    """Centres, widths and complex amplitudes of a smooth object of a few parts."""
    u = torch.rand(count, 5, generator=gen, dtype=torch.float64).to(DEV)
    ctr = (u[:, :2] - 0.5) * 0.7 * N
    sig = N * (0.03 + 0.1 * u[:, 2])
    amp = (0.2 + 0.8 * u[:, 3]) * torch.exp(2j * math.pi * u[:, 4])
    return ctr, sig, amp


def _kspace(c):
    """k of every sample: two [B, L, R] arrays of doubles, cycles a pixel."""
    theta, _, _ = _geometry(c)
    th = torch.tensor(theta, device=DEV)[:, None, None]
    kr = ((torch.arange(c["R"], device=DEV, dtype=torch.float64) - c["R"] / 2) / c["N"])[None, None, :]
    kp = ((torch.arange(c["L"], device=DEV, dtype=torch.float64) - c["L"] / 2) / c["N"])[None, :, None]
    return kr * torch.cos(th) - kp * torch.sin(th), kr * torch.sin(th) + kp * torch.cos(th)


def _noise(gen, shape, scale):
    g = torch.Generator(device=DEV).manual_seed(int(torch.randint(1 << 40, (1,), generator=gen)))
    return scale * torch.randn(*shape, generator=g, device=DEV, dtype=torch.complex64)


def _blob_spectrum(kx, ky, blobs, N):
    out = torch.zeros(kx.shape, dtype=torch.complex128, device=DEV)
    for (cx, cy), s, a in zip(*blobs):
        out += a * (2 * math.pi * s * s) * torch.exp(-2 * math.pi ** 2 * s * s * (kx * kx + ky * ky)) \
            * torch.exp(-2j * math.pi * (kx * cx + ky * cy))
    return (out / N).to(torch.complex64)


def _data(c, gen):
    """Measured blades: the spectrum of a few smooth parts, and noise."""
    kx, ky = _kspace(c)
    return (_blob_spectrum(kx, ky, _blobs(gen, c["N"]), c["N"]) + _noise(gen, kx.shape, 1e-2)).contiguous()


def _volume(c, gen):
    """A volume in mid-reconstruction: a smooth object spread over the bins, and noise."""
    N = c["N"]
    x = torch.arange(N, device=DEV, dtype=torch.float32) - N / 2
    img = torch.zeros(N, N, dtype=torch.complex64, device=DEV)
    for (cx, cy), s, a in zip(*_blobs(gen, N)):
        img += a.to(torch.complex64) * torch.exp(-((x[None, :] - cx) ** 2 + (x[:, None] - cy) ** 2) / (2 * s * s)).float()
    spec = torch.rand(c["T"], 1, 1, c["Nf"], generator=gen).to(DEV)
    return (img[None, :, :, None] * spec + _noise(gen, (c["T"], N, N, c["Nf"]), 0.02)).contiguous()


def _recon_params(c):
    return ReconParams(iters=c["iters"], lr=1e-2, eps=ADAM_EPS, tv_xy=1e-3, tv_t=1e-2 if c["T"] > 1 else 0.0)


def _proj_params(c):
    return ProjParams(iters=c["iters"], lr=1e-2, eps=ADAM_EPS, tv_xy=1e-3, tv_f=1e-3,
                      tv_t=1e-2 if c["T"] > 1 else 0.0, l1=1e-4)


def _inputs(c, seed):
    """The tensors of a case, from its seed alone."""
    gen = torch.Generator().manual_seed(int(seed))
    s = {}
    if c["kind"] == "batch":
        s["ys"] = [_data(g, gen) for g in _members(c)]
    elif c["kind"] == "proj":
        k = (torch.arange(c["N"], device=DEV, dtype=torch.float64) - c["N"] / 2) / c["N"]
        ky, kx = torch.meshgrid(k, k, indexing="ij")
        y = _blob_spectrum(kx, ky, _blobs(gen, c["N"]), c["N"])
        s["y"] = (y[None] + _noise(gen, (c["B"], c["N"], c["N"]), 1e-2)).contiguous()
    elif c["kind"] != "forward":
        s["y"] = _data(c, gen)
    if c["kind"] in ("forward", "autograd", "grad"):
        s["V"] = _volume(c, gen)
    if c["kind"] == "kplanes":
        # products of six planes of order 1: features around 0.5 with random phases
        s["kp"] = (0.5 * torch.exp(_noise(gen, (_kp_params(c),), 0.5))).contiguous()
    return s


def prepare(c, seed):
    s = _inputs(c, seed)
    s["case"] = c
    if c["kind"] == "batch":
        s["plans"] = [_plan(g) for g in _members(c)]
    else:
        s["plan"] = _plan(c)
    if c["kind"] == "autograd":
        s["V"].requires_grad_(True)
    return s


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "forward":
        return s["plan"].forward(s["V"])
    if k == "adjoint":
        return s["plan"].adjoint(s["y"])
    if k == "autograd":
        V = s["V"]
        V.grad = None
        r = prop_apply(V, s["plan"]) - s["y"]
        loss = (r.real.square() + r.imag.square()).sum()
        loss.backward()
        return {"residual": r.detach(), "grad": V.grad}
    if k == "grad":
        loss, grad = s["plan"].loss_grad(s["y"], _recon_params(c), s["V"])
        return {"loss": loss, "grad": grad}
    if k == "recon":
        V, trace = s["plan"].reconstruct(s["y"], _recon_params(c))
        return {"V": V, "trace": [float(v) for v in trace], "image": s["plan"].render(V)}
    if k == "batch":
        Vs, _ = prop_reconstruct_batch(s["plans"], s["ys"], [_recon_params(g) for g in _members(c)], trace=False)
        return {"V": Vs}
    if k == "proj":
        V, trace = s["plan"].proj_reconstruct(s["y"], _proj_params(c))
        return {"V": V, "trace": [float(v) for v in trace]}
    V = s["plan"].kplanes_render(s["kp"], c["F"], c["S"])
    loss, gV = s["plan"].loss_grad(s["y"], _recon_params(c), V)
    return {"V": V, "loss": loss, "gV": gV, "grad": s["plan"].kplanes_vjp(s["kp"], gV, c["F"], c["S"])}


# --- the same in 64 bits ------------------------------------------------------------


class _Exact:
    """The non-uniform transform of one geometry as it is defined, in 64 bits."""

    def __init__(self, c):
        self.c = c
        _, delta, frames = _geometry(c)
        self.frames = frames
        kx, ky = _kspace(c)                                     # [B, L, R]
        x = torch.arange(c["N"], device=DEV, dtype=torch.float64) - c["N"] / 2
        self.kx, self.ky, self.x = kx, ky, x
        kr = (torch.arange(c["R"], device=DEV, dtype=torch.float64) - c["R"] / 2) / c["N"]
        self.P = torch.exp(-2j * math.pi * kr[:, None] * torch.tensor(delta, device=DEV)[None, :])  # [R, Nf]

    def _frame(self, t):
        b = np.nonzero(self.frames == t)[0]
        if not len(b):
            return None, None, None
        b = torch.tensor(b, device=DEV)
        E = []
        for k in (self.kx, self.ky):
            q = k[b].permute(2, 0, 1).reshape(self.c["R"], -1, 1)  # [R, B L, 1]
            E.append(torch.exp(-2j * math.pi * q * self.x))
        return b, E[0], E[1]

    def forward(self, V):
        c = self.c
        y = torch.zeros(c["B"], c["L"], c["R"], dtype=torch.complex128, device=DEV)
        for t in range(c["T"]):
            b, E1, E2 = self._frame(t)
            if b is None:
                continue
            img = (self.P @ V[t].reshape(-1, c["Nf"]).T).reshape(c["R"], c["N"], c["N"])  # [R, x2, x1]
            v = (torch.bmm(E1, img.transpose(1, 2)) * E2).sum(2)                         # [R, B L]
            y[b] = v.reshape(c["R"], len(b), c["L"]).permute(1, 2, 0)
        return y / c["N"]

    def adjoint(self, r):
        c = self.c
        V = torch.zeros(c["T"], c["N"], c["N"], c["Nf"], dtype=torch.complex128, device=DEV)
        for t in range(c["T"]):
            b, E1, E2 = self._frame(t)
            if b is None:
                continue
            q = r[b].permute(2, 0, 1).reshape(c["R"], -1, 1)
            img = torch.bmm((E2.conj() * q).transpose(1, 2), E1.conj())                  # [R, x2, x1]
            V[t] = (img.reshape(c["R"], -1).T @ self.P.conj()).reshape(c["N"], c["N"], c["Nf"])
        return V / c["N"]

    def loss_grad(self, V, y, tv_xy, tv_t, tv_eps):
        r = self.forward(V) - y
        g = 2 * self.adjoint(r)
        v = V.detach().requires_grad_(True)
        with torch.enable_grad():
            reg = _tv(v, tv_xy, 0.0, tv_t, tv_eps)
        (h,) = torch.autograd.grad(reg, v)
        return float((r.abs() ** 2).sum() + reg.detach()), g + h


def _tv(V, xy, f, t, eps):
    total = torch.zeros((), dtype=torch.float64, device=DEV)
    for axis, w in ((1, xy), (2, xy), (3, f), (0, t)):
        if w and V.shape[axis] > 1:
            d = torch.diff(V, dim=axis)
            total = total + w * torch.sqrt(d.real ** 2 + d.imag ** 2 + eps * eps).sum()
    return total


def _f32(v):
    return float(np.float32(v))


class _Adam:
    def __init__(self, p, shape):
        self.lr, self.b1, self.b2, self.eps = (_f32(v) for v in (p.lr, p.beta1, p.beta2, p.eps))
        self.m = torch.zeros(*shape, 2, dtype=torch.float64, device=DEV)
        self.v = torch.zeros_like(self.m)
        self.k = 0

    def step(self, V, g):
        self.k += 1
        g = torch.view_as_real(g)
        self.m = self.b1 * self.m + (1 - self.b1) * g
        self.v = self.b2 * self.v + (1 - self.b2) * g * g
        up = (self.m / (1 - self.b1 ** self.k)) / (torch.sqrt(self.v / (1 - self.b2 ** self.k)) + self.eps)
        return V - self.lr * torch.view_as_complex(up.contiguous())


def _exact_recon(g, y):
    p = _recon_params(g)
    op = _Exact(g)
    V = torch.zeros(g["T"], g["N"], g["N"], g["Nf"], dtype=torch.complex128, device=DEV)
    adam, trace = _Adam(p, V.shape), []
    for _ in range(p.iters):
        loss, grad = op.loss_grad(V, y.to(torch.complex128), _f32(p.tv_xy), _f32(p.tv_t), _f32(p.tv_eps))
        trace.append(loss)
        V = adam.step(V, grad)
    return V, trace


def _fft(z):
    return torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(z), norm="ortho"))


def _exact_proj(c, y):
    """The projection at the blade's tilt, the centred DFT under its mask, the gradient by autograd."""
    p = _proj_params(c)
    theta, delta, frames = _geometry(c)
    N, Nf = c["N"], c["Nf"]
    V = torch.zeros(c["T"], N, N, Nf, dtype=torch.complex128, device=DEV)
    adam, trace = _Adam(p, V.shape), []
    wk, wi, l1, eps = (_f32(v) for v in (p.w_kspace, p.w_image, p.l1, p.tv_eps))
    u = torch.arange(N, device=DEV, dtype=torch.float64) - N / 2
    pad = int(np.max(np.abs(delta))) + 3
    for k in range(p.iters):
        b = k % c["B"]
        cs, sn = math.cos(theta[b]), math.sin(theta[b])

        def snap(a):
            h = torch.round(2 * a) / 2
            return torch.where((a - h).abs() < 1e-9, h, a)

        rho, q = snap(u[None, :] * cs + u[:, None] * sn), snap(-u[None, :] * sn + u[:, None] * cs)
        R, L = c["R"], c["L"]
        M = (rho >= -R / 2 - 0.5) & (rho < R / 2 - 0.5) & (q >= -L / 2 - 0.5) & (q < L / 2 - 0.5)
        v = V.detach().requires_grad_(True)
        with torch.enable_grad():
            vp = torch.nn.functional.pad(torch.view_as_real(v[frames[b]]), (0, 0, 0, 0, pad, pad, pad, pad))
            vp = torch.view_as_complex(vp)
            img = torch.zeros(N, N, dtype=torch.complex128, device=DEV)
            for f in range(Nf):
                s1, s2 = delta[f] * cs, delta[f] * sn
                o1, o2 = math.floor(-s1), math.floor(-s2)
                w1, w2 = -s1 - o1, -s2 - o2
                for d2, c2 in ((0, 1 - w2), (1, w2)):
                    for d1, c1 in ((0, 1 - w1), (1, w1)):
                        r0, c0 = pad + o2 + d2, pad + o1 + d1
                        img = img + (c1 * c2) * vp[r0:r0 + N, c0:c0 + N, f]
            r = torch.where(M, _fft(img) - y[b].to(torch.complex128), 0)
            # the image term, of U^H M Z against U^H M y, through the unitary DFT
            loss = (wk + wi) * (r.real ** 2 + r.imag ** 2).sum()
            loss = loss + _tv(v, _f32(p.tv_xy), _f32(p.tv_f), _f32(p.tv_t), eps)
            loss = loss + l1 * torch.sqrt(v.real ** 2 + v.imag ** 2 + eps * eps).sum()
        (g,) = torch.autograd.grad(loss, v)
        trace.append(float(loss.detach()))
        V = adam.step(V, g)
    return V, trace


def _kp_axis(count, nodes):
    """[count, nodes] interpolation weights: voxel i at (i + 1/2) nodes / count - 1/2, clamped."""
    i = np.arange(count, dtype=np.float64)
    p = i if nodes == count else (i + 0.5) * nodes / count - 0.5
    p = np.clip(p, 0, nodes - 1)
    lo = np.minimum(np.floor(p).astype(int), max(nodes - 2, 0))
    W = np.zeros((count, nodes))
    W[np.arange(count), lo] += 1 - (p - lo)
    W[np.arange(count), np.minimum(lo + 1, nodes - 1)] += p - lo
    return torch.tensor(W, dtype=torch.complex128, device=DEV)


def _kp_expanded(c, kp):
    """Per scale the planes at the volume's resolution and a; functions of the flat parameters."""
    N, Nf, T, F = c["N"], c["Nf"], c["T"], c["F"]
    got, at = [], 0
    for s in range(c["S"]):
        m = N >> s
        X = _kp_axis(N, m)

        def take(*shape):
            nonlocal at
            v = kp[at:at + math.prod(shape)].reshape(shape)
            at += math.prod(shape)
            return v

        xy = torch.einsum("ya,xb,abk->yxk", X, X, take(m, m, F))
        xw, xt, yw, yt = (torch.einsum("xb,abk->axk", X, take(rows, m, F)) for rows in (Nf, T, Nf, T))
        got.append((xy, xw, xt, yw, yt, take(T, Nf, F), take(F)))
    return got


def _kp_frame(planes, t):
    """Frame t of the model: [y, x, w]."""
    out = 0
    for xy, xw, xt, yw, yt, wt, a in planes:
        for k in range(a.shape[0]):
            m = xy[:, :, k] * xt[t, None, :, k] * yt[t, :, None, k] * a[k]
            out = out + m[:, :, None] * xw[:, :, k].T[None] * (yw[:, :, k].T * wt[t, None, :, k])[:, None, :]
    return out


def _exact_kplanes(c, s):
    kp = s["kp"].to(torch.complex128)
    with torch.no_grad():
        planes = _kp_expanded(c, kp)
        V = torch.stack([_kp_frame(planes, t) for t in range(c["T"])])
    p = _recon_params(c)
    loss, gV = _Exact(c).loss_grad(V, s["y"].to(torch.complex128), _f32(p.tv_xy), _f32(p.tv_t), _f32(p.tv_eps))
    leaf = kp.clone().requires_grad_(True)
    planes = [tuple(v.detach().requires_grad_(True) for v in sc) for sc in _kp_expanded(c, leaf)]
    flat = [v for sc in planes for v in sc]
    total = [torch.zeros_like(v) for v in flat]
    for t in range(c["T"]):  # the frames one after the other: a graph of one frame at a time
        out = _kp_frame(planes, t)
        for a, g in zip(total, torch.autograd.grad(out, flat, gV[t])):
            a += g
    again = [v for sc in _kp_expanded(c, leaf) for v in sc]
    (grad,) = torch.autograd.grad(again, leaf, total)
    return {"V": V, "loss": loss, "gV": gV, "grad": grad}


@torch.no_grad()
def exact(c, seed):
    s = _inputs(c, seed)
    k = c["kind"]
    wide = {n: v.to(torch.complex128) for n, v in s.items() if isinstance(v, torch.Tensor)}
    if k == "forward":
        return _Exact(c).forward(wide["V"])
    if k == "adjoint":
        return _Exact(c).adjoint(wide["y"])
    if k == "autograd":
        op = _Exact(c)
        r = op.forward(wide["V"]) - wide["y"]
        return {"residual": r, "grad": 2 * op.adjoint(r)}
    if k == "grad":
        p = _recon_params(c)
        loss, grad = _Exact(c).loss_grad(wide["V"], wide["y"], _f32(p.tv_xy), _f32(p.tv_t), _f32(p.tv_eps))
        return {"loss": loss, "grad": grad}
    if k == "recon":
        V, trace = _exact_recon(c, wide["y"])
        return {"V": V, "trace": trace, "image": V.sum(3)}
    if k == "batch":
        return {"V": [_exact_recon(g, y)[0] for g, y in zip(_members(c), s["ys"])]}
    if k == "proj":
        V, trace = _exact_proj(c, s["y"])
        return {"V": V, "trace": trace}
    with torch.enable_grad():
        return _exact_kplanes(c, s)
