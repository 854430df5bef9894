"""Timing cases of the NLINV library: what a program that uses it has it do, through the public Python entry points.

The sizes are those of the repository's workloads (64 x 64 grid with 4 coils, 256 x 256 with 8, 384 x 384 with 10,
512 x 512 with 16, and the 64-frame batch of uneven grid sides and coil counts), plus ragged ones in between.

* Operator cases apply F, DF, DF^H or the normal operator once, as a solver outside the library does, or F together
  with its gradient, as a training program does.
* Frame cases are whole Gauss-Newton reconstructions (one CUDA graph per frame after the first), alone or batched.
* The gradient case differentiates through a whole reconstruction.
* The gridding case turns one frame's radial samples into gridded data.

Inputs are drawn on the GPU from the seed: an ellipse phantom, smooth coils, radial spokes, 30 dB noise.  ``exact``
restates the method (unitary FFTs, Sobolev weight, conjugate gradients, Gauss-Newton) in complex128 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1301_1215_gb300 import autograd, synth
from paper_1301_1215_gb300.nlinv import Gridder, Nlinv, NlinvBatch

SIDES = (16, 32, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512)
SOBOLEV_A, SOBOLEV_L = 220.0, 32.0
OPS = ("forward", "grad", "derivative", "adjoint", "normal")


def _op(name, kind, n, coils, spokes, fov=None):
    return {"name": name, "kind": kind, "n": n, "coils": coils, "spokes": spokes, "fov": n // 4 if fov is None else fov}


def listed():
    return [
        # F on the small single-frame problem: the smallest call, three launches long
        _op("forward_64x4", "forward", 64, 4, 16),
        # F and the gradient of |F(x) - y|^2, the 256 x 256 differentiation workload
        _op("grad_256x8", "grad", 256, 8, 25),
        # DF on a field of view that is not n/4, odd, with ragged column strips: zoomed acquisitions
        _op("derivative_320x7_fov75", "derivative", 320, 7, 21, 75),
        # DF^H with a coil count that divides nothing: the gradient of an external solver
        _op("adjoint_192x13", "adjoint", 192, 13, 17),
        # the normal operator of the real-time series, what conjugate gradients apply
        _op("normal_384x10", "normal", 384, 10, 13),
        # the same on the largest grid
        _op("normal_512x16", "normal", 512, 16, 32),
        # gridding of one real-time frame's radial samples
        {"name": "grid_384x10", "kind": "grid", "n": 384, "coils": 10, "spokes": 13},
        # the small single frame, start to end: launch-bound
        {"name": "frame_64x4", "kind": "frame", "n": 64, "coils": 4, "spokes": 16, "newton": 7, "cg": 30,
         "previous": False},
        # one frame of the real-time series, started from and regularised toward the frame before
        {"name": "frame_384x10", "kind": "frame", "n": 384, "coils": 10, "spokes": 13, "newton": 7, "cg": 30,
         "previous": True},
        # the largest single frame
        {"name": "frame_512x16", "kind": "frame", "n": 512, "coils": 16, "spokes": 32, "newton": 8, "cg": 30,
         "previous": False},
        # 64 independent frames of uneven grid side, coil count and spokes, together
        {"name": "batch_64", "kind": "batch", "frames": 64, "shapes_seed": 1004, "newton": 7, "cg": 30},
        # reconstruction inside a training program: forward with checkpoints, then the gradient
        {"name": "vjp_128x6", "kind": "vjp", "n": 128, "coils": 6, "spokes": 15, "newton": 4, "cg": 12},
    ]


def draw(rng):
    kind = rng.choice(OPS + OPS + ("grid", "frame", "frame", "batch", "vjp"))
    if kind == "batch":
        return {"kind": kind, "frames": int(round(2.0 ** rng.uniform(1.0, 5.0))), "shapes_seed": rng.randrange(1, 1 << 20),
                "newton": rng.randrange(2, 8), "cg": rng.randrange(6, 31)}
    n = rng.choice(SIDES)
    coils = int(round(2.0 ** rng.uniform(1.0, 4.5)))
    case = {"kind": kind, "n": n, "coils": coils, "spokes": rng.randrange(7, 42)}
    if kind in OPS:
        # the un-oversampled image (n/4) as a rule, other widths now and then, odd ones among them
        case["fov"] = n // 4 if rng.random() < 0.6 else rng.randrange(max(2, n // 8), n // 2 + 1)
    elif kind == "frame":
        case.update(newton=rng.randrange(2, 9), cg=rng.randrange(6, 41), previous=rng.random() < 0.5)
    elif kind == "vjp":
        case.update(newton=rng.randrange(1, 6), cg=rng.randrange(6, 25))
    return case


# ------------------------------------------------------------------------------------------------- inputs ----
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _coords(n, dev):
    i = torch.arange(n, device=dev)
    return ((i + n // 2) % n - n // 2).to(torch.float64)


def _weight(n, dev):
    g = _coords(n, dev)
    k2 = (g[:, None] ** 2 + g[None, :] ** 2) / float(n * n)
    return (1.0 + SOBOLEV_A * k2) ** (-0.5 * SOBOLEV_L)


def _omega(n, fov, dev):
    g = _coords(n, dev)
    inside = (g >= -fov) & (g < fov)
    return (inside[:, None] & inside[None, :]).to(torch.float64)


def _noise(shape, gen, dev):
    return torch.randn(shape, dtype=torch.complex64, device=dev, generator=gen) * math.sqrt(2.0)


def _fft(a):
    return torch.fft.fft2(a, norm="ortho")


def _ifft(a):
    return torch.fft.ifft2(a, norm="ortho")


def _scene(n, coils, fov, rng, dev):
    """Ellipse phantom with a smooth phase and Gaussian coils on a circle, complex64 in natural FFT order."""
    g = _coords(n, dev) / (2.0 * fov)
    u1, u2 = g[:, None], g[None, :]
    img = torch.zeros((n, n), dtype=torch.float64, device=dev)
    for _ in range(8):
        r, phi, th = 0.3 * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi), rng.uniform(0, math.pi)
        ax, ay = rng.uniform(0.05, 0.4, size=2)
        d1, d2 = u1 - r * math.sin(phi), u2 - r * math.cos(phi)
        e1, e2 = (d2 * math.cos(th) + d1 * math.sin(th)) / ax, (d1 * math.cos(th) - d2 * math.sin(th)) / ay
        img += rng.uniform(0.1, 1.0) * ((e1 * e1 + e2 * e2) <= 1.0)
    img = img * _omega(n, fov, dev)
    img = img / img.max().clamp_min(1e-3)
    k1, k2, p0 = rng.uniform(0.5, 1.5), rng.uniform(0.5, 1.5), rng.uniform(0, 2 * math.pi)
    rho = torch.polar(img, 0.3 * torch.sin(2 * math.pi * (k1 * u1 + k2 * u2) + p0))
    c = []
    for j in range(coils):
        px, py = 0.5 * math.cos(2 * math.pi * j / coils), 0.5 * math.sin(2 * math.pi * j / coils)
        mag = torch.exp(-((u2 - px) ** 2 + (u1 - py) ** 2) / (2 * 0.35 ** 2))
        c.append(torch.polar(mag, torch.full_like(mag, rng.uniform(0, 2 * math.pi))))
    return rho.to(torch.complex64), torch.stack(c).to(torch.complex64)


def _mask(n, spokes, rng, dev):
    return torch.from_numpy(synth.radial_mask(n, spokes, float(rng.uniform(0, math.pi / spokes)))).to(dev)


def _data(rho, c, mask, fov, gen):
    """Gridded data of the scene with noise 30 dB below the sampled signal."""
    n, dev = rho.shape[-1], rho.device
    clean = mask * _fft(_omega(n, fov, dev).to(torch.float32) * rho * c)
    power = clean.abs().square().sum() / (mask.sum() * c.shape[0])
    return clean + mask * _noise(c.shape, gen, dev) * torch.sqrt(0.5 * power * 1e-3)


def _estimate(rho, c, w):
    """An estimate x = (rho, chat) as the method finds it: chat in the range of w FFT, image-domain coils near c."""
    return torch.cat([rho[None], (w * _fft(c)).to(torch.complex64)])


def _start(n, coils, dev):
    x = torch.zeros((1 + coils, n, n), dtype=torch.complex64, device=dev)
    x[0] = 1.0
    return x


def _frame_inputs(n, coils, spokes, seed, previous):
    dev = _device()
    rng, gen = np.random.default_rng(seed), torch.Generator(device=dev).manual_seed(seed)
    fov = n // 4
    rho, c = _scene(n, coils, fov, rng, dev)
    mask = _mask(n, spokes, rng, dev)
    y = _data(rho, c, mask, fov, gen)
    # the frame before: the same object a little blurred in contrast, with the noise of an undersampled frame
    x0 = _estimate(0.9 * rho + 0.02 * _omega(n, fov, dev) * _noise((n, n), gen, dev), c, _weight(n, dev)).contiguous() \
        if previous else _start(n, coils, dev)
    return {"y": y.contiguous(), "mask": mask, "x0": x0.to(torch.complex64)}


def _batch_shapes(case):
    return synth.uneven_batch_shapes(case["frames"], case["shapes_seed"])


def _spoke_angles(case, seed):
    first = float(np.random.default_rng(seed).uniform(0, math.pi / case["spokes"]))
    return [math.pi * s / case["spokes"] + first for s in range(case["spokes"])]


def _inputs(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "batch":
        return {"frames": [_frame_inputs(n, j, s, 1000 * seed + i, False)
                           for i, (n, j, s) in enumerate(_batch_shapes(case))]}
    n, coils = case["n"], case["coils"]
    rng, gen = np.random.default_rng(seed), torch.Generator(device=dev).manual_seed(seed)
    if kind == "grid":
        return {"samples": _noise((coils, case["spokes"], 2 * n), gen, dev)}
    if kind == "frame":
        return _frame_inputs(n, coils, case["spokes"], seed, case["previous"])
    if kind == "vjp":
        got = _frame_inputs(n, coils, case["spokes"], seed, False)
        got["g"] = _noise((1 + coils, n, n), gen, dev)
        got["g"][1:] *= _weight(n, dev).to(torch.float32)
        return got
    w = _weight(n, dev)
    rho, c = _scene(n, coils, case["fov"], rng, dev)
    mask = _mask(n, case["spokes"], rng, dev)
    got = {"x": _estimate(rho, c, w).contiguous(), "mask": mask}
    if kind in ("derivative", "normal"):
        d = _noise((1 + coils, n, n), gen, dev)
        d[1:] *= w.to(torch.float32)
        got["d"] = d.contiguous()
    if kind == "adjoint":
        got["r"] = (mask * _noise((coils, n, n), gen, dev)).contiguous()
    if kind == "grad":
        got["y"] = _data(rho, c, mask, case["fov"], gen).contiguous()
    return got


ALPHA = 0.0625       # alpha_n of a middle Gauss-Newton step, for the normal operator


def prepare(case, seed):
    state = _inputs(case, seed)
    state["kind"] = kind = case["kind"]
    if kind == "batch":
        state["op"] = NlinvBatch([(n, j) for n, j, _ in _batch_shapes(case)], newton_steps=case["newton"],
                                 cg_iters=case["cg"])
    elif kind == "grid":
        angles = _spoke_angles(case, seed)
        state["op"] = Gridder(case["n"], [(math.cos(a), math.sin(a)) for a in angles])
    elif kind in ("frame", "vjp"):
        state["op"] = Nlinv(case["n"], case["coils"], newton_steps=case["newton"], cg_iters=case["cg"])
    else:
        state["op"] = Nlinv(case["n"], case["coils"], fov=case["fov"])
    if kind == "grad":
        state["x"].requires_grad_(True)
    if kind == "vjp":
        state["y"].requires_grad_(True)
        state["x0"].requires_grad_(True)
    return state


def run(state):
    kind, op = state["kind"], state["op"]
    if kind == "forward":
        return op.forward(state["x"], state["mask"])
    if kind == "derivative":
        return op.derivative(state["x"], state["mask"], state["d"])
    if kind == "adjoint":
        return op.adjoint(state["x"], state["mask"], state["r"])
    if kind == "normal":
        return op.normal(state["x"], state["mask"], state["d"], ALPHA)
    if kind == "grad":
        fx = autograd.forward(op, state["x"], state["mask"])
        (gx,) = torch.autograd.grad(fx, state["x"], fx.detach() - state["y"])
        return {"F": fx.detach(), "grad": gx}
    if kind == "grid":
        y, mask = op.grid(state["samples"])
        return {"y": y, "mask": mask}
    if kind == "frame":
        return op.reconstruct(state["y"], state["mask"], state["x0"])
    if kind == "batch":
        fr = state["frames"]
        return op.reconstruct([f["y"] for f in fr], [f["mask"] for f in fr], [f["x0"].clone() for f in fr])
    x = autograd.reconstruct(op, state["y"], state["mask"], state["x0"])
    gy, g0 = torch.autograd.grad(x, (state["y"], state["x0"]), state["g"])
    return {"x": x.detach(), "grad_y": gy, "grad_x0": g0}


# --------------------------------------------------------------------------------------------------- work ----
def _fft2_flops(n, planes):
    return 10.0 * n * n * math.log2(n) * planes


def _frame_work(n, coils, newton, cg):
    """y, mask, x_0 read, x_N written; two 2D transforms per coil and operator: coil maps, F and DF^H per Newton
    step, DF and DF^H per conjugate-gradient iteration."""
    u = 8.0 * n * n
    return (3 * coils + 2) * u + n * n, newton * (4 + 4 * cg) * _fft2_flops(n, coils)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_frame_work(n, j, case["newton"], case["cg"]) for n, j, _ in _batch_shapes(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    n, j = case["n"], case["coils"]
    u = 8.0 * n * n
    if kind == "grid":
        return {"bytes": 8.0 * j * case["spokes"] * 2 * n + j * u + n * n, "flops": 2.0 * j * case["spokes"] * 2 * n}
    if kind == "frame":
        b, f = _frame_work(n, j, case["newton"], case["cg"])
        return {"bytes": b, "flops": f}
    if kind == "vjp":
        b, f = _frame_work(n, j, case["newton"], case["cg"])
        return {"bytes": b + (1 + j) * u + (1 + 2 * j) * u, "flops": 2.0 * f}
    planes = {"forward": 1 + 2 * j, "derivative": 2 + 3 * j, "adjoint": 2 + 3 * j, "normal": 3 + 3 * j,
              "grad": 2 + 4 * j}[kind]
    transforms = {"forward": 2, "derivative": 3, "adjoint": 3, "normal": 5, "grad": 5}[kind]
    return {"bytes": planes * u + n * n, "flops": transforms * _fft2_flops(n, j)}


# -------------------------------------------------------------------------------------------------- exact ----
class _Method:
    """The method in complex128 torch."""

    def __init__(self, n, fov, mask, dev):
        self.w, self.m, self.p = _weight(n, dev), _omega(n, fov, dev), mask.to(torch.float64)

    def coils(self, x):
        return _ifft(self.w * x[1:])

    def forward(self, x, c):
        return self.p * _fft(self.m * x[0] * c)

    def derivative(self, x, c, d):
        return self.p * _fft(self.m * (d[0] * c + x[0] * _ifft(self.w * d[1:])))

    def adjoint(self, x, c, r):
        z = self.m * _ifft(self.p * r)
        return torch.cat([(c.conj() * z).sum(0, keepdim=True), self.w * _fft(x[0].conj() * z)])

    def normal(self, x, c, d, alpha):
        return self.adjoint(x, c, self.derivative(x, c, d)) + alpha * d

    def solve(self, x, c, alpha, b, iters):
        """Conjugate gradients from zero for a fixed count, ending early at the single-precision rounding floor."""
        dx, r, p = torch.zeros_like(b), b.clone(), b.clone()
        rr = rr0 = float(torch.linalg.vector_norm(r)) ** 2
        for _ in range(iters):
            if not rr > 2.0 ** -48 * rr0:
                break
            q = self.normal(x, c, p, alpha)
            pq = float((p.conj() * q).sum().real)
            if not pq > 0.0:
                break
            a = rr / pq
            dx += a * p
            r -= a * q
            new = float(torch.linalg.vector_norm(r)) ** 2
            p = r + (new / rr) * p
            rr = new
        return dx

    def iterates(self, y, x0, newton, cg):
        xs, alphas = [x0], [0.5 ** k for k in range(newton)]
        for alpha in alphas:
            x = xs[-1]
            c = self.coils(x)
            b = self.adjoint(x, c, y - self.forward(x, c)) - alpha * (x - x0)
            xs.append(x + self.solve(x, c, alpha, b, cg))
        return xs, alphas

    def backward(self, y, xs, alphas, g, cg):
        """Gradients with respect to y and the start value, each Newton step differentiated implicitly."""
        gy, gref = torch.zeros_like(y), torch.zeros_like(g)
        for k in reversed(range(len(alphas))):
            x, alpha = xs[k], alphas[k]
            dx = xs[k + 1] - x
            c, dc = self.coils(x), self.coils(dx)
            u = self.solve(x, c, alpha, g, cg)
            v = self.derivative(x, c, u)
            s = y - self.forward(x, c) - self.derivative(x, c, dx)
            gy += v
            gref += alpha * u
            g = self.adjoint(u, self.coils(u), s) - self.adjoint(dx, dc, v)
        return gy, g + gref


def _wide(t):
    return t.detach().to(torch.complex128)


def _exact_frame(fr, newton, cg):
    m = _Method(fr["y"].shape[-1], fr["y"].shape[-1] // 4, fr["mask"], fr["y"].device)
    return m.iterates(_wide(fr["y"]), _wide(fr["x0"]), newton, cg)[0][-1]


def _exact_grid(case, samples, angles):
    """Every grid point holds the mean of the samples that round to it."""
    n = case["n"]
    t = (np.arange(2 * n) - n) * 0.5
    kx = np.floor(np.outer(np.cos(angles), t) + 0.5).astype(np.int64)
    ky = np.floor(np.outer(np.sin(angles), t) + 0.5).astype(np.int64)
    ok = (kx >= -n // 2) & (kx < n // 2) & (ky >= -n // 2) & (ky < n // 2)
    at = torch.from_numpy(((ky % n) * n + kx % n)[ok]).to(samples.device)
    vals = samples.to(torch.complex128)[:, torch.from_numpy(ok).to(samples.device)]
    total = torch.zeros((samples.shape[0], n * n), dtype=torch.complex128, device=samples.device)
    total.index_add_(1, at, vals)
    count = torch.bincount(at, minlength=n * n)
    return (total / count.clamp_min(1)).reshape(-1, n, n)


def exact(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    if kind == "batch":
        return [_exact_frame(f, case["newton"], case["cg"]) for f in s["frames"]]
    if kind == "grid":
        return {"y": _exact_grid(case, s["samples"], _spoke_angles(case, seed)), "mask": None}
    if kind == "frame":
        return _exact_frame(s, case["newton"], case["cg"])
    n, dev = case["n"], s["mask"].device
    if kind == "vjp":
        m, y = _Method(n, n // 4, s["mask"], dev), _wide(s["y"])
        xs, alphas = m.iterates(y, _wide(s["x0"]), case["newton"], case["cg"])
        gy, g0 = m.backward(y, xs, alphas, _wide(s["g"]), case["cg"])
        return {"x": xs[-1], "grad_y": gy, "grad_x0": g0}
    m, x = _Method(n, case["fov"], s["mask"], dev), _wide(s["x"])
    c = m.coils(x)
    if kind == "forward":
        return m.forward(x, c)
    if kind == "derivative":
        return m.derivative(x, c, _wide(s["d"]))
    if kind == "adjoint":
        return m.adjoint(x, c, _wide(s["r"]))
    if kind == "normal":
        return m.normal(x, c, _wide(s["d"]), ALPHA)
    fx = m.forward(x, c)
    return {"F": fx, "grad": m.adjoint(x, c, fx - _wide(s["y"]))}
