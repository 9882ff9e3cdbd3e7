"""The calls this library is timed on: what each stands for, its inputs, and its result in 64 bits.

A case is one call of the public Python interface (`fresnel.FresnelPlan`,
`FresnelBatch`, `LinePlan`, `direct_sum`, the learned-kernel calls of `capi`) at
one size.  `listed()` names twelve of them, from a 64 x 64 transform, which is
all latency, to gradients on 4096 x 4096 samples; `draw(rng)` gives others of
the same ranges.  `exact(case, seed)` evaluates the same sums in float64 with
torch alone: a non-uniform FFT with a width-14 kernel (error about 1e-12), or
the direct sum where that is small.

Lengths are in micrometres and nanometres in a case, in metres everywhere else.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1203_3583_gb300 import capi
from paper_1203_3583_gb300.fresnel import FresnelBatch, FresnelPlan, LinePlan, direct_sum

UM, NM, TAU = 1e-6, 1e-9, 2.0 * math.pi


# ---- the cases ----------------------------------------------------------------

def _grid(call, n1x, n1y, m2x, m2y, p1, p2, lam, z0, surface, height, field="random", **more):
    """A case of a surface on an n1x x n1y grid of pitch p1 (um) and a destination
    of m2x x m2y points of pitch p2 (um), wavelength lam (nm), distance z0 (m)."""
    return dict(call=call, n1x=n1x, n1y=n1y, m2x=m2x, m2y=m2y, p1=p1, p2=p2, lam=lam, z0=z0,
                surface=surface, height=height, field=field, **more)


def listed():
    return [
        # one small transform: a tile of a larger scene, or an interactive preview
        dict(_grid("forward", 64, 64, 64, 64, 10.0, 10.0, 633, 0.05, "sinusoid", 20.0, width=7),
             name="forward_64"),
        # the line sources of the paper's own experiments: 1024 samples along a curve
        dict(call="line", n=1024, m2=1024, p1=10.0, p2=10.0, lam=633, z0=1.0, width=7,
             name="line_1024"),
        # a binary mask on a spherical cap
        dict(_grid("forward", 1024, 1024, 1024, 1024, 8.0, 8.0, 532, 0.2, "cap", 0.0, "mask",
                   width=7), name="forward_cap_1024"),
        # an odd-sized, non-square surface under tilted light, at a preview's accuracy
        dict(_grid("forward", 1502, 998, 1024, 512, 5.0, 7.0, 532, 0.12, "smooth", 40.0, width=5,
                   sx=0.011, sy=-0.017), name="forward_ragged_w5"),
        # the standard transform: random field on a smooth random surface
        dict(_grid("forward", 2048, 2048, 2048, 2048, 4.0, 4.0, 633, 0.1, "smooth", 50.0, width=7),
             name="forward_2048"),
        # the same at the width that reference fields are computed with
        dict(_grid("forward", 2048, 2048, 2048, 2048, 4.0, 4.0, 633, 0.1, "smooth", 50.0, width=12),
             name="forward_2048_w12"),
        # the same with bit-reproducible results
        dict(_grid("forward", 2048, 2048, 2048, 2048, 4.0, 4.0, 633, 0.1, "smooth", 50.0, width=7,
                   deterministic=True), name="forward_2048_repeatable"),
        # a step of a surface and hologram optimisation through autograd: a new
        # height map, the transform, the gradients of both inputs
        dict(_grid("step", 1024, 1024, 1024, 1024, 8.0, 8.0, 532, 0.2, "smooth", 30.0, width=7),
             name="step_1024"),
        # both gradients of the largest standard surface
        dict(_grid("adjoint", 4096, 4096, 4096, 4096, 3.74, 3.74, 532, 0.15, "tiltbump", 30.0,
                   "phase", width=7), name="adjoint_4096"),
        # many surfaces of mixed sizes in red, green and blue, one call
        dict(call="batch", count=24, smallest=256, largest=2048, pick=4, width=7, name="batch_24"),
        # the gradient of a training step of the learned kernel
        dict(_grid("learned", 2048, 2048, 2048, 2048, 4.0, 4.0, 633, 0.1, "smooth", 50.0),
             name="learned_gradient_2048"),
        # the direct sum of Eq. 7 at sampled points, the check of a transform
        dict(_grid("direct", 1024, 1024, 1024, 1024, 8.0, 8.0, 532, 0.2, "cap", 0.0, form=7,
                   points=256), name="direct_1024"),
    ]


def _even(rng, lo, hi):
    return 2 * int(round(0.5 * lo * (hi / lo) ** rng.random()))


def _pow2(rng, lo, hi):
    return 2 ** rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def _drawn_grid(rng, call, lo, hi, mhi, **more):
    """Source sizes over [lo, hi], now and then square; destination sizes powers
    of two up to mhi (the fine grid's); the distance puts the samples over 0.2
    to 0.9 of the fine grid, so that no footprint wraps."""
    n1x = _even(rng, lo, hi)
    n1y = n1x if rng.random() < 0.4 else min(hi, max(lo, _even(rng, max(lo, n1x // 3), n1x * 2)))
    m2x = _pow2(rng, 64, mhi)
    m2y = m2x if rng.random() < 0.6 else max(64, m2x // 2)
    p1, p2 = round(rng.uniform(3.0, 10.0), 2), round(rng.uniform(3.0, 10.0), 2)
    lam = rng.choice((450, 532, 633))
    z0 = max(n1x, n1y) * p1 * UM * p2 * UM / (lam * NM * rng.uniform(0.2, 0.9))
    surface = rng.choice(("smooth", "smooth", "sinusoid", "tiltbump"))
    height = round(min(rng.uniform(5.0, 50.0), 2e-3 * z0 / UM), 3)
    return _grid(call, n1x, n1y, m2x, m2y, p1, p2, lam, round(z0, 6), surface, height,
                 rng.choice(("random", "phase", "mask")), **more)


def draw(rng: random.Random):
    what = rng.random()
    if what < 0.45:
        more = dict(width=rng.choice((4, 5, 6, 7, 7, 7, 8, 10, 12)))
        if rng.random() < 0.25:
            more["deterministic"] = True
        if rng.random() < 0.25:
            more.update(sx=round(rng.uniform(-0.02, 0.02), 4), sy=round(rng.uniform(-0.02, 0.02), 4))
        return _drawn_grid(rng, "forward", 48, 2400, 2048, **more)
    if what < 0.57:
        return _drawn_grid(rng, "step", 128, 1536, 1024, width=rng.choice((5, 7, 7)))
    if what < 0.69:
        return _drawn_grid(rng, "adjoint", 128, 3000, 2048, width=rng.choice((4, 7, 7, 8)))
    if what < 0.78:
        n = int(round(300 * (16384 / 300) ** rng.random()))
        return dict(call="line", n=n, m2=_pow2(rng, 128, 4096), p1=round(rng.uniform(4.0, 12.0), 2),
                    p2=round(rng.uniform(4.0, 12.0), 2), lam=rng.choice((450, 532, 633)),
                    z0=round(rng.uniform(0.8, 1.5), 3), width=rng.choice((5, 7, 9)))
    if what < 0.86:
        return dict(call="batch", count=rng.randint(2, 16), smallest=256,
                    largest=rng.choice((512, 1024)), pick=rng.randrange(1 << 20), width=7)
    if what < 0.92:
        return _drawn_grid(rng, "learned", 128, 1024, 1024)
    return _drawn_grid(rng, "direct", 48, 1024, 1024, form=rng.choice((7, 7, 5, 2)),
                       points=rng.randint(16, 256))


# ---- inputs -------------------------------------------------------------------

def _geometry(c):
    g = dict(n1x=c["n1x"], n1y=c["n1y"], p1x=c["p1"] * UM, p1y=c["p1"] * UM, m2x=c["m2x"],
             m2y=c["m2y"], p2x=c["p2"] * UM, p2y=c["p2"] * UM, lam=c["lam"] * NM, z0=c["z0"])
    g.update({k: c[k] for k in ("sx", "sy") if k in c})
    return g


def _axes(g, which="1"):
    n, m = ("n1x", "n1y") if which == "1" else ("m2x", "m2y")
    p = "p" + which
    at = lambda k, q: (torch.arange(g[k], dtype=torch.float64, device="cuda") - g[k] // 2) * g[q]  # noqa: E731
    return at(n, p + "x"), at(m, p + "y")


def _surface(kind, g, height, rng):
    """Height map in metres, float64, of `height` micrometres."""
    x, y = _axes(g)
    h = height * UM
    if kind == "sinusoid":
        k = TAU / (320 * UM)
        return h * torch.sin(k * y)[:, None] * torch.sin(k * x)[None, :]
    rho2 = (y * y)[:, None] + (x * x)[None, :]
    if kind == "cap":
        r2 = 0.02 ** 2
        edge = (g["n1x"] / 2 * g["p1x"]) ** 2 + (g["n1y"] / 2 * g["p1y"]) ** 2
        return torch.sqrt(r2 - rho2) - math.sqrt(r2 - edge)
    if kind == "tiltbump":
        tilt = math.tan(math.radians(2.0)) if g["n1x"] * g["p1x"] > 8e-3 else 2.0 * h / (g["n1x"] * g["p1x"])
        return x[None, :] * tilt + h * torch.exp(-rho2 / (2 * (g["n1x"] * g["p1x"] / 8) ** 2))
    noise = torch.randn(g["n1y"], g["n1x"], dtype=torch.float64, device="cuda", generator=rng)
    sigma = min(40.0, min(g["n1x"], g["n1y"]) / 8)
    fy = torch.fft.fftfreq(g["n1y"], dtype=torch.float64, device="cuda")[:, None]
    fx = torch.fft.fftfreq(g["n1x"], dtype=torch.float64, device="cuda")[None, :]
    s = torch.fft.ifft2(torch.fft.fft2(noise) * torch.exp(-2 * (math.pi * sigma) ** 2 * (fx * fx + fy * fy))).real
    s = s - s.min()
    return s * (h / s.max())


def _field(kind, shape, rng):
    u = torch.rand(*shape, dtype=torch.float64, device="cuda", generator=rng)
    if kind == "mask":
        return (u < 0.5).to(torch.complex64)
    amp = torch.rand(*shape, dtype=torch.float64, device="cuda", generator=rng) if kind == "random" else torch.ones_like(u)
    return torch.polar(amp, TAU * u).to(torch.complex64)


def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _inputs(c, seed):
    """(geometry, heights float64, field complex64, generator) of a surface's case."""
    rng, g = _rng(seed), _geometry(c)
    d1 = _surface(c["surface"], g, c["height"], rng).contiguous()
    return g, d1, _field(c["field"], (g["n1y"], g["n1x"]), rng), rng


def _gradient_in(g, rng):
    """dL/du2 of a loss on the destination: a random complex field."""
    return torch.view_as_complex(torch.randn(g["m2y"], g["m2x"], 2, device="cuda", generator=rng))


def _line_inputs(c, seed):
    """A line source sampled along a smooth curve, its heights and weights."""
    rng = np.random.default_rng(seed)
    p, n = c["p1"] * UM, c["n"]
    slope = np.interp(np.arange(n), np.linspace(0, n, 17), rng.uniform(-1.0, 1.0, 17))
    dx = p / np.sqrt(1 + slope ** 2)
    x1, d1 = np.cumsum(dx), np.cumsum(slope * dx)
    u1 = (rng.random(n) * np.exp(1j * TAU * rng.random(n))).astype(np.complex64)
    line = dict(m2=c["m2"], p2=c["p2"] * UM, lam=c["lam"] * NM, z0=c["z0"])
    return line, x1 - x1.mean(), d1 - d1.mean(), dx, torch.as_tensor(u1, device="cuda")


def _batch_items(c, seed):
    """Sizes, colours and distances from the case, surfaces and fields from the seed."""
    pick, rng, items = random.Random(c["pick"]), _rng(seed), []
    sizes = [n for n in (256, 512, 1024, 2048) if c["smallest"] <= n <= c["largest"]]
    for i in range(c["count"]):
        n = pick.choice(sizes)
        g = dict(n1x=n, n1y=n, p1x=3 * UM, p1y=3 * UM, m2x=n, m2y=n, p2x=3 * UM, p2y=3 * UM,
                 lam=(450 * NM, 532 * NM, 633 * NM)[i % 3], z0=pick.uniform(0.05, 0.3))
        d1 = _surface(pick.choice(("sinusoid", "smooth")), g, pick.uniform(5.0, 50.0), rng)
        items.append((g, d1.contiguous(), _field("random", (n, n), rng)))
    return items


_W4, _COEF, _FEAT, _HID, _CHEB = 4, 8, 6, 32, 6  # the learned model's sizes (include/asfd.h)


def _learned_params(seed):
    """A model early in its training: tap polynomials that only roughly fit the
    width-4 kernel, a random hidden layer and deconvolution correction."""
    rng = np.random.default_rng(seed)
    t = np.cos(math.pi * (np.arange(64) + 0.5) / 64)
    base = []
    for a in range(_W4):
        u = (t + 1 + 2 * a - _W4) / _W4
        psi = np.exp(2.30 * _W4 * (np.sqrt(np.maximum(0.0, 1 - u * u)) - 1))
        base.append(np.linalg.lstsq(t[:, None] ** np.arange(_COEF), psi, rcond=None)[0])
    base = np.stack([np.stack(base)] * 2) * (1 + 0.25 * rng.standard_normal((2, _W4, _COEF)))
    rest = [rng.uniform(-0.5, 0.5, _HID * _FEAT), rng.uniform(-0.1, 0.1, _HID),
            0.3 * rng.standard_normal(2 * _W4 * _COEF * _HID), 0.1 * rng.standard_normal(2 * _W4 * _COEF),
            0.01 * rng.standard_normal(2 * _CHEB)]
    return np.concatenate([base.ravel()] + rest).astype(np.float32)


def _points(c, g, seed):
    rng = np.random.default_rng(seed)
    flat = rng.choice(g["m2x"] * g["m2y"], size=c["points"], replace=False)
    return [torch.as_tensor(v.astype(np.int32), device="cuda") for v in (flat % g["m2x"], flat // g["m2x"])]


def prepare(case, seed):
    c, call = case, case["call"]
    if call == "line":
        line, x1, d1, w, u1 = _line_inputs(c, seed)
        return call, LinePlan(line, x1, d1, w, kernel_width=c["width"]), u1
    if call == "batch":
        items = _batch_items(c, seed)
        return call, FresnelBatch([(g, d1) for g, d1, _ in items], kernel_width=c["width"]), [u for _, _, u in items]
    g, d1, u1, rng = _inputs(c, seed)
    if call == "direct":
        return call, g, d1, u1, c["form"], _points(c, g, seed)
    if call == "learned":
        plan = FresnelPlan(g, d1, kind="learned")
        capi.asfd_learned_set_params(plan.handle, _learned_params(seed))
        return call, plan, u1, _type1(g, d1, u1).to(torch.complex64)
    plan = FresnelPlan(g, d1, kernel_width=c["width"], deterministic=c.get("deterministic", False))
    if call == "forward":
        return call, plan, u1
    if call == "step":  # heights as an optimiser holds them: float32 leaves
        return call, plan, u1.requires_grad_(), d1.float().requires_grad_(), _gradient_in(g, rng)
    return (call, plan, u1, _gradient_in(g, rng), torch.empty_like(u1),
            torch.empty(u1.shape, dtype=torch.float32, device="cuda"))


def run(state):
    call = state[0]
    if call in ("forward", "line", "batch"):
        return state[1].execute(state[2])
    if call == "direct":
        _, g, d1, u1, form, points = state
        return direct_sum(g, d1, u1, form, points)
    if call == "learned":
        _, plan, u1, ref = state
        gradient, loss = capi.asfd_learned_gradient(plan.handle, u1, ref, plan.shape1, plan.shape2)
        return {"gradient": gradient, "loss": loss}
    if call == "step":
        _, plan, u1, d1, g2 = state
        u2 = plan(u1, d1)
        gu1, gd1 = torch.autograd.grad(u2, (u1, d1), g2)
        return {"u2": u2.detach(), "u1": gu1, "d1": gd1}
    _, plan, u1, g2, gu1, gd1 = state
    plan.adjoint(u1, g2, gu1, gd1)
    return {"u1": gu1, "d1": gd1}


def work(case):
    c, call = case, case["call"]
    fft = lambda cells: 5.0 * cells * math.log2(cells)  # noqa: E731
    if call == "line":  # field, prefactor and position of each sample; the destination
        return {"bytes": 24.0 * c["n"] + 8.0 * c["m2"],
                "flops": (4.0 * c["width"] + 6) * c["n"] + fft(2.0 * c["m2"])}
    if call == "batch":
        pick, total = random.Random(c["pick"]), {"bytes": 0.0, "flops": 0.0}
        sizes = [n for n in (256, 512, 1024, 2048) if c["smallest"] <= n <= c["largest"]]
        for _ in range(c["count"]):
            n = pick.choice(sizes)
            pick.uniform(0, 1), pick.choice((0, 1)), pick.uniform(0, 1)
            total["bytes"] += 20.0 * n * n
            total["flops"] += 4.0 * c["width"] ** 2 * n * n + fft(4.0 * n * n)
        return total
    n, m, w = float(c["n1x"] * c["n1y"]), float(c["m2x"] * c["m2y"]), c.get("width", _W4)
    if call == "direct":  # heights and field; phase, sine, cosine and a complex sum a pair
        return {"bytes": 16.0 * n + 16.0 * c["points"], "flops": 30.0 * n * c["points"]}
    if call == "learned":  # field, heights, reference; taps both ways, their polynomials
        return {"bytes": 12.0 * n + 8.0 * m, "flops": (8.0 * w * w + 8.0 * w * _COEF) * n + 2 * fft(4 * m)}
    if call == "forward":
        return {"bytes": 12.0 * n + 8.0 * m, "flops": 4.0 * w * w * n + fft(4 * m)}
    if call == "adjoint":
        return {"bytes": 24.0 * n + 8.0 * m, "flops": 8.0 * w * w * n + fft(4 * m)}
    return {"bytes": 24.0 * n + 16.0 * m, "flops": 12.0 * w * w * n + 2 * fft(4 * m)}


# ---- the same in 64 bits, with torch alone ---------------------------------------

_WIDTH = 14
_BETA = 2.30 * _WIDTH


def _psi(z):
    return torch.exp(_BETA * (torch.sqrt(torch.clamp(1 - (2 * z / _WIDTH) ** 2, min=0.0)) - 1))


def _psi_hat(m, width=_WIDTH, beta=_BETA):
    """Fourier transform of the width-`width` kernel at the centred modes of a
    length-m axis oversampled twice."""
    z, w = np.polynomial.legendre.leggauss(200)
    psi = w * width / 2 * np.exp(beta * (np.sqrt(1 - z * z) - 1))
    k = np.arange(m) - m // 2
    return torch.as_tensor(np.cos(TAU / (2 * m) * np.outer(k, z * width / 2)) @ psi, device="cuda")


class _Uneven:
    """Sums over samples at the frequencies tx, ty (radians per destination
    index) and over the centred m2x x m2y destination indices, both ways."""

    def __init__(self, tx, ty, mx, my):
        self.n, self.m = (2 * my, 2 * mx), (my, mx)
        self.at = []
        for t, nf in ((ty, 2 * my), (tx, 2 * mx)):
            g = t.reshape(-1) * (nf / TAU)
            first = torch.ceil(g - _WIDTH / 2)
            self.at.append((first.long(), first - g))
        self.keep = [torch.remainder(torch.arange(m, device="cuda") - m // 2, nf) for m, nf in ((my, 2 * my), (mx, 2 * mx))]
        self.hat = _psi_hat(my)[:, None] * _psi_hat(mx)[None, :]

    def _taps(self, axis):
        first, off = self.at[axis]
        for i in range(_WIDTH):
            yield torch.remainder(first + i, self.n[axis]), _psi(off + i)

    def out(self, c):
        """sum_n c_n exp(-i (tx mx + ty my))"""
        c = c.reshape(-1)
        grid = torch.zeros(self.n[0] * self.n[1], 2, dtype=torch.float64, device="cuda")
        columns = list(self._taps(1))
        for iy, wy in self._taps(0):
            cy = c * wy
            for ix, wx in columns:
                grid.index_add_(0, iy * self.n[1] + ix, torch.view_as_real(cy * wx))
        f = torch.fft.fft2(torch.view_as_complex(grid).view(self.n))
        return f[self.keep[0]][:, self.keep[1]] / self.hat

    def back(self, a):
        """sum_m a_m exp(+i (tx mx + ty my))"""
        f = torch.zeros(self.n, dtype=torch.complex128, device="cuda")
        f[self.keep[0][:, None], self.keep[1][None, :]] = a / self.hat
        grid = (torch.fft.ifft2(f) * (self.n[0] * self.n[1])).view(-1)
        columns = list(self._taps(1))
        total = torch.zeros(self.at[0][0].numel(), dtype=torch.complex128, device="cuda")
        for iy, wy in self._taps(0):
            row = torch.zeros_like(total)
            for ix, wx in columns:
                row += grid[iy * self.n[1] + ix] * wx
            total += row * wy
        return total


def _terms(g, d1):
    """k, prefactor exp(i theta) p1x p1y of each sample, its frequencies and r0."""
    k = TAU / g["lam"]
    x, y = _axes(g)
    x, y = x[None, :], y[:, None]
    r0 = g["z0"] - d1
    sx, sy = g.get("sx", 0.0), g.get("sy", 0.0)
    sz = math.sqrt(1 - sx * sx - sy * sy)
    theta = k * (sx * x + sy * y + (sz - 1) * d1) + k * (x * x + y * y) / (2 * r0)
    e = torch.polar(torch.full_like(theta, g["p1x"] * g["p1y"]), theta)
    return k, e, k * g["p2x"] * x / r0, k * g["p2y"] * y / r0, r0, x, y, sz


def _outer(g, chirp=True):
    k = TAU / g["lam"]
    x2, y2 = _axes(g, "2")
    ph = k * g["z0"] + (k * ((x2 * x2)[None, :] + (y2 * y2)[:, None]) / (2 * g["z0"]) if chirp else torch.zeros(g["m2y"], g["m2x"], dtype=torch.float64, device="cuda"))
    return torch.polar(torch.full_like(ph, 1 / (g["lam"] * g["z0"])), ph - math.pi / 2)


def _type1(g, d1, u1):
    _, e, tx, ty = _terms(g, d1)[:4]
    return _outer(g) * _Uneven(tx, ty, g["m2x"], g["m2y"]).out(u1.to(torch.complex128) * e)


def _gradients(g, d1, u1, g2):
    k, e, tx, ty, r0, x, y, sz = _terms(g, d1)
    x2, y2 = _axes(g, "2")
    a = _outer(g).conj() * g2.to(torch.complex128)
    sums = _Uneven(tx, ty, g["m2x"], g["m2y"])
    s0, s1, s2 = (sums.back(v).view(d1.shape) for v in (a, a * x2[None, :], a * y2[:, None]))
    slope = (k * (sz - 1) + k * (x * x + y * y) / (2 * r0 * r0)) * s0.conj()
    slope = slope - k / (r0 * r0) * (x * s1.conj() + y * s2.conj())
    return {"u1": e.conj() * s0, "d1": (u1.to(torch.complex128) * e * 1j * slope).real}


def _exact_line(c, seed):
    line, x1, d1, w, u1 = _line_inputs(c, seed)
    k, z0 = TAU / line["lam"], line["z0"]
    x1, d1, w = (torch.as_tensor(v, device="cuda") for v in (x1, d1, w))
    r0 = z0 - d1
    a = u1.to(torch.complex128) * torch.polar(w, k * x1 * x1 / (2 * r0))
    x2 = (torch.arange(line["m2"], dtype=torch.float64, device="cuda") - line["m2"] // 2) * line["p2"]
    one = torch.ones((), dtype=torch.float64, device="cuda")
    s = torch.cat([torch.polar(one, -k * x[:, None] * (x1 / r0)[None, :]) @ a for x in x2.split(512)])
    ph = k * (z0 + x2 * x2 / (2 * z0)) - math.pi / 4
    return torch.polar(torch.full_like(ph, 1 / math.sqrt(line["lam"] * z0)), ph) * s


def _exact_direct(c, seed):
    g, d1, u1, _ = _inputs(c, seed)
    mx, my = _points(c, g, seed)
    k, e, _, _, r0, x, y, _ = _terms(g, d1)
    x2 = (mx.double() - g["m2x"] // 2) * g["p2x"]
    y2 = (my.double() - g["m2y"] // 2) * g["p2y"]
    a, one = u1.to(torch.complex128), torch.ones((), dtype=torch.float64, device="cuda")
    out = []
    for px, py in zip(x2.tolist(), y2.tolist()):
        if c["form"] == 2:
            r2 = (px - x) ** 2 + (py - y) ** 2 + r0 * r0
            out.append((a * torch.polar(1 / r2, k * (d1 + torch.sqrt(r2)))).sum() * (g["p1x"] * g["p1y"]))
            continue
        ph = -k * (px * x + py * y) / r0
        if c["form"] == 5:
            ph = ph + k * (px * px + py * py) / (2 * r0)
        out.append((a * e * torch.polar(one, ph)).sum())
    out = torch.stack(out)
    if c["form"] == 2:
        return out * (g["z0"] / (1j * g["lam"]))
    return out * _outer(g, c["form"] == 7)[my.long(), mx.long()]


def _exact_learned(c, seed):
    """Loss and gradient of the model that include/asfd.h lays out, by autograd in float64."""
    g, d1, u1, _ = _inputs(c, seed)
    ref = _type1(g, d1, u1).to(torch.complex64).to(torch.complex128)
    prm = torch.as_tensor(_learned_params(seed).astype(np.float64), device="cuda").requires_grad_()
    sizes = [2 * _W4 * _COEF, _HID * _FEAT, _HID, 2 * _W4 * _COEF * _HID, 2 * _W4 * _COEF, _CHEB, _CHEB]
    base, w1, b1, w2, b2, dx, dy = prm.split(sizes)
    _, e, tx, ty, r0 = _terms(g, d1)[:5]
    nf = (2 * g["m2y"], 2 * g["m2x"])
    pos = [t * (n / TAU) for t, n in ((ty, nf[0]), (tx, nf[1]))]
    # features of each 16 x 16 block of samples: means over the block
    ny, nx = d1.shape
    wide = (nx + 15) // 16
    block = (torch.arange(ny, device="cuda") // 16)[:, None] * wide + (torch.arange(nx, device="cuda") // 16)[None, :]
    blocks = wide * ((ny + 15) // 16)

    def mean(v, b, none):
        zero = torch.zeros(blocks, dtype=torch.float64, device="cuda")
        s = zero.index_add(0, b.reshape(-1), v.reshape(-1))
        n = zero.index_add(0, b.reshape(-1), torch.ones_like(v).reshape(-1))
        return torch.where(n > 0, s / n.clamp(min=1), torch.full_like(s, none))

    f = torch.stack([torch.ones(blocks, dtype=torch.float64, device="cuda"),
                     mean(pos[1] / (nf[1] / 2), block, 0.0), mean(pos[0] / (nf[0] / 2), block, 0.0),
                     mean(pos[1][:, 1:] - pos[1][:, :-1], block[:, :-1], 1.0) - 1,
                     mean(pos[0][1:] - pos[0][:-1], block[:-1], 1.0) - 1,
                     100 * mean(d1 / r0, block, 0.0)], 1)
    hidden = torch.tanh(f @ w1.view(_HID, _FEAT).T + b1)
    table = (base + 1e-3 * (hidden @ w2.view(-1, _HID).T + b2)).view(blocks, 2, _W4, _COEF)
    at, taps, block = [], [], block.reshape(-1)
    for axis, p in ((0, pos[1]), (1, pos[0])):  # tables hold x first
        first = torch.ceil(p.reshape(-1) - _W4 / 2)
        t = 2 * (first - p.reshape(-1)) + _W4 - 1  # 2 dx - 1, dx in [0, 1) from the window's edge
        at.append(first.long())
        row = []
        for a in range(_W4):
            coef = table[:, axis, a][block]
            v = coef[:, -1]
            for k in range(_COEF - 2, -1, -1):
                v = v * t + coef[:, k]
            row.append(v)
        taps.append(row)
    a = (u1.to(torch.complex128) * e).reshape(-1)
    grid = torch.zeros(nf[0] * nf[1], dtype=torch.complex128, device="cuda")
    for b in range(_W4):
        ab = a * taps[1][b]
        iy = torch.remainder(at[1] + b, nf[0]) * nf[1]
        for i in range(_W4):
            grid = grid.index_add(0, iy + torch.remainder(at[0] + i, nf[1]), ab * taps[0][i])
    spectrum = torch.fft.fft2(grid.view(nf))
    u2 = _outer(g)
    for axis, (m, d) in enumerate(((g["m2y"], dy), (g["m2x"], dx))):
        k = torch.arange(m, device="cuda") - m // 2
        spectrum = spectrum.index_select(axis, torch.remainder(k, 2 * m))
        u = (2.0 * k / m).clamp(-1, 1)
        fix = 1 + sum(d[j] * torch.cos(2 * (j + 1) * torch.acos(u)) for j in range(_CHEB))
        fix = fix / _psi_hat(m, _W4, 2.30 * _W4)
        u2 = u2 * (fix[:, None] if axis == 0 else fix[None, :])
    u2 = u2 * spectrum
    loss = ((u2 - ref).abs() ** 2).sum() / (ref.abs() ** 2).sum()
    grad, = torch.autograd.grad(loss, prm)
    return {"gradient": grad, "loss": loss.detach()}


def exact(case, seed):
    c, call = case, case["call"]
    if call == "line":
        return _exact_line(c, seed)
    if call == "batch":
        return [_type1(g, d1, u1) for g, d1, u1 in _batch_items(c, seed)]
    if call == "direct":
        return _exact_direct(c, seed)
    if call == "learned":
        return _exact_learned(c, seed)
    g, d1, u1, rng = _inputs(c, seed)
    if call == "forward":
        return _type1(g, d1, u1)
    g2 = _gradient_in(g, rng)
    if call == "adjoint":
        return _gradients(g, d1, u1, g2)
    d1 = d1.float().double()
    return {"u2": _type1(g, d1, u1), **_gradients(g, d1, u1, g2)}
