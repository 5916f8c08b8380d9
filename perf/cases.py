"""Performance cases of the solver: what is timed, on which inputs, and what
the results are in 64 bits.

Every case goes through the package's public entry points (Plan.solve, Batch,
potential_of_wave, evolve).  Kinds of case:

* "solve":  one density -> one potential on an existing plan, for the DS
  multiplier, another multiplier of the family, or the standard periodic
  solver; plans from explicit polar parameters or from Plan.auto.
* "grad":   Phi(|u|^2) of a wave function and the gradient of sum w Phi with
  respect to u (one solve and one adjoint solve).
* "evolve": time steps of the DS loop (Strang or Yoshida), with the gradient
  with respect to the initial field through checkpointed recomputation where
  the case says so.
* "batch":  many densities on several grid sizes, one captured graph.

Grid sizes are powers of two per axis (all the library accepts); what is odd
or ragged is the rest: unequal axes, domain lengths, disk radii, node counts,
kernel widths, batch compositions.

A program that works in single precision (a mixed plan, complex64 fields)
keeps the potential in single precision too: its cases return it as float32.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1409_2014_gb300 import Batch, Plan
from paper_1409_2014_gb300.ds import DSPlan, evolve, potential_of_wave

TWO_PI = 2.0 * math.pi


def listed():
    split = dict(partition="gauss", multiplier="ds", width=0, auto_eps=0.0)
    return [
        # the smallest call in earnest: the closed-form check of the paper's first example, FP64 (latency)
        dict(split, name="fp64_solve_128", kind="solve", precision="fp64", nx=128, ny=128, lx=16.0, ly=16.0,
             cut=4.0, n_r=32, n_theta=64, density="gauss1"),
        # one small density in mixed precision: what a parameter scan or an interactive user calls (latency)
        dict(split, name="mixed_solve_256", kind="solve", precision="mixed", nx=256, ny=256, lx=32.0, ly=32.0,
             cut=8.0, n_r=64, n_theta=256, density="sum8"),
        # the ordinary FP64 solve: eight anisotropic Gaussians on 1024^2
        dict(split, name="fp64_solve_1024", kind="solve", precision="fp64", nx=1024, ny=1024, lx=32.0, ly=32.0,
             cut=8.0, n_r=64, n_theta=256, density="sum8"),
        # a rectangle chosen by the automatic parameters (Gauss-Jacobi radial rule), FP64
        dict(split, name="fp64_auto_1024x256", kind="solve", precision="fp64", nx=1024, ny=256, lx=24.0, ly=10.0,
             cut=0.0, n_r=0, n_theta=0, density="sum8", auto_eps=1e-10),
        # the benchmark workload, mixed precision: rho = |u|^2 of 16 complex Gaussians on 4096^2
        dict(split, name="mixed_solve_4096", kind="solve", precision="mixed", nx=4096, ny=4096, lx=64.0, ly=64.0,
             cut=8.0, n_r=64, n_theta=256, density="abs16"),
        # the same density through the FP64 solver (the largest call)
        dict(split, name="fp64_solve_4096", kind="solve", precision="fp64", nx=4096, ny=4096, lx=64.0, ly=64.0,
             cut=8.0, n_r=64, n_theta=256, density="abs16"),
        # another multiplier (2D Coulomb, 2 pi/|k|) on a long rectangle with uneven node counts
        dict(split, name="mixed_coulomb_2048x512", kind="solve", precision="mixed", nx=2048, ny=512, lx=40.0,
             ly=12.0, cut=7.3, n_r=51, n_theta=226, density="sum8", multiplier="coulomb"),
        # the standard periodic FFT solver that the method is compared with, mixed precision
        dict(split, name="mixed_standard_2048", kind="solve", precision="mixed", nx=2048, ny=2048, lx=32.0,
             ly=32.0, cut=0.0, n_r=0, n_theta=0, density="sum8", partition="none"),
        # differentiation of a loss on Phi(|u|^2) in complex128 at 1024^2: a forward and a backward solve
        dict(split, name="c128_grad_1024", kind="grad", precision="fp64", nx=1024, ny=1024, lx=32.0, ly=32.0,
             cut=8.0, n_r=64, n_theta=256),
        # a differentiated Strang loop in complex64 at 1024^2, checkpointed every two steps
        dict(split, name="c64_strang_grad_1024", kind="evolve", precision="mixed", nx=1024, ny=1024, lx=32.0,
             ly=32.0, cut=8.0, n_r=64, n_theta=256, scheme="strang", steps=4, checkpoint=2, grad=True, tau=1e-3,
             alpha=1.0, beta=1.0),
        # fourth-order (Yoshida) time steps in complex128, forward only: the loop of the paper's moving lump
        dict(split, name="c128_yoshida_512", kind="evolve", precision="fp64", nx=512, ny=512, lx=32.0, ly=32.0,
             cut=2.25, n_r=64, n_theta=128, scheme="yoshida", steps=2, checkpoint=0, grad=False, tau=1e-3,
             alpha=1.0, beta=-1.0),
        # throughput over uneven densities: 64 members on 256^2 .. 2048^2, one captured graph
        dict(split, name="mixed_batch_64", kind="batch", precision="mixed", members=64, mix=5, smallest=256,
             largest=2048, lx=32.0, ly=32.0, cut=8.0, n_r=64, n_theta=256),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def _polar(rng, nx, ny, width):
    """A domain and a polar rule whose disk (with the ES stencil) fits the padded grid."""
    n = min(nx, ny)
    lx = round(math.exp(rng.uniform(math.log(8.0), math.log(64.0))), 3)
    ly = round(lx * rng.uniform(0.7, 1.4) * (1.0 if ny >= nx / 2 else 0.5), 3)
    h = 2.0 * max(lx / nx, ly / ny)
    # P h + w pi/(2 n) < pi, and no more than what the densities reach
    top = min(8.0, 0.8 * (math.pi - 16 * math.pi / (2.0 * n)) / h)
    cut = round(rng.uniform(0.5, 1.0) * top, 3)
    return dict(lx=lx, ly=ly, cut=cut, n_r=rng.randint(20, 64), n_theta=2 * rng.randint(24, 128), width=width)


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "solve", "grad", "evolve", "batch"))
    precision = rng.choice(("mixed", "mixed", "fp64"))
    case = dict(kind=kind, precision=precision, partition="gauss", multiplier="ds", auto_eps=0.0)
    if kind == "batch":
        low = _pow2(rng, 128, 512)
        case.update(members=rng.randint(3, 40), mix=rng.randint(1, 10**6), smallest=low,
                    largest=min(2048, low * _pow2(rng, 2, 8)), lx=round(rng.uniform(8.0, 20.0), 3),
                    ly=round(rng.uniform(8.0, 20.0), 3), cut=0.0, n_r=rng.randint(20, 64),
                    n_theta=2 * rng.randint(24, 128), width=0)
        h = 2.0 * max(case["lx"], case["ly"]) / low
        case["cut"] = round(min(8.0, 0.6 * (math.pi - 8 * math.pi / low) / h), 3)
        if precision == "fp64":
            case["largest"] = min(case["largest"], 1024)
        return case
    largest = {"solve": 4096, "grad": 2048, "evolve": 1024}[kind]
    if precision == "fp64" and kind != "solve":
        largest //= 2
    nx = _pow2(rng, 64, largest)
    ny = max(64, min(largest, int(nx * 2.0 ** rng.randint(-2, 2))))
    width = rng.choice((0, 0, 0, 6, 7) if precision == "mixed" else (0, 0, 0, 13, 14))
    case.update(nx=nx, ny=ny, **_polar(rng, nx, ny, width))
    if kind == "solve":
        case["density"] = rng.choice(("gauss1", "sum8", "abs16"))
        what = rng.random()
        if what < 0.2:
            case.update(partition="none", cut=0.0, n_r=0, n_theta=0)
        elif what < 0.35:
            case["multiplier"] = rng.choice(("coulomb", "rotated"))
        elif what < 0.45:
            case["partition"] = "sharp"
    elif kind == "evolve":
        case.update(scheme=rng.choice(("strang", "yoshida")), steps=rng.randint(1, 3), checkpoint=0, grad=False,
                    tau=round(math.exp(rng.uniform(math.log(2e-4), math.log(5e-3))), 7), alpha=1.0,
                    beta=rng.choice((-1.0, 1.0)))
        if rng.random() < 0.5:
            case.update(grad=True, checkpoint=rng.choice((0, 1, 2)))
    return case


# --------------------------------------------------------------------------- inputs

_MULT = {"coulomb": (-1, TWO_PI, 0.0, 0.0), "rotated": (0, -0.5, -0.3, 0.4)}


def _axis(n, half, device):
    return -half + (2.0 * half / n) * torch.arange(n, dtype=torch.float64, device=device)


def _gaussians(nx, ny, lx, ly, seed, count, complex_valued=False, device="cuda"):
    """sum_k A_k e^{i phi_k} of axis-aligned Gaussians: centres U[-4, 4]^2, widths U[0.5, 2], amplitudes
    U[0.5, 1.5], phases U[0, 2 pi) (centres drawn closer in on domains narrower than 24)."""
    rng = random.Random(seed)
    c = min(4.0, min(lx, ly) / 3.0)
    cx, cy, sx, sy, amp, ph = ([rng.uniform(*r) for _ in range(count)] for r in (
        (-c, c), (-c, c), (0.5, 2.0), (0.5, 2.0), (0.5, 1.5), (0.0, TWO_PI)))

    def t(v):
        return torch.tensor(v, dtype=torch.float64, device=device)[:, None]

    gx = torch.exp(-((_axis(nx, lx, device)[None] - t(cx)) ** 2) / (2.0 * t(sx) ** 2))
    gy = torch.exp(-((_axis(ny, ly, device)[None] - t(cy)) ** 2) / (2.0 * t(sy) ** 2))
    if not complex_valued:
        return (gy * t(amp)).T.contiguous() @ gx
    re = (gy * t(amp) * torch.cos(t(ph))).T.contiguous() @ gx
    im = (gy * t(amp) * torch.sin(t(ph))).T.contiguous() @ gx
    return torch.complex(re, im)


def _density(what, nx, ny, lx, ly, seed, device="cuda"):
    if what == "gauss1":  # one isotropic Gaussian near the origin
        return _gaussians(nx, ny, lx, ly, seed, 1, device=device)
    if what == "sum8":
        return _gaussians(nx, ny, lx, ly, seed, 8, device=device)
    u = _gaussians(nx, ny, lx, ly, seed, 16, complex_valued=True, device=device)
    return u.real * u.real + u.imag * u.imag


def _normal(shape, seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return torch.randn(shape, dtype=torch.float64, generator=g, device=device)


def _members(case):
    rng = random.Random(case["mix"])
    sizes = [1 << k for k in range(int(math.log2(case["smallest"])), int(math.log2(case["largest"])) + 1)]
    return [(rng.choice(sizes), rng.randint(4, 16)) for _ in range(case["members"])]


def _member_density(case, i, n, count, seed):
    return _gaussians(n, n, case["lx"], case["ly"], seed * 1000 + i, count)


def _field(case, seed):
    """The complex field and the real loss weights / cotangent of a wave case, in 64 bits."""
    nx, ny = case["nx"], case["ny"]
    u = _gaussians(nx, ny, case["lx"], case["ly"], seed, 16, complex_valued=True)
    if case["precision"] == "mixed":
        u = u.to(torch.complex64)
    if case["kind"] == "grad":
        return u, _normal((ny, nx), seed + 1)
    g = torch.complex(_normal((ny, nx), seed + 1), _normal((ny, nx), seed + 2))
    return u, g.to(u.dtype)


def _plan(case, nx, ny):
    if case["auto_eps"] > 0.0:
        return Plan.auto(nx, ny, case["lx"], case["ly"], eps=case["auto_eps"], precision=case["precision"])
    if case["partition"] == "none":
        return Plan(nx, ny, case["lx"], case["ly"], precision=case["precision"], partition="none",
                    multiplier=_MULT.get(case["multiplier"]))
    return Plan(nx, ny, case["lx"], case["ly"], cut_radius=case["cut"], n_r=case["n_r"], n_theta=case["n_theta"],
                kernel_width=case["width"], precision=case["precision"], partition=case["partition"],
                multiplier=_MULT.get(case["multiplier"]))


def prepare(case, seed):
    state = dict(case=case)
    if case["kind"] == "batch":
        members = _members(case)
        plans = {n: _plan(case, n, n) for n in sorted({n for n, _ in members})}
        # the potentials side by side in one allocation, as a program that post-processes them together has them
        flat = torch.empty(sum(n * n for n, _ in members), dtype=torch.float64, device="cuda")
        rhos, phis, at = [], [], 0
        for i, (n, count) in enumerate(members):
            rhos.append(_member_density(case, i, n, count, seed))
            phis.append(flat[at:at + n * n].view(n, n))
            at += n * n
        batch = Batch([plans[n] for n, _ in members], rhos, phis)
        batch.capture_graph()
        state.update(plans=plans, batch=batch, flat=flat)
        return state
    nx, ny = case["nx"], case["ny"]
    state["plan"] = _plan(case, nx, ny)
    if case["kind"] == "solve":
        state["rho"] = _density(case["density"], nx, ny, case["lx"], case["ly"], seed)
        state["phi"] = torch.empty_like(state["rho"])
        return state
    state["ds"] = DSPlan(nx, ny, case["lx"], case["ly"], precision=case["precision"])
    u, g = _field(case, seed)
    state["u"] = u.requires_grad_(case["kind"] == "grad" or case["grad"])
    state["g"] = g
    return state


def run(state):
    case = state["case"]
    mixed = case["precision"] == "mixed"
    if case["kind"] == "batch":
        state["batch"].solve()
        return state["flat"].float() if mixed else state["flat"]
    if case["kind"] == "solve":
        phi = state["plan"].solve(state["rho"], out=state["phi"])
        return phi.float() if mixed else phi
    u, g = state["u"], state["g"]
    if case["kind"] == "grad":
        phi = potential_of_wave(u, state["ds"], state["plan"])
        grad, = torch.autograd.grad(phi, u, g)
        return [phi.detach().float() if mixed else phi.detach(), grad]
    v = evolve(u, case["steps"], state["ds"], state["plan"], case["tau"], case["alpha"], case["beta"],
               checkpoint_every=case["checkpoint"], scheme=case["scheme"])
    if not case["grad"]:
        return v
    grad, = torch.autograd.grad(v, u, g)
    return [v.detach(), grad]


# --------------------------------------------------------------------------- compulsory work

def _solve_flops(case, nx, ny):
    """One solve by the method: a forward and an inverse real transform of the padded grid (2.5 M log2 M each),
    the multiplier, and both stencil sums of the polar nodes (a multiply-add per real component and point)."""
    pad = 1 if case["partition"] == "none" else 2
    m = pad * pad * nx * ny
    flops = 2 * 2.5 * m * math.log2(m) + 2.0 * m
    nodes = case["n_r"] * case["n_theta"]
    if case["auto_eps"] > 0.0:
        p = _auto_polar(case)
        nodes = p["n_r"] * p["n_theta"]
    w = case["width"] or (15 if case["precision"] == "fp64" else 8)
    return flops + 2 * nodes * w * w * 4.0


def work(case):
    out = 4 if case["precision"] == "mixed" else 8  # the potential
    c = 2 * out                                     # a complex field
    if case["kind"] == "batch":
        ns = [n for n, _ in _members(case)]
        return {"bytes": sum((8.0 + out) * n * n for n in ns), "flops": sum(_solve_flops(case, n, n) for n in ns)}
    n = float(case["nx"] * case["ny"])
    one = _solve_flops(case, case["nx"], case["ny"])
    if case["kind"] == "solve":
        return {"bytes": (8.0 + out) * n, "flops": one}
    if case["kind"] == "grad":  # u and w in; Phi and the gradient out
        return {"bytes": (c + 8.0 + out + c) * n, "flops": 2 * one + 8 * n}
    linear, nonlinear = (2, 1) if case["scheme"] == "strang" else (4, 3)
    step = linear * (2 * 5.0 * n * math.log2(n) + 8 * n) + nonlinear * (one + 20 * n)
    return {"bytes": (2 + (2 if case["grad"] else 0)) * c * n, "flops": case["steps"] * step * (2 if case["grad"] else 1)}


# --------------------------------------------------------------------------- the results in 64 bits

def _legendre(n, cut):
    t, v = np.polynomial.legendre.leggauss(n)
    r = 0.5 * cut * (t + 1.0)
    return r, r * (0.5 * cut * v)


def _jacobi01(n, cut):
    """Gauss rule for the weight 1 + t on [-1, 1] (Golub-Welsch)."""
    k = np.arange(n, dtype=np.float64)
    a = 1.0 / ((2 * k + 1) * (2 * k + 3))
    k = k[1:]
    b = np.sqrt(4 * k * (k + 1) * k * (k + 1) / ((2 * k + 1) ** 2 * (2 * k + 2) * 2 * k))
    t, q = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
    return 0.5 * cut * (t + 1.0), (0.5 * cut) ** 2 * 2.0 * q[0] ** 2


def _auto_polar(case):
    """The automatic parameters, from their published rule (sigma L = 12, p(P) = eps, node counts from P R)."""
    eps = min(max(case["auto_eps"], 1e-7 if case["precision"] == "mixed" else 1e-15), 1e-2)
    sigma = 12.0 / min(case["lx"], case["ly"])
    cut = sigma * math.sqrt(math.log(1.0 / eps))
    cr = cut * math.hypot(case["lx"], case["ly"])
    return dict(sigma=sigma, cut=cut, n_theta=4 * math.ceil((cr + 16.0) / 4.0), n_r=8 * math.ceil((0.5 * cr + 4.0) / 8.0))


class _Exact:
    """Phi = A rho in 64 bits by plain torch: the padded FFT with the multiplier outside the disk plus the
    direct nonuniform sums of the polar quadrature (differentiable)."""

    def __init__(self, case, nx, ny):
        self.nx, self.ny = nx, ny
        lx, ly = case["lx"], case["ly"]
        self.pad = 1 if case["partition"] == "none" else 2
        mult = _MULT.get(case["multiplier"], (0, -0.5, -0.5, 0.0))
        hx, hy = 2.0 * lx / nx, 2.0 * ly / ny
        dev = "cuda"
        wx = TWO_PI * torch.fft.rfftfreq(self.pad * nx, d=hx, dtype=torch.float64, device=dev)[None, :]
        wy = TWO_PI * torch.fft.fftfreq(self.pad * ny, d=hy, dtype=torch.float64, device=dev)[:, None]
        w2 = wx * wx + wy * wy
        safe = torch.where(w2 > 0, w2, torch.ones_like(w2))
        alpha, a0, ac, as_ = mult
        odd = 2.0 * wx * wy  # averaged over the two aliases at an axis' Nyquist frequency
        odd[:, -1] = 0.0
        odd[(self.pad * ny) // 2, :] = 0.0
        if case["multiplier"] == "ds":
            m = -(wx * wx) / safe
        else:
            m = safe ** (0.5 * alpha) * (a0 + (ac * (wx * wx - wy * wy) + as_ * odd) / safe)
        self.split = case["partition"] != "none"
        if self.split:
            auto = case["auto_eps"] > 0.0
            p = _auto_polar(case) if auto else dict(sigma=case["cut"] / 6.0, cut=case["cut"], n_r=case["n_r"],
                                                    n_theta=case["n_theta"])
            if case["partition"] == "sharp":
                m = m * (w2 > p["cut"] ** 2)
            else:
                m = m * -torch.expm1(-w2 / p["sigma"] ** 2)
            r, wr = (_jacobi01 if auto else _legendre)(p["n_r"], p["cut"])
            # the rule is symmetric under k -> -k and rho is real: half the angles, doubled
            th = TWO_PI * np.arange(p["n_theta"] // 2) / p["n_theta"]
            rad = wr * r ** float(alpha) * (1.0 if case["partition"] == "sharp" else np.exp(-(r / p["sigma"]) ** 2))
            ang = a0 + ac * np.cos(2 * th) + as_ * np.sin(2 * th)
            d = 2.0 * np.outer(rad, ang) * (TWO_PI / p["n_theta"]) / TWO_PI**2 * hx * hy

            def t(v):
                return torch.from_numpy(np.ascontiguousarray(v.ravel())).to(dev)

            self.d, self.kx, self.ky = t(d), t(np.outer(r, np.cos(th))), t(np.outer(r, np.sin(th)))
            self.x, self.y = _axis(nx, lx, dev), _axis(ny, ly, dev)
        self.m = torch.where(w2 > 0, m, torch.zeros_like(m))

    def __call__(self, rho):
        s = (self.pad * self.ny, self.pad * self.nx)
        phi = torch.fft.irfft2(self.m * torch.fft.rfft2(rho, s=s), s=s)[:self.ny, :self.nx]
        if not self.split:
            return phi.contiguous()
        step = max(1, (1 << 24) // max(self.nx, self.ny))
        for at in range(0, self.d.numel(), step):
            kx, ky, d = (v[at:at + step, None] for v in (self.kx, self.ky, self.d))
            ax, ay = kx * self.x, ky * self.y
            cx, sx, cy, sy = torch.cos(ax), torch.sin(ax), torch.cos(ay), torch.sin(ay)
            ic, is_ = (rho @ cx.T).T, (rho @ sx.T).T          # sum over x of rho cos, rho sin
            re = d * (cy * ic - sy * is_).sum(1, keepdim=True)  # D_j rho_hat_j = re - i im
            im = d * (cy * is_ + sy * ic).sum(1, keepdim=True)
            phi = phi + (re * cy + im * sy).T @ cx + (im * cy - re * sy).T @ sx
        return phi


def _exact_evolve(case, u, solve):
    nx, ny = case["nx"], case["ny"]
    kx = TWO_PI * torch.fft.fftfreq(nx, d=2.0 * case["lx"] / nx, dtype=torch.float64, device="cuda")[None, :]
    ky = TWO_PI * torch.fft.fftfreq(ny, d=2.0 * case["ly"] / ny, dtype=torch.float64, device="cuda")[:, None]
    k2 = kx * kx - case["alpha"] * ky * ky

    def linear(v, tau):
        return torch.fft.ifft2(torch.fft.fft2(v) * torch.exp(-1j * tau * k2))

    def nonlinear(v, tau):
        rho = v.real * v.real + v.imag * v.imag
        return v * torch.exp(1j * tau * case["beta"] * (2.0 * rho + 4.0 * solve(rho)))

    tau = case["tau"]
    for _ in range(case["steps"]):
        if case["scheme"] == "strang":
            u = linear(nonlinear(linear(u, 0.5 * tau), tau), 0.5 * tau)
            continue
        c = 2.0 ** (1.0 / 3.0)
        b3 = 1.0 / (2.0 - c)
        b2 = -c * b3
        u = linear(u, 0.5 * b3 * tau)
        u = linear(nonlinear(u, b3 * tau), 0.5 * (b3 + b2) * tau)
        u = linear(nonlinear(u, b2 * tau), 0.5 * (b3 + b2) * tau)
        u = linear(nonlinear(u, b3 * tau), 0.5 * b3 * tau)
    return u


def exact(case, seed):
    if case["kind"] == "batch":
        members = _members(case)
        solvers = {n: _Exact(case, n, n) for n in {n for n, _ in members}}
        out = [solvers[n](_member_density(case, i, n, count, seed)).reshape(-1) for i, (n, count) in enumerate(members)]
        return torch.cat(out)
    nx, ny = case["nx"], case["ny"]
    solve = _Exact(case, nx, ny)
    if case["kind"] == "solve":
        return solve(_density(case["density"], nx, ny, case["lx"], case["ly"], seed))
    u, g = _field(case, seed)
    u = u.to(torch.complex128)
    if case["kind"] == "grad":  # the operator is symmetric: its transpose is itself
        rho = u.real * u.real + u.imag * u.imag
        return [solve(rho), 2.0 * solve(g) * u]
    if not case["grad"]:
        return _exact_evolve(case, u, solve)
    u = u.requires_grad_(True)
    v = _exact_evolve(case, u, solve)
    grad, = torch.autograd.grad(v, u, g.to(torch.complex128))
    return [v.detach(), grad]
