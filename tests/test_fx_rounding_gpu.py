"""How many bits the fixed-point FP64 passes keep, where no ES kernel hides it.

The standard solver against the same transforms in long double (extended or
quadruple precision), relative to ||rho|| max |m| in the L2 norm.  Every stage
rounds to at most 2^-56 of its block's largest component, product and dropped
terms together 3/4 of that at most: 0.6 x 2^-56 c in the norm, c the ratio of
the largest component to the root mean square of the complex values.  Two
transforms of two passes have at most 4 ceil(12/3) + 10 such roundings, which
add up as their root, 5.1: 4.3e-17 c, and the result's own rounding 0.3 eps.
Noise has c <= 4.5 (1.2 eps in all); a blob has c <= 9 in most of its blocks, of
either width in space or frequency (2.1 eps), and in its spectrum at length 4096,
which two roundings see, 29.  Asked are 2 and 4 eps.  (A multiplication whose
rounding follows the multiplier's bound instead of its products gave 5.1 for the
half Laplacian of the blob at length 4096.)

The split solver with the widest ES kernel (w = 16: error exp(-pi w sqrt(1/2)) =
4e-16, ten times that at most by its constants, in each of the two nonuniform
sums) against the direct sums: 1e-14 in the L2 norm."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

EPS = float(np.finfo(np.float64).eps)
LX, LY = 4.0, 5.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2014_gb300.build import build

    build()


def _solve(rho, multiplier, **prm):
    from paper_1409_2014_gb300 import Plan

    plan = Plan(precision="fp64", multiplier=multiplier, **prm)
    out = plan.solve(torch.from_numpy(np.ascontiguousarray(rho)).cuda()).cpu().numpy()
    plan.close()
    return out


def _density(kind, nx, ny):
    if kind == "noise":
        return synth.normal_field(nx, ny, seed=nx + 7 * ny)
    x = (np.arange(nx) - nx / 2) / nx
    y = (np.arange(ny) - ny / 2) / ny
    return np.exp(-((x - 0.1)[None] ** 2 + (y + 0.05)[:, None] ** 2) / (2 * 0.06 ** 2))


def _reference(rho, multiplier):
    """F^-1 m F rho in long double, and max |m|: m(0) = 0, the sin 2theta term dropped at the Nyquist frequencies."""
    ld = np.longdouble
    ny, nx = rho.shape
    pi = ld(4) * np.arctan(ld(1))
    qx, qy = (np.fft.fftfreq(n, 1.0 / n).astype(ld) for n in (nx, ny))
    kx, ky = (pi / ld(LX) * qx)[None], (pi / ld(LY) * qy)[:, None]
    sx, sy = kx * (np.abs(qx) != nx // 2)[None], ky * (np.abs(qy) != ny // 2)[:, None]
    k2 = kx * kx + ky * ky
    k2[0, 0] = 1
    alpha, a0, ac, as_ = multiplier
    m = (ld(a0) + (ld(ac) * (kx * kx - ky * ky) + 2 * ld(as_) * sx * sy) / k2) * np.sqrt(k2) ** alpha
    m[0, 0] = 0
    spec = np.fft.fft2(rho.astype(ld))
    assert spec.dtype == np.clongdouble
    return np.fft.ifft2(spec * m).real, float(np.abs(m).max())


@pytest.mark.parametrize("kind,tol", [("noise", 2 * EPS), ("blob", 4 * EPS)])
@pytest.mark.parametrize("mult", [None, (0, -0.5, -0.3, 0.4), (1, 1.0, 0.2, -0.5), (-1, 2 * np.pi, 0.0, 0.0)],
                         ids=["ds", "rotated", "abs_k", "coulomb"])
@pytest.mark.parametrize("nx,ny", [(32, 32), (1024, 64), (64, 1024), (2048, 32), (32, 4096), (256, 512)])
def test_standard_solver_keeps_the_bits(nx, ny, mult, kind, tol):
    rho = _density(kind, nx, ny)
    ref, top = _reference(rho, mult or (0, -0.5, -0.5, 0.0))
    out = _solve(rho, mult, nx=nx, ny=ny, lx=LX, ly=LY, partition="none")
    err = np.linalg.norm((out - ref).astype(np.float64)) / (top * np.linalg.norm(rho))
    assert err <= tol, err / EPS


@pytest.mark.parametrize("kind", ["noise", "blob"])
@pytest.mark.parametrize("nx,ny", [(16, 16), (128, 16), (32, 1024), (2048, 16), (32, 4096), (512, 256)])
def test_split_solver_with_the_widest_kernel(nx, ny, kind):
    prm = dict(nx=nx, ny=ny, lx=4.0, ly=4.0, cut_radius=2.0, n_r=12, n_theta=24)
    rho = _density(kind, nx, ny)
    ref = oracle.solve(rho, oracle.OracleParams(**prm))
    out = _solve(rho, None, kernel_width=16, **prm)
    err = np.linalg.norm(out - ref) / np.linalg.norm(ref)
    assert err <= 1e-14, err
