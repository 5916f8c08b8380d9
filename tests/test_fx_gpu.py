"""The fixed-point FFT passes of the FP64 plans against the FP64 oracle: every
transform length 16 .. 4096 on either axis, inputs that stretch the block
scaling (noise, single points, a constant, rows of very different size), the
multipliers with and without a sin 2theta term; special values; scaling by a
power of two, which only moves exponents; members of very different size in
one batch.  Tolerance: the FP64 plans' relative L-infinity bound 1e-12 (ES
width-15 error about 1e-14 plus rounding)."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-12
GRIDS = [(16, 16), (32, 64), (128, 16), (16, 256), (512, 32), (32, 1024), (2048, 16), (16, 2048), (4096, 32), (32, 4096)]
DS = (0, -0.5, -0.5, 0.0)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2014_gb300.build import build

    build()


def _params(nx, ny, **kw):  # a disk whose stencils fit 16 points per axis
    return dict(nx=nx, ny=ny, lx=4.0, ly=4.0, cut_radius=2.0, n_r=12, n_theta=24, **kw)


def _solve(rho, multiplier=DS, **prm):
    from paper_1409_2014_gb300 import Plan

    plan = Plan(precision="fp64", multiplier=None if multiplier == DS else multiplier, **prm)
    x = torch.from_numpy(np.ascontiguousarray(rho)).cuda()
    phi, adj = plan.solve(x).cpu().numpy(), plan.solve_adjoint(x).cpu().numpy()
    plan.close()
    return phi, adj


def _rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def _field(kind, nx, ny):
    w = synth.normal_field(nx, ny, seed=nx + 3 * ny)
    if kind == "noise":
        return w
    if kind == "rows":  # rows and columns over many orders of magnitude
        g = np.random.Generator(np.random.PCG64(nx * ny))
        return w * 10.0 ** g.uniform(-14, 6, (ny, 1)) * 10.0 ** g.uniform(-6, 3, (1, nx))
    if kind == "points":
        f = np.zeros((ny, nx))
        f[0, 0], f[ny - 1, nx // 2], f[ny // 2, nx - 1] = 1.0, -0.3, 1e-9
        return f
    return np.full((ny, nx), -0.7)


@pytest.mark.parametrize("kind", ["noise", "rows", "points", "constant"])
@pytest.mark.parametrize("nx,ny", GRIDS)
def test_every_length_matches_the_oracle(nx, ny, kind):
    prm = _params(nx, ny)
    rho = _field(kind, nx, ny)
    ref = oracle.solve(rho, oracle.OracleParams(**prm))
    phi, adj = _solve(rho, **prm)
    assert _rel(phi, ref) <= TOL
    assert _rel(adj, ref) <= TOL


@pytest.mark.parametrize("mult", [(0, -0.5, -0.3, 0.4), (1, 1.0, 0.2, -0.5), (-1, 2 * np.pi, 0.0, 0.0), (-1, 0.0, 1.0, 0.5),
                                  (0, 0.0, 0.0, 0.0)])
@pytest.mark.parametrize("nx,ny,part", [(64, 16, "gauss"), (16, 512, "gauss"), (256, 128, "sharp")])
def test_multipliers_match_the_oracle(nx, ny, part, mult):
    prm = _params(nx, ny, partition=part)
    rho = _field("noise", nx, ny)
    ref = oracle.solve(rho, oracle.OracleParams(multiplier=mult, **prm))
    phi, _ = _solve(rho, multiplier=mult, **prm)
    assert np.abs(phi - ref).max() <= TOL * max(np.abs(ref).max(), 1e-300)


@pytest.mark.parametrize("nx,ny", [(16, 32), (128, 64), (1024, 16)])
def test_special_values(nx, ny):
    prm = _params(nx, ny)
    rho = _field("noise", nx, ny)
    for v in (np.nan, np.inf, -np.inf):
        bad = rho.copy()
        bad[ny // 3, nx // 2] = v
        assert np.isnan(_solve(bad, **prm)[0]).all()
    assert not _solve(np.zeros_like(rho), **prm)[0].any()
    base = _solve(rho, **prm)[0]
    for k in (-400, 400):  # exponents only: bitwise
        assert np.array_equal(_solve(np.ldexp(rho, k), **prm)[0], np.ldexp(base, k))
    tiny = _solve(np.ldexp(rho, -1040), **prm)[0]  # subnormal inputs and results
    assert np.abs(np.ldexp(tiny, 1040) - base).max() <= 2.0 ** -34 * nx * ny  # quantum 2^-1074


def test_batch_members_keep_their_own_scale():
    from paper_1409_2014_gb300 import Batch, Plan

    prms = [_params(64, 32), _params(32, 256)]
    plans = [Plan(precision="fp64", **p) for p in prms]
    which, scale = [0, 1, 0, 1, 0, 1], [1.0, 1e-30, 1e30, 1.0, 0.0, 1e12]
    rhos = [torch.from_numpy(synth.normal_field(prms[w]["nx"], prms[w]["ny"], seed=i) * s).cuda()
            for i, (w, s) in enumerate(zip(which, scale))]
    phis = [torch.full_like(r, 7.0) for r in rhos]
    b = Batch([plans[w] for w in which], rhos, phis)
    b.solve()
    for w, r, f in zip(which, rhos, phis):
        assert torch.equal(f, plans[w].solve(r))
    b.close()
    for p in plans:
        p.close()


@pytest.mark.parametrize("mult", [DS, (0, -0.5, -0.3, 0.4), (1, 1.0, 0.2, -0.5), (-1, 2 * np.pi, 0.0, 0.0)])
@pytest.mark.parametrize("nx,ny,kind", [(n, m, k) for n, m in GRIDS for k in ("noise", "rows")] + [(64, 512, "points")])
def test_standard_solver_matches_the_oracle(nx, ny, kind, mult):
    rho = _field(kind, nx, ny)
    ref = oracle.standard_fft_solve(rho, 4.0, 5.0, multiplier=mult)
    phi, adj = _solve(rho, multiplier=mult, nx=nx, ny=ny, lx=4.0, ly=5.0, partition="none")
    assert _rel(phi, ref) <= TOL
    assert _rel(adj, ref) <= TOL


@pytest.mark.parametrize("nx,ny", GRIDS)
def test_linear_flow_matches_numpy(nx, ny):
    """u -> F^-1[e^{-i tau (kx^2 - alpha ky^2)} F u] and its inverse.  Tolerance: FP64 rounding of two 2D
    transforms (about 1e-15) plus the phase's own, eps times its largest angle."""
    from paper_1409_2014_gb300.ds import DSPlan

    tau, alpha = 0.7e-3, 1.3
    ds = DSPlan(nx, ny, 4.0, 5.0, precision="fp64")
    for kind in ("noise", "rows", "points"):
        im = synth.normal_field(nx, ny, seed=7) * (1e-3 if kind == "points" else 1.0)
        u = _field(kind, nx, ny) + 1j * im
        kx = 2 * np.pi * np.fft.fftfreq(nx, 8.0 / nx)[None]
        ky = 2 * np.pi * np.fft.fftfreq(ny, 10.0 / ny)[:, None]
        ang = tau * (kx ** 2 - alpha * ky ** 2)
        ref = np.fft.ifft2(np.fft.fft2(u) * np.exp(-1j * ang))
        tol = 1e-14 + 4 * np.finfo(float).eps * np.abs(ang).max()
        ds.set_linear_step(tau, alpha)
        v = ds.linear_(torch.from_numpy(u).cuda())
        assert np.linalg.norm(v.cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
        back = ds.linear_(v, adjoint=True).cpu().numpy()
        assert np.linalg.norm(back - u) <= 2 * tol * np.linalg.norm(u)
    for z in (0.0, np.nan, np.inf):
        w = torch.zeros((ny, nx), dtype=torch.complex128, device="cuda")
        w[1, 2] = z
        w = ds.linear_(w)
        assert bool(torch.isnan(w.real).all()) if z != 0.0 else not bool(w.abs().any())
    ds.close()
