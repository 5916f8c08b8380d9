"""The standard solver's widened FP32 outputs in mixed plans and the DS flows
of complex64 fields, over the sizes where their kernels change shape."""

import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

EPS = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2014_gb300.build import build

    build()


@pytest.mark.parametrize("nx,ny", [(16, 16), (64, 16), (16, 128), (2048, 32), (4096, 16)])
def test_standard_outputs_are_widened_exactly(nx, ny):
    """Every value is a float (widening is exact), also zeros and non-finite
    ones, and agrees with the FP64 plan: 2 EPS per level of the four
    transforms and of the multiplier, in the L2 norm."""
    from paper_1409_2014_gb300 import Plan

    g = torch.Generator().manual_seed(nx * 5000 + ny)
    rho = torch.rand(ny, nx, generator=g, dtype=torch.float64).cuda()
    mixed, full = (Plan(nx, ny=ny, lx=8.0, ly=6.0, partition="none", precision=p) for p in ("mixed", "fp64"))
    phi, ref = mixed.solve(rho), full.solve(rho)
    assert torch.equal(phi, phi.float().double())
    tol = 2 * EPS * (2 * math.log2(nx * ny) + 4)
    # (rho's mean is removed by the multiplier: relative to rho's norm, |m| <= 1)
    assert float((phi - ref).norm() / rho.norm()) <= tol
    assert torch.equal(mixed.solve(torch.zeros_like(rho)), torch.zeros_like(rho))
    rho[ny // 2, nx // 3] = math.inf
    assert not bool(torch.isfinite(mixed.solve(rho)).any())


@pytest.mark.parametrize("nx,ny", [(16, 16), (32, 64), (512, 128), (16, 1024), (2048, 64), (4096, 32), (64, 4096)])
def test_complex64_flows_match_numpy(nx, ny):
    """Linear and nonlinear flow of a complex64 field against 64 bits, in place
    and into a new tensor (bitwise the same, the input unchanged)."""
    from paper_1409_2014_gb300.ds import DSPlan

    rng = np.random.default_rng(nx + ny)
    u = (rng.standard_normal((ny, nx)) + 1j * rng.standard_normal((ny, nx))).astype(np.complex64)
    lx, ly, tau, alpha, beta = 5.0, 7.0, 3e-3, 0.7, 1.3
    ds = DSPlan(nx, ny, lx, ly, precision="mixed")
    ds.set_linear_step(tau, alpha)
    t = torch.from_numpy(u).cuda()
    kx = 2 * np.pi * np.fft.fftfreq(nx, 2 * lx / nx)
    ky = 2 * np.pi * np.fft.fftfreq(ny, 2 * ly / ny)
    ph = np.exp(-1j * tau * (kx[None, :] ** 2 - alpha * ky[:, None] ** 2))
    for adjoint in (False, True):
        ref = np.fft.ifft2(np.fft.fft2(u.astype(np.complex128)) * (ph.conj() if adjoint else ph))
        out = ds.linear(t, adjoint)
        assert torch.equal(torch.view_as_real(t), torch.view_as_real(torch.from_numpy(u).cuda()))
        err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= 2 * EPS * (2 * math.log2(nx * ny) + 4)  # 2 EPS per level
        assert torch.equal(torch.view_as_real(ds.linear_(t.clone(), adjoint)), torch.view_as_real(out))
    phi = torch.from_numpy(rng.standard_normal((ny, nx))).cuda()
    th = tau * (2 * beta * np.abs(u.astype(np.complex128)) ** 2 + 4 * beta * phi.cpu().numpy())
    ref = u * np.exp(1j * th)
    out = ds.nonlinear(t, phi, tau, beta)
    assert torch.equal(torch.view_as_real(t), torch.view_as_real(torch.from_numpy(u).cuda()))
    # a few roundings of the angle (relative) and of the product
    assert np.abs(out.cpu().numpy() - ref).max() <= 4 * EPS * (np.abs(th).max() + 2) * np.abs(u).max()
    assert torch.equal(torch.view_as_real(ds.nonlinear_(t.clone(), phi, tau, beta)), torch.view_as_real(out))


@pytest.mark.parametrize("multiplier", [None, (0, 0.3, -0.2, 0.4)], ids=["ds", "generic"])
@pytest.mark.parametrize("nx,ny", [(16, 16), (32, 16), (16, 64), (128, 32), (256, 512), (512, 256), (512, 1024), (1024, 64)])
def test_mixed_short_lengths_match_fp64(nx, ny, multiplier):
    """Every CTA shape of the mixed passes, several members of one plan among
    them: within the mixed plans' 2e-5 of the FP64 result."""
    from paper_1409_2014_gb300 import Batch, Plan

    prm = dict(nx=nx, ny=ny, lx=4.0, ly=4.0, cut_radius=2.0, n_r=12, n_theta=24, multiplier=multiplier)
    rho = torch.from_numpy(np.random.default_rng(nx * ny).standard_normal((3, ny, nx))).cuda()
    mixed, full = Plan(precision="mixed", **prm), Plan(precision="fp64", **prm)
    phi = torch.stack([mixed.solve(r) for r in rho])
    ref = torch.stack([full.solve(r) for r in rho])
    assert float((phi - ref).abs().max() / ref.abs().max()) <= 2e-5
    ref = full.solve_adjoint(rho[0])
    assert float((mixed.solve_adjoint(rho[0]) - ref).abs().max() / ref.abs().max()) <= 2e-5
    out = [torch.empty_like(r) for r in rho]
    Batch([mixed] * 3, list(rho), out).solve()
    torch.cuda.synchronize()
    assert torch.equal(torch.stack(out), phi)
