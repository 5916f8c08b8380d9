"""dsnu_solve_noalloc at the limit of its 32 MiB: an FP64 plan whose spectra,
band and node values fit is taken, although its workspace with the exponents
of its rows and columns is larger."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LIMIT = 32 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2014_gb300.build import build

    build()


def _exponents(nx, ny, q):
    return sum((4 * k + 255) & ~255 for k in (ny, ny, nx + 1, q + 1))


def test_exponents_do_not_count(monkeypatch):
    from paper_1409_2014_gb300 import Plan, _abi

    monkeypatch.setenv("DSNU_SPREAD_CFG", "0")  # (the partial tiles' sizes)
    n = 1024

    def plan(n_r):
        return Plan(n, lx=32.0, cut_radius=19.02, n_r=n_r, n_theta=2, precision="fp64")

    fits, p, big = plan(1024), plan(2592), plan(4096)
    sizes = [_abi.dsnu_workspace_bytes(q.handle) for q in (fits, p, big)]
    exps = [_exponents(n, n, q.info.band_q) for q in (fits, p, big)]
    assert sizes[0] <= LIMIT and sizes[1] - exps[1] <= LIMIT < sizes[1] and sizes[2] - exps[2] > LIMIT
    g = torch.Generator(device="cuda").manual_seed(5)
    rho = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    stream = torch.cuda.current_stream().cuda_stream
    for q in (fits, p):
        out = torch.full_like(rho, float("nan"))
        _abi.dsnu_solve_noalloc(q.handle, rho.data_ptr(), out.data_ptr(), stream)
        assert torch.equal(out, q.solve(rho))
    with pytest.raises(_abi.DsnuError) as e:  # the spectra themselves beyond it: refused as before
        _abi.dsnu_solve_noalloc(big.handle, rho.data_ptr(), out.data_ptr(), stream)
    assert e.value.status == _abi.DSNU_EINVAL
    for q in (p, fits, big):
        q.close()
