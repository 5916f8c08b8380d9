"""The band chain and the column pass side by side, in both arrangements (the
column pass on the side stream below 2048 in either axis, the band chain from
2048 x 2048), against the same plan in line: bit for bit, for runs of solves
with changing inputs and no wait between them, on two streams in turn, and
from a captured graph."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GRIDS = [(16, 64), (128, 128), (512, 1024), (2048, 512), (2048, 2048)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2014_gb300.build import build

    build()


@pytest.mark.parametrize("mult", [None, (0, -0.5, -0.3, 0.4)], ids=["ds", "sin2theta"])
@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_side_by_side_equals_in_line(prec, nx, ny, mult, monkeypatch):
    from paper_1409_2014_gb300 import Plan

    monkeypatch.setenv("DSNU_SPREAD_CFG", "0")  # one order of the spreading's sums
    kw = dict(nx=nx, ny=ny, lx=4.0, ly=4.0, cut_radius=2.0, n_r=24, n_theta=96, precision=prec, multiplier=mult)

    def plan(pdl=None, band=None):
        for name, v in (("DSNU_PDL", pdl), ("DSNU_BAND_SMS", band)):
            if v is None:
                monkeypatch.delenv(name, raising=False)
            else:
                monkeypatch.setenv(name, v)
        return Plan(**kw)

    g = torch.Generator(device="cuda").manual_seed(nx + 3 * ny)
    k = 6 if nx * ny > 1 << 20 else 24
    rhos = torch.randn(k, ny, nx, dtype=torch.float64, device="cuda", generator=g)
    rhos *= torch.from_numpy(10.0 ** np.linspace(-3, 3, k)).cuda()[:, None, None]  # changing exponents
    ref_plan = plan("0", "0")
    ref = torch.stack([ref_plan.solve(r) for r in rhos])
    adj = torch.stack([ref_plan.solve_adjoint(r) for r in rhos])
    ref_plan.close()
    for pdl, band in ((None, None), ("0", None), (None, "0"), (None, "24"), ("0", "100"), (None, "151"), (None, "152")):
        p = plan(pdl, band)
        out = torch.full_like(rhos, float("nan"))
        for i in range(k):
            p.solve(rhos[i], out=out[i])
        assert torch.equal(out, ref), (pdl, band)
        for i in range(k):
            p.solve_adjoint(rhos[i], out=out[i])
        assert torch.equal(out, adj), (pdl, band)
        if band is None:
            streams = [torch.cuda.Stream() for _ in range(2)]
            out.fill_(float("nan"))
            torch.cuda.synchronize()
            last = None
            for i in range(k):  # one workspace: each solve after the one before
                with torch.cuda.stream(streams[i % 2]):
                    if last is not None:
                        streams[i % 2].wait_event(last)
                    p.solve(rhos[i], out=out[i])
                    last = torch.cuda.Event()
                    last.record()
            torch.cuda.synchronize()
            assert torch.equal(out, ref), (pdl, "streams")
            x, y = torch.zeros(2, ny, nx, dtype=torch.float64, device="cuda"), torch.empty(2, ny, nx, dtype=torch.float64, device="cuda")
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                for i in range(2):
                    p.solve(x[i], out=y[i])
            for i in range(0, k, 2):
                x.copy_(rhos[i:i + 2])
                graph.replay()
                assert torch.equal(y, ref[i:i + 2]), (pdl, "graph")
            del graph
        assert p.status_poll() == 0
        p.close()
