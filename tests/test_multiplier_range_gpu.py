"""FP64 plans whose multiplier leaves the FP64 range: an infinite entry makes
every result a NaN, as the product with it does in FP64 arithmetic."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2014_gb300.build import build

    build()


def _solve(part, multiplier, lx=4.0):
    from paper_1409_2014_gb300 import Plan

    kw = dict(partition="none") if part == "none" else dict(partition=part, cut_radius=2.0, n_r=12, n_theta=24)
    plan = Plan(64, 32, lx, lx, precision="fp64", multiplier=multiplier, **kw)
    rho = torch.from_numpy(synth.normal_field(64, 32, seed=3)).cuda()
    out = plan.solve(rho)
    plan.close()
    return out.cpu().numpy()


@pytest.mark.parametrize("part", ["none", "gauss", "sharp"])
@pytest.mark.parametrize("mult", [(0, 1e308, 1e308, 0.0), (0, -1e308, 0.0, 1.7e308), (1, 1.7e308, 0.0, 0.0),
                                  (-1, 1.7e308, 0.0, 0.9e308)])
def test_an_infinite_entry_gives_nans(part, mult):
    assert np.isnan(_solve(part, mult)).all()


def test_wave_numbers_beyond_the_range():
    """k_x^2/|k|^2 is inf/inf there."""
    assert np.isnan(_solve("none", None, lx=1e-155)).all()
    assert np.isnan(_solve("none", (0, -0.5, -0.5, 0.0), lx=1e-155)).all()
