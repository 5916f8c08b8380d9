"""The DS time loop on the GPU: lazily conjugated fields and cotangents give
the bits of the resolved ones, checkpoints those of the loop without them."""

import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N, L, TAU = 64, 8.0, 1e-2


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2014_gb300.build import build

    build()


@pytest.fixture(params=["fp64", "mixed"])
def loop(request):
    """(field(seed), the arguments of the loop after the field and the steps)"""
    from paper_1409_2014_gb300 import Plan
    from paper_1409_2014_gb300.ds import DSPlan

    cdt = torch.complex128 if request.param == "fp64" else torch.complex64

    def field(seed):
        return torch.complex(*(torch.from_numpy(synth.normal_field(N, N, seed=seed + i)) for i in (0, 50))).to(cdt).cuda()

    ds = DSPlan(N, N, L, L, precision=request.param)
    plan = Plan(N, lx=L, cut_radius=5.0, n_r=16, n_theta=48, precision=request.param)
    yield field, (ds, plan, TAU, 1.0, 1.0)
    ds.close()
    plan.close()


@pytest.mark.parametrize("scheme,ck", [("strang", 0), ("strang", 2), ("yoshida", 0)])
def test_lazily_conjugated_fields_and_cotangents(loop, scheme, ck):
    from paper_1409_2014_gb300.ds import evolve

    field, a = loop
    u, w = field(1), field(2)

    def run(x):
        return evolve(x, 3, *a, checkpoint_every=ck, scheme=scheme)

    assert torch.equal(run(u.conj()), run(u.conj().resolve_conj()))
    x = u.clone().requires_grad_(True)
    got, = torch.autograd.grad(run(x), x, w.conj())
    ref, = torch.autograd.grad(run(x), x, w.conj().resolve_conj())
    assert torch.equal(got, ref)


def test_overlap_loss_equals_its_real_form(loop):
    """|<v, w>| by complex operations (a lazily conjugated cotangent) and by real ones: the cotangents agree
    to a few roundings of the two sums' order, the linear map of both is the same."""
    from paper_1409_2014_gb300.ds import evolve

    field, a = loop
    u, w = field(3), field(4)
    eps = torch.finfo(u.real.dtype).eps

    def grad(loss):
        x = u.clone().requires_grad_(True)
        return torch.autograd.grad(loss(evolve(x, 2, *a)), x)[0]

    def real_form(v):
        (vr, vi), (wr, wi) = torch.view_as_real(v).unbind(-1), torch.view_as_real(w).unbind(-1)
        return torch.hypot((vr * wr + vi * wi).sum(), (vr * wi - vi * wr).sum())

    got, ref = grad(lambda v: (v.conj() * w).sum().abs()), grad(real_form)
    # sums of N^2 terms in another order: sqrt(N^2) roundings of their norm against |<v, w>| of that size
    assert float((got - ref).norm()) <= 16 * N * eps * float(ref.norm())


@pytest.mark.parametrize("scheme", ["strang", "yoshida"])
def test_checkpoints_do_not_change_a_bit(loop, scheme):
    from paper_1409_2014_gb300.ds import evolve

    field, a = loop

    def run(every):
        x = field(5).requires_grad_(True)
        v = evolve(x, 5, *a, checkpoint_every=every, scheme=scheme)
        return v.detach(), torch.autograd.grad(v, x, field(6))[0]

    ref = run(0)
    for every in (1, 2, 3, 5):
        assert all(torch.equal(p, q) for p, q in zip(run(every), ref))
