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


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_partly_overlapping_outputs_are_refused(prec):
    """The flows into another buffer take the input's own or a disjoint one, down to neighbouring bytes; what
    overlaps in part (a race between rows) is refused before anything is launched."""
    from paper_1409_2014_gb300 import _abi
    from paper_1409_2014_gb300.ds import DSPlan

    ds = DSPlan(32, 16, 4.0, 4.0, precision=prec)
    ds.set_linear_step(1e-2, 1.0)
    n = 32 * 16
    pool = torch.zeros(4 * n, dtype=ds.cdtype, device="cuda")
    pool[:n] = torch.randn(n, dtype=ds.cdtype, device="cuda")
    before, size = pool.clone(), pool.element_size()
    base, stream = pool.data_ptr(), torch.cuda.current_stream().cuda_stream
    phi = torch.ones(16, 32, dtype=torch.float64, device="cuda")

    def flows(out, phi_ptr=phi.data_ptr()):
        return (lambda: _abi.dsnu_ds_linear_to(ds._h, base, out, 0, stream),
                lambda: _abi.dsnu_ds_nonlinear_to(ds._h, base, phi_ptr, out, 0.1, 1.0, stream))

    refused = [f for e in (1, 32, n - 1) for f in flows(base + e * size)]
    refused.append(flows(base + n * size, base + (2 * n - 2) * size)[1])  # phi's first bytes
    refused.append(flows(base + 3 * n * size, base + 3 * n * size)[1])
    for f in refused:
        with pytest.raises(_abi.DsnuError) as e:
            f()
        assert e.value.status == _abi.DSNU_EINVAL and "overlap" in str(e.value)
    torch.cuda.synchronize()
    assert torch.equal(pool, before)
    for i in (0, 1):
        for out in (base + n * size, base):
            pool.copy_(before)
            flows(out)[i]()
            want = ds.linear(before[:n].view(16, 32)) if i == 0 else ds.nonlinear(before[:n].view(16, 32), phi, 0.1, 1.0)
            at = 0 if out == base else n
            assert torch.equal(pool[at:at + n].view(16, 32), want)
    ds.close()
