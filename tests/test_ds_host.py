"""Host side of the DS time loop (CPU): what reaches the library's entry points.

The entry points are replaced by functions that read and write raw memory, as
the library does: they see a tensor's memory and nothing else."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1409_2014_gb300 import ds as D  # noqa: E402

NY, NX = 4, 8


def _mem(ptr, dtype):
    n = NY * NX * np.dtype(dtype).itemsize
    return np.frombuffer((ctypes.c_char * n).from_address(ptr), dtype=dtype)


class _Solver:
    """Phi = A rho with a diagonal A, from and to memory."""

    weight = np.linspace(0.5, 2.0, NY * NX)

    def solve(self, x, out=None):
        assert x.is_contiguous()
        out = torch.empty_like(x)
        _mem(out.data_ptr(), np.float64)[:] = self.weight * _mem(x.data_ptr(), np.float64)
        return out

    solve_adjoint = solve


@pytest.fixture()
def loop(monkeypatch):
    """(ds, solver, log): a plan on the CPU; log holds the flows' steps in the order they ran."""
    log, state = [], {}
    c128 = np.complex128

    def step(h, tau, alpha, stream=0):
        state["tau"] = tau

    def linear_to(h, u, out, adjoint, stream=0):
        log.append(("linear", state["tau"], adjoint))
        ph = np.exp(-1j * state["tau"] * np.arange(NY * NX))
        _mem(out, c128)[:] = _mem(u, c128) * (ph.conj() if adjoint else ph)

    def angle(u, phi, tau, beta):
        return np.exp(1j * tau * (2 * beta * np.abs(_mem(u, c128)) ** 2 + 4 * beta * _mem(phi, np.float64)))

    def nonlinear_to(h, u, phi, out, tau, beta, stream=0):
        log.append(("nonlinear", tau, 0))
        _mem(out, c128)[:] = _mem(u, c128) * angle(u, phi, tau, beta)

    def abs2(h, u, rho, stream=0):
        _mem(rho, np.float64)[:] = np.abs(_mem(u, c128)) ** 2

    def abs2_vjp(h, u, g, grad, stream=0):
        _mem(grad, c128)[:] = 2 * _mem(g, np.float64) * _mem(u, c128)

    def vjp(h, u, phi, g, tau, beta, s, part, stream=0):
        e = angle(u, phi, tau, beta)
        _mem(part, c128)[:] = _mem(g, c128) * e.conj()
        _mem(s, np.float64)[:] = (_mem(g, c128) * (_mem(u, c128) * e).conj()).imag

    def finish(h, u, s, ats, tau, beta, grad, stream=0):
        w = 2 * tau * (2 * beta * _mem(s, np.float64) + 4 * beta * _mem(ats, np.float64))
        _mem(grad, c128)[:] += w * _mem(u, c128)

    for name, fn in (("set_linear_step", step), ("linear_to", linear_to), ("nonlinear_to", nonlinear_to),
                     ("linear", lambda h, u, adj, stream=0: linear_to(h, u, u, adj)),
                     ("nonlinear", lambda h, u, phi, tau, beta, stream=0: nonlinear_to(h, u, phi, u, tau, beta)),
                     ("abs2", abs2), ("abs2_vjp", abs2_vjp), ("nonlinear_vjp", vjp), ("nonlinear_vjp_finish", finish)):
        monkeypatch.setattr(D._abi, "dsnu_ds_" + name, fn)
    monkeypatch.setattr(D, "_stream", lambda device: 0)
    ds = D.DSPlan.__new__(D.DSPlan)
    ds.device, ds.shape, ds.precision, ds.cdtype, ds._h = torch.device("cpu"), (NY, NX), "fp64", torch.complex128, None
    return ds, _Solver(), log


def _field(seed, real=False):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(NY, NX, generator=g, dtype=torch.float64 if real else torch.complex128)


def _lazy(t):
    """The same values behind a lazy conjugate (complex) or negation (real)."""
    v = t.conj().resolve_conj().conj() if t.is_complex() else torch._neg_view(-t)
    assert (v.is_conj() if t.is_complex() else v.is_neg()) and v.is_contiguous() and torch.equal(v, t)
    return v


def _calls(ds, solver):
    a = (ds, solver, 0.02, 1.0, -1.0)
    return {
        "strang": lambda u: D.evolve(u, 2, *a), "strang checkpointed": lambda u: D.evolve(u, 2, *a, checkpoint_every=1),
        "yoshida": lambda u: D.evolve(u, 1, *a, scheme="yoshida"), "strang_step": lambda u: D.strang_step(u, *a),
        "yoshida_step": lambda u: D.yoshida_step(u, *a), "linear": lambda u: D.LinearFlow.apply(u, ds, 0.02, 1.0),
        "nonlinear": lambda u: D.NonlinearFlow.apply(u, ds, solver, 0.02, -1.0),
        "potential_of_wave": lambda u: D.potential_of_wave(u, ds, solver)}


@pytest.mark.parametrize("name", _calls(None, None))
def test_lazily_conjugated_fields_and_cotangents(loop, name):
    fn = _calls(*loop[:2])[name]
    u = _field(1)
    assert torch.equal(fn(_lazy(u)), fn(u))
    x = u.clone().requires_grad_(True)
    v = fn(x)
    w = _field(2, real=not v.is_complex())
    ref, = torch.autograd.grad(v, x, w, retain_graph=True)
    assert torch.equal(torch.autograd.grad(v, x, _lazy(w))[0], ref)
    y = u.conj().resolve_conj().requires_grad_(True)  # the field a lazy view in the graph
    got, = torch.autograd.grad(fn(y.conj()), y, w)
    assert torch.equal(got, ref.conj())


def test_potential_of_a_lazily_negated_density(loop):
    solver = loop[1]
    r, w = _field(3, real=True), _field(4, real=True)
    assert torch.equal(D.potential(_lazy(r), solver), D.potential(r, solver))
    x = r.clone().requires_grad_(True)
    v = D.potential(x, solver)
    ref, = torch.autograd.grad(v, x, w, retain_graph=True)
    assert torch.equal(torch.autograd.grad(v, x, _lazy(w))[0], ref)


def test_overlap_loss_equals_its_real_form(loop):
    ds, solver, _ = loop
    target = _field(5)

    def grad(loss):
        x = _field(6).requires_grad_(True)
        return torch.autograd.grad(loss(D.evolve(x, 2, ds, solver, 0.02, 1.0, -1.0)), x)[0]

    def real_form(v):
        a, b = torch.view_as_real(v).unbind(-1), torch.view_as_real(target).unbind(-1)
        return torch.hypot((a[0] * b[0] + a[1] * b[1]).sum(), (a[0] * b[1] - a[1] * b[0]).sum())

    ref = grad(real_form)
    err = (grad(lambda v: (v.conj() * target).sum().abs()) - ref).abs().max()
    assert float(err) <= 1e-13 * float(ref.abs().max())


def test_plan_methods_take_lazy_views(loop):
    ds, _, _ = loop
    u, g, phi, s = _field(7), _field(8), _field(9, real=True), _field(10, real=True)
    ds.set_linear_step(0.02, 1.0)
    for fn in (ds.linear, lambda a: ds.linear(a, True), ds.abs2, lambda a: ds.nonlinear(a, phi, 0.1, 1.0),
               lambda a: ds.abs2_vjp(a, s)):
        assert torch.equal(fn(_lazy(u)), fn(u))
    assert torch.equal(ds.nonlinear(u, _lazy(phi), 0.1, 1.0), ds.nonlinear(u, phi, 0.1, 1.0))
    assert torch.equal(ds.abs2_vjp(u, _lazy(s)), ds.abs2_vjp(u, s))
    ref = ds.nonlinear_vjp(u, phi, g, 0.1, 1.0)
    for args in ((_lazy(u), phi, g), (u, _lazy(phi), g), (u, phi, _lazy(g))):
        assert all(torch.equal(a, b) for a, b in zip(ds.nonlinear_vjp(*args, 0.1, 1.0), ref))
    # in place: the view itself holds the result
    for fn in (ds.linear_, lambda a: ds.nonlinear_(a, phi, 0.1, 1.0),
               lambda a: ds.nonlinear_vjp_finish_(_lazy(g), s, _lazy(s), 0.1, 1.0, a)):
        v, want = _lazy(u), fn(u.clone())
        assert fn(v) is v and v.is_conj() and torch.equal(v, want)


@pytest.mark.parametrize("scheme", ["strang", "yoshida"])
@pytest.mark.parametrize("steps", [0, -1, -5])
def test_no_steps_return_the_field(loop, steps, scheme):
    ds, solver, log = loop
    u = _field(11)
    for every in (0, 2):
        assert D.evolve(u, steps, ds, solver, 0.02, 1.0, -1.0, checkpoint_every=every, scheme=scheme) is u
    assert not log


@pytest.mark.parametrize("scheme,single", [("strang", D.strang_step), ("yoshida", D.yoshida_step)])
def test_flows_do_not_depend_on_checkpoints(loop, scheme, single):
    """One sequence of flows for every checkpoint_every (so one result, bit for bit), equal to single steps up to
    the merged linear flows' rounding."""
    ds, solver, log = loop
    a, steps = (ds, solver, 0.02, 1.0, -1.0), 5
    out, grads, flows = [], [], []
    for every in (0, 1, 2, 3, 5, 7):
        x = _field(12).requires_grad_(True)
        del log[:]
        v = D.evolve(x, steps, *a, checkpoint_every=every, scheme=scheme)
        flows.append(list(log))
        out.append(v.detach())
        grads.append(torch.autograd.grad(v, x, _field(13))[0])
    assert all(f == flows[0] for f in flows) and len(flows[0]) == steps * (2 if scheme == "strang" else 6) + 1
    assert all(torch.equal(v, out[0]) for v in out) and all(torch.equal(g, grads[0]) for g in grads)
    x = _field(12).requires_grad_(True)
    v = x
    for _ in range(steps):
        v = single(v, *a)
    g, = torch.autograd.grad(v, x, _field(13))
    assert float((v.detach() - out[0]).abs().max()) <= 1e-13 and float((g - grads[0]).abs().max()) <= 1e-12
    assert torch.equal(single(_field(12), *a), D.evolve(_field(12), 1, *a, scheme=scheme))
