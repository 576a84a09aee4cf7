"""The forward sweep that keeps its checkpoints for the reverse sweep: the same
bits as the pair that does not, for every interval, and the autograd function
with and without room for them."""
import pytest

import synth

pytestmark = pytest.mark.gpu
PERIODIC, DIRICHLET = 1, 0


@pytest.fixture(scope="module")
def st():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2303_08365_gb300 import build
    build.build()
    import paper_2303_08365_gb300 as st
    return st


def inputs(shape, seed):
    import torch
    u0, kappa, lam = synth.uniform(seed, shape), synth.lognormal(seed + 1, shape, 0.5), synth.normal(seed + 2, shape)
    return [torch.from_numpy(a).cuda() for a in (u0, kappa, lam)] + [0.1 / float(kappa.max())]


@pytest.mark.parametrize("shape,boundary", [((9, 13, 11), PERIODIC), ((15, 21), DIRICHLET), ((7, 1, 9), DIRICHLET),
                                            ((1, 40), PERIODIC)])
@pytest.mark.parametrize("T", [0, 1, 2, 12, 17])
def test_kept_states_give_the_same_bits(st, shape, boundary, T):
    import torch
    u0, kappa, lam, dt = inputs(shape, 51)
    p = st.Plan.varcoef(shape, boundary)
    want = u0.clone()
    p.run(want, T, kappa, dt)
    gu, gk, hu, hk, uT = (torch.empty_like(u0) for _ in range(5))
    for ckpt in (0, 1, 3, 4, T + 1, T + 5):
        n = st.stencil_kept_states(T, ckpt)
        buf = torch.full((n + 2, *shape), 7.0, dtype=torch.float64, device="cuda")
        kept, before = buf[1:n + 1], u0.clone()
        st.stencil_run_kept(p.handle, u0, uT, T, kappa, dt, ckpt, kept)
        assert torch.equal(uT, want) and torch.equal(u0, before), ckpt
        st.stencil_adjoint_vjp_kept(p.handle, u0, kappa, dt, T, ckpt, kept, lam, gu, gk)
        st.stencil_adjoint_vjp(p.handle, u0, kappa, dt, T, ckpt, lam, hu, hk)
        assert torch.equal(gu, hu) and torch.equal(gk, hk), ckpt
        assert bool((buf[0] == 7.0).all()) and bool((buf[-1] == 7.0).all()), ckpt
    p.close()


def test_autograd_with_and_without_room(st, monkeypatch):
    import torch
    from paper_2303_08365_gb300 import autograd
    shape = (12, 10, 14)
    u0, kappa, lam, dt = inputs(shape, 61)
    p = st.Plan.varcoef(shape, DIRICHLET)
    got = []
    for room in (True, False):
        if not room:
            monkeypatch.setattr(autograd, "_room_for_states", lambda *a: None)
        u, k = u0.clone().requires_grad_(), kappa.clone().requires_grad_()
        out = autograd.diffuse(u, k, p, dt, 19)
        got.append([out.detach(), *torch.autograd.grad(out, (u, k), lam)])
    assert all(torch.equal(a, b) for a, b in zip(*got))
    with torch.no_grad():
        assert torch.equal(autograd.diffuse(u0, kappa, p, dt, 19), got[0][0])
    p.close()


@pytest.mark.parametrize("short", ["driver", "states", "output", "scratch"])
def test_autograd_short_of_memory(st, monkeypatch, short):
    """Where the checkpoints would take what the rest needs, the passes go without them, with
    the same results: too little free memory, or an allocation of the kept pass that fails."""
    import torch
    from paper_2303_08365_gb300 import autograd
    shape, T = (12, 10, 14), 19
    u0, kappa, lam, dt = inputs(shape, 71)
    p = st.Plan.varcoef(shape, DIRICHLET)

    def forward():
        u, k = u0.clone().requires_grad_(), kappa.clone().requires_grad_()
        out = autograd.diffuse(u, k, p, dt, T)
        return out, u, k, len(out.grad_fn.saved_tensors) == 3

    def fails(error):
        def f(*args, **kwargs):
            raise error
        return f

    def results(out, u, k, kept):
        return [out.detach(), *torch.autograd.grad(out, (u, k), lam)]

    plenty = forward()
    assert plenty[-1]
    with monkeypatch.context() as m:
        if short == "driver":  # other graphs hold a sixteenth, and half of the device is not free any more
            total = torch.cuda.get_device_properties(0).total_memory
            n = st.stencil_kept_states(T)  # and a segment of at most T / n, scratch and outputs
            need = 8 * u0.numel() * (n + T // n + 16)
            m.setitem(autograd._Held.alive, u0.device, total // 16)
            m.setattr(torch.cuda, "mem_get_info", lambda *a: (total // 2 + need, total))
            assert forward()[-1]
            m.setattr(torch.cuda, "mem_get_info", lambda *a: (total // 2 + need - 1, total))
        elif short == "states":
            m.setattr(torch, "empty", fails(torch.OutOfMemoryError("no room")))
        elif short == "output":
            m.setattr(torch, "empty_like", fails(torch.OutOfMemoryError("no room")))
        else:
            m.setattr(autograd, "stencil_run_kept", fails(st.StencilError(st.ERR_OOM, "no room")))
        without = forward()
    assert not without[-1]
    held = autograd._Held.alive[u0.device]
    assert held >= 8 * u0.numel() * st.stencil_kept_states(T)
    assert all(torch.equal(a, b) for a, b in zip(results(*plenty), results(*without)))
    del plenty
    assert autograd._Held.alive[u0.device] == held - 8 * u0.numel() * st.stencil_kept_states(T)
    p.close()


def test_kept_calls_leave_no_earlier_message(st):
    import torch
    u0, kappa, lam, dt = inputs((5, 6, 7), 81)
    p = st.Plan.varcoef((5, 6, 7), DIRICHLET)
    uT, gu, gk = (torch.empty_like(u0) for _ in range(3))
    kept = torch.empty((st.stencil_kept_states(9), 5, 6, 7), dtype=torch.float64, device="cuda")
    for call in (lambda: st.stencil_run_kept(p.handle, u0, uT, 9, kappa, dt, 0, kept),
                 lambda: st.stencil_adjoint_vjp_kept(p.handle, u0, kappa, dt, 9, 0, kept, lam, gu, gk)):
        with pytest.raises(st.StencilError):
            p.run(uT, 1, kappa, -1.0)
        assert st.last_error() != ""
        call()
        assert st.last_error() == ""
    p.close()
