"""torch.autograd.Functions over the library's sweeps and their adjoints.

ConstStencilFn.apply(u0, plan, adjoint_plan, T) returns u^T for a
constant-weight plan; its backward sweeps the transposed stencil (the
reflected weights w_{-o}, same boundary rule: the transpose of the zero-ghost
and of the periodic operator) T steps over the upstream gradient.
`sweep(u0, dims, radius, weights, boundary, T)` builds both plans.

StencilAdjointFn.apply(u0, kappa, plan, dt, T, ckpt_every) returns u^T, the
field after T explicit steps of du/dt = div(kappa grad u) (the paper's Eq. 1
with a per-cell diffusivity).  Its backward takes the upstream gradient
dL/du^T as lambda^T and sweeps the transposed stencil backward in time
(stencil_adjoint_vjp), recomputing the forward states from checkpoints every
ckpt_every steps (0: about sqrt(T)).  dt is a constant (no gradient).  Every
step runs in the library's CUDA kernels.  diffuse() lets the forward pass keep
those checkpoints, about T / ckpt_every grids until the graph is freed, where a
gradient is asked for, so that the backward pass does not sweep forward again.
It keeps them only as long as that leaves half of the device's memory free (a
sixteenth of the device, all graphs together, goes without the question), for
the sweeps' own scratch and whatever else the program is yet to allocate.
Otherwise a pass keeps u0 and kappa alone.
"""
import functools
import threading

import numpy as np
import torch

from . import (ERR_OOM, Plan, StencilError, stencil_adjoint_vjp, stencil_adjoint_vjp_kept, stencil_kept_states,
               stencil_run, stencil_run_kept)


class StencilAdjointFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, u0, kappa, plan, dt, T, ckpt_every=0, keep=False):
        ctx.plan, ctx.dt, ctx.T, ctx.ckpt = plan, float(dt), int(T), int(ckpt_every)
        done = _run_kept(u0, kappa, plan, ctx.dt, ctx.T, ctx.ckpt) if keep else None
        if done is None:
            u = u0.detach().clone().contiguous()
            stencil_run(plan.handle, u, T, kappa.detach().contiguous(), dt)
            ctx.save_for_backward(u0.detach(), kappa.detach())
            return u
        u, kept, ctx.held = done
        ctx.save_for_backward(u0.detach(), kappa.detach(), kept)
        return u

    @staticmethod
    def backward(ctx, grad_out):
        u0, kappa, *kept = ctx.saved_tensors
        lam = grad_out.detach().contiguous()
        gu = torch.empty_like(u0)
        gk = torch.empty_like(u0)
        if kept:
            stencil_adjoint_vjp_kept(ctx.plan.handle, u0.contiguous(), kappa.contiguous(), ctx.dt, ctx.T, ctx.ckpt,
                                     kept[0], lam, gu, gk)
        else:
            stencil_adjoint_vjp(ctx.plan.handle, u0.contiguous(), kappa.contiguous(), ctx.dt, ctx.T,
                                ctx.ckpt, lam, gu, gk)
        return gu, gk, None, None, None, None, None


class _Held:
    """The bytes that a graph's checkpoints take, summed per device over the graphs alive."""
    alive = {}
    lock = threading.Lock()

    def __init__(self, device, n):
        self.device, self.n = device, n
        with self.lock:
            self.alive[device] = self.alive.get(device, 0) + n

    def __del__(self):
        with self.lock:
            self.alive[self.device] -= self.n


def _run_kept(u0, kappa, plan, dt, T, ckpt_every):
    """(u^T, its checkpoints, their _Held); None where there is no room for them."""
    try:
        kept = _room_for_states(u0, T, ckpt_every)
        if kept is None:
            return None
        u = torch.empty_like(u0, memory_format=torch.contiguous_format)
        stencil_run_kept(plan.handle, u0.detach().contiguous(), u, T, kappa.detach().contiguous(), dt, ckpt_every, kept)
        return u, kept, _Held(kept.device, 8 * kept.numel())
    except torch.OutOfMemoryError:
        return None
    except StencilError as e:
        if e.code != ERR_OOM:
            raise
        return None


@functools.lru_cache
def _total_memory(device):
    return torch.cuda.get_device_properties(device).total_memory


def _room_for_states(u0, T, ckpt_every):
    """An uninitialised tensor for the checkpoints of a forward pass; None when the device
    has no room for it, or u0 is not what the sweep takes (it says so itself)."""
    if u0.device.type != "cuda" or u0.dtype != torch.float64 or T < 0 or ckpt_every < 0:
        return None
    n = stencil_kept_states(T, ckpt_every)
    # with the sweeps' scratch (5 grids forward, 8 and a segment's states backward) and the
    # outputs, 3 grids
    need = 8 * u0.numel() * (n + (T // n if n else T) + 16)
    total = _total_memory(u0.device)
    # the driver's answer takes 15 to 20 us, a small pass 370: asked from a thousandth of the
    # device on, and once the graphs alive hold a sixteenth
    if need > total // 1024 or need + _Held.alive.get(u0.device, 0) > total // 16:
        if torch.cuda.mem_get_info(u0.device)[0] < total // 2 + need:
            return None
    return torch.empty((n, *u0.shape), dtype=u0.dtype, device=u0.device)


def diffuse(u0, kappa, plan, dt, T, ckpt_every=0):
    """u^T with autograd support for u0 and kappa."""
    keep = torch.is_grad_enabled() and (u0.requires_grad or kappa.requires_grad)
    return StencilAdjointFn.apply(u0, kappa, plan, dt, T, ckpt_every, keep)


def reflected(weights):
    """w_{-o}: the weights of the transposed stencil (every axis reversed)."""
    w = np.asarray(weights, dtype=np.float64)
    return np.ascontiguousarray(w[(slice(None, None, -1),) * w.ndim])


class ConstStencilFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, u0, plan, adjoint_plan, T):
        u = u0.detach().clone().contiguous()
        stencil_run(plan.handle, u, T)
        ctx.adjoint_plan, ctx.T = adjoint_plan, int(T)
        return u

    @staticmethod
    def backward(ctx, grad_out):
        lam = grad_out.detach().clone().contiguous()
        stencil_run(ctx.adjoint_plan.handle, lam, ctx.T)
        return lam, None, None, None


def sweep(u0, dims, radius, weights, boundary, T, plans=None):
    """u^T of a constant-weight stencil with autograd support for u0.  Pass
    `plans` = (plan, adjoint_plan) to reuse plans across calls; otherwise they
    are built here (the adjoint plan takes the reflected weights)."""
    if plans is None:
        plans = (Plan(dims, radius, weights, boundary), Plan(dims, radius, reflected(weights), boundary))
    return ConstStencilFn.apply(u0, plans[0], plans[1], T)
