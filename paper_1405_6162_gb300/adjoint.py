"""Gradients through the FP64 timestep: a torch.autograd.Function.

``trajectory(phi0, kappa, dims, params, nsteps)`` returns phi at time T
(from the equilibrium start with order parameter phi0) and back-propagates
to phi0 and kappa.  The forward keeps the state every ``segment`` steps; the
backward, segment by segment from the last, restores the checkpoint,
recomputes and keeps that segment's states, then sweeps them in reverse with
liblb's adjoint kernel pair (``lb_adjoint_step``, started from
``lb_adjoint_seed``, the transpose of phi_T = sum_i g_i) and finally the
initialisation's reverse (``lb_adjoint_init``).  The default keeps every state
(segment 1, nothing recomputed) where the T states of 38 N doubles take at
most 1/8 of the memory that is free on the GPU -- several trajectories can be
kept for one backward, each taking its part of what the others left -- and
one every ~sqrt(T) steps otherwise (square-root checkpointing, about
2 sqrt(T) states).  64^3, T = 200 (15.9 GB of states): the gradient 86 -> 65 ms.
Argument marshalling only: all arithmetic is in liblb's kernels.
"""
from __future__ import annotations

import math

import torch

from . import _lib as L
from .lattice import Lattice


def _p(t):
    return t.data_ptr()


_CHUNK_BYTES = 1 << 30   # states are allocated together up to this size


class _States:
    """``count`` states of n sites in device memory."""

    def __init__(self, n, count):
        self.n = n
        self.per = max(1, _CHUNK_BYTES // (38 * n * 8))
        self.chunks = [torch.empty(min(self.per, count - k) * 38 * n, device="cuda", dtype=torch.float64)
                       for k in range(0, count, self.per)]

    def __getitem__(self, k):
        """Device addresses of f and g ([19 N] each) of state k."""
        f = self.chunks[k // self.per].data_ptr() + (k % self.per) * 38 * self.n * 8
        return f, f + 19 * self.n * 8


def _free_bytes():
    """Memory an allocation can get: free on the GPU, or held unused by
    torch's caching allocator."""
    free, _ = torch.cuda.mem_get_info()
    return free + torch.cuda.memory_reserved() - torch.cuda.memory_allocated()


def _keep(n, nsteps, segment):
    """(steps between kept states, room for them)."""
    if not segment:
        if nsteps * 38 * n * 8 <= _free_bytes() // 8:
            try:
                return 1, _States(n, nsteps)
            except torch.cuda.OutOfMemoryError:   # free, but not in pieces of this size
                pass
        segment = max(1, int(round(math.sqrt(nsteps))))
    return int(segment), _States(n, -(-nsteps // int(segment)))


def _steps(nsteps, segment):
    """Steps to take.  A negative count without a segment, and a segment that
    takes no step of some, are refused before anything is allocated."""
    if not segment and nsteps < 0:
        raise ValueError(f"nsteps = {nsteps} is negative")
    if segment and int(segment) < 1 and nsteps > 0:
        raise L.LBError(L.LB_ERR_INVALID, f"trajectory in segments of {segment} steps")
    return max(nsteps, 0)


class LBTrajectory(torch.autograd.Function):
    @staticmethod
    def forward(ctx, phi0, kappa, dims, params, nsteps, segment, keep=True):
        nsteps = _steps(nsteps, segment)
        p = dict(params)
        p["kappa"] = float(kappa)
        lat, lib = Lattice.from_params(dims, p, precision="fp64"), L.lib()
        phi0 = phi0.detach().to(device="cuda", dtype=torch.float64).contiguous()
        lat.init(phi0)
        seg = kept = None
        if keep and any(ctx.needs_input_grad):
            seg, kept = _keep(lat.N, nsteps, segment)
            for t in range(0, nsteps, seg):
                L.check(lib.lb_get_state(lat.handle, *kept[t // seg], L.LB_DEVICE), "lb_get_state")
                lat.step(min(seg, nsteps - t))
        elif nsteps > 0:   # no backward can follow
            lat.step(nsteps)
        _, _, phi_t = lat.moments(device=True)
        ctx.lat, ctx.kept, ctx.nsteps, ctx.seg, ctx.phi0 = lat, kept, int(nsteps), seg, phi0
        ctx.kappa_shape = kappa.shape if torch.is_tensor(kappa) else None
        return phi_t

    @staticmethod
    def backward(ctx, grad_phi_t):
        lat, lib, kept, seg = ctx.lat, L.lib(), ctx.kept, ctx.seg
        h = lat.handle
        n = lat.N
        dev = dict(device="cuda", dtype=torch.float64)
        af = torch.empty(19 * n, **dev)
        ag = torch.empty(19 * n, **dev)
        phi_bar = grad_phi_t.detach().to(**dev).contiguous()
        L.check(lib.lb_adjoint_seed(h, _p(phi_bar), _p(af), _p(ag)), "lb_adjoint_seed")
        af2 = torch.empty_like(af)
        ag2 = torch.empty_like(ag)
        dk = torch.zeros(1, **dev)
        between = _States(n, min(seg, ctx.nsteps) - 1)   # the states between two kept ones
        for t0 in reversed(range(0, ctx.nsteps, seg)):
            t1 = min(t0 + seg, ctx.nsteps)
            if t1 - t0 > 1:
                L.check(lib.lb_set_state(h, *kept[t0 // seg], L.LB_DEVICE), "lb_set_state")
            for t in range(t0 + 1, t1):
                lat.step(1)
                L.check(lib.lb_get_state(h, *between[t - t0 - 1], L.LB_DEVICE), "lb_get_state")
            for t in range(t1 - 1, t0 - 1, -1):
                f, g = between[t - t0 - 1] if t > t0 else kept[t0 // seg]
                L.check(lib.lb_adjoint_step(h, f, g, _p(af), _p(ag), _p(af2), _p(ag2), _p(dk)), "lb_adjoint_step")
                af, af2 = af2, af
                ag, ag2 = ag2, ag
        phi0_bar = torch.empty(n, **dev)
        L.check(lib.lb_adjoint_init(h, _p(ctx.phi0), None, _p(af), _p(ag), _p(phi0_bar), _p(dk)), "lb_adjoint_init")
        lat.close()
        ctx.kept = None
        dkappa = dk[0] if ctx.kappa_shape is None else dk.reshape(ctx.kappa_shape)
        return phi0_bar, dkappa, None, None, None, None, None


def trajectory(phi0, kappa, dims, params, nsteps, segment=None):
    """phi_T of the FP64 lattice started at equilibrium with order parameter
    ``phi0`` (CUDA float64 tensor [N]) and gradient coefficient ``kappa``
    (tensor, may require grad); other parameters from ``params``."""
    if not torch.is_tensor(kappa):
        kappa = torch.tensor(float(kappa), dtype=torch.float64, device="cuda")
    return LBTrajectory.apply(phi0, kappa, tuple(dims), dict(params), int(nsteps), segment, torch.is_grad_enabled())
