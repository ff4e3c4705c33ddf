"""Differentiable rollout of the relative-velocity scheme for PyTorch.

``Rollout.apply(u0, s_nu, amp, sim, n, seg, rho0)`` sets the state of ``sim`` to the
equilibrium of (rho0, u0), advances n steps with checkpoints every ``seg`` steps, and returns
the final density and velocity fields. With ``seg`` None or 0 the checkpoints are as dense as
the free memory allows, see ``default_workspace``; the gradient does not depend on
the interval, bit for bit. The backward pass runs the hand-written
discrete adjoint of the library (moments adjoint, reverse sweep, equilibrium adjoint),
giving gradients with respect to the initial velocity field, the shear rate s_nu (the
shared rate of p_xx and p_xy) and the amplitude of a prescribed relative velocity.
All arithmetic runs in the CUDA library; this module only moves tensors.
"""
from __future__ import annotations

import math
import threading
import time

import torch


# Shares of a device's memory that checkpoints may take without being asked for: one rollout's,
# of all memory; what those of all live rollouts hold beyond sqrt(n) checkpoints, of the free
# memory; and what needs no look at the free memory. The look makes a pass 60 us longer (15 steps
# at 1024^2 1050 -> 1110 us), so it is taken at most every LOOK_SECONDS.
CHECKPOINT_SHARE = 1 / 16
LIVE_SHARE = 1 / 8
SMALL_SHARE = 1 / 1024
LOOK_SECONDS = 0.25

# Bytes that the workspaces alive on each device hold beyond those of sqrt(n) checkpoints.
_extra: dict = {}
# Per device: when the free memory was last looked at, and what was free without those bytes.
_seen: dict = {}
_extra_lock = threading.RLock()  # a workspace may be collected while its own thread holds it


def checkpoint_interval(sim, n: int, budget: float | None = None) -> int:
    """The shortest checkpoint interval whose workspace stays within `budget` bytes (default:
    CHECKPOINT_SHARE of the device's memory), at most sqrt(n), which needs the least. Every step
    within an interval is recomputed before it is reversed, a quarter of a gradient's time with
    sqrt(n): 200 steps at 1024^2 take 7.8 ms with 15 steps between checkpoints (1.2 GB) and
    6.1 ms with none (7.6 GB)."""
    longest = max(1, math.ceil(math.sqrt(n)))
    if budget is None:
        budget = CHECKPOINT_SHARE * torch.cuda.get_device_properties(sim.device).total_memory
    for seg in range(1, longest):
        if sim.adjoint_workspace_bytes(n, seg) <= budget:
            return seg
    return longest


class _Lease:
    """Bytes of _extra[device], given back when it goes."""

    __slots__ = ("device", "nbytes")

    def __init__(self, device, nbytes: int):
        self.device, self.nbytes = device, nbytes

    def __del__(self):
        if _extra_lock is not None:  # else the interpreter is going down
            with _extra_lock:
                _extra[self.device] -= self.nbytes


def default_workspace(sim, n: int):
    """Checkpoint interval and workspace of a rollout that names no interval. The workspace takes
    at most CHECKPOINT_SHARE of the device's memory, unless sqrt(n) checkpoints need more. What
    it holds beyond those, together with what all others alive on the device hold beyond
    theirs, stays within LIVE_SHARE of the memory that the driver would have free with sqrt(n)
    checkpoints only: a program that keeps many rollouts alive, or that leaves little memory
    free, gets sqrt(n) checkpoints, as it does where the allocation fails."""
    longest = max(1, math.ceil(math.sqrt(n)))
    if longest == 1:
        return 1, sim.adjoint_workspace(n, 1)
    device = sim.device
    least, most = (sim.adjoint_workspace_bytes(n, seg) for seg in (longest, 1))
    total = torch.cuda.get_device_properties(device).total_memory
    with _extra_lock:
        held = _extra.setdefault(device, 0)
        if held + most - least <= SMALL_SHARE * total:
            seg = 1
        else:
            now = time.monotonic()
            when, free = _seen.get(device, (-math.inf, 0))
            if now - when > LOOK_SECONDS:
                index = device.index if device.index is not None else torch.cuda.current_device()
                free = torch.cuda.cudart().cudaMemGetInfo(index)[0] + held
                _seen[device] = now, free
            room = LIVE_SHARE * max(0, free - least) - held
            budget = min(least + room, CHECKPOINT_SHARE * total)
            seg = 1 if most <= budget else checkpoint_interval(sim, n, budget)
        more = max(0, (most if seg == 1 else sim.adjoint_workspace_bytes(n, seg)) - least)
        _extra[device] += more
    lease = _Lease(device, more)
    try:
        ws = sim.adjoint_workspace(n, seg)
    except torch.cuda.OutOfMemoryError:
        _seen.pop(device, None)
        if more == 0:
            raise
        return longest, sim.adjoint_workspace(n, longest)
    ws.lease = lease  # given back with the workspace, or on the way out
    return seg, ws


class Rollout(torch.autograd.Function):
    @staticmethod
    def forward(ctx, u0, s_nu, amp, sim, n, seg, rho0):
        s = list(sim.s)
        s[4] = s[5] = float(s_nu)
        sim.set_rates(s)
        sim.set_utilde(sim._ut0, float(amp), sim.period)
        u0c = u0.detach().to(device=sim.device, dtype=torch.float32).contiguous()
        rho0c = None if rho0 is None else rho0.detach().to(sim.device, torch.float32).contiguous()
        rho_in = rho0c if rho0c is not None else torch.ones((sim.ny, sim.nx), device=sim.device)
        sim.init_equilibrium(rho_in, u0c[0], u0c[1])
        if seg:
            seg = int(seg)
            ws = sim.adjoint_workspace(n, seg)
        else:
            seg, ws = default_workspace(sim, n)
        sim.forward_checkpointed(n, seg, ws)
        rho, ux, uy = sim.moments()
        ctx.sim, ctx.n, ctx.seg, ctx.ws = sim, n, seg, ws
        ctx.meta = [(t.dtype, t.device) if torch.is_tensor(t) else (torch.float64, None)
                    for t in (s_nu, amp)]
        ctx.save_for_backward(u0c, rho_in)
        return rho, torch.stack([ux, uy])

    @staticmethod
    def backward(ctx, grad_rho, grad_u):
        sim = ctx.sim
        u0c, rho_in = ctx.saved_tensors
        dL_dS = sim.moments_vjp(grad_rho, grad_u)
        d0, ds, da, _ = sim.adjoint(ctx.n, ctx.seg, ctx.ws, dL_dS)
        _, du0 = sim.equilibrium_vjp(rho_in, u0c, d0)
        (sd, sdev), (ad, adev) = ctx.meta
        g_snu = torch.tensor(ds[4] + ds[5], dtype=sd, device=sdev)
        g_amp = torch.tensor(da, dtype=ad, device=adev)
        return du0.to(u0c.dtype), g_snu, g_amp, None, None, None, None
