"""Differentiable rollouts through the CUDA forward and adjoint kernels.

`HydroRollout.apply(U0, gamma, mesh, dts, every)` advances U0 by len(dts)
Heun steps with the given (recorded) time steps and is differentiable with
respect to U0 and gamma.  The dt schedule is a constant of the derivative:
record it once with `schedule` and reuse it, so that finite differences and
the adjoint see the same steps.

Memory: the forward pass keeps a checkpoint every `every` steps.  The
backward pass re-runs each segment from its checkpoint (keeping that
segment's states) and then applies hard_hydro_step_backward step by step in
reverse, accumulating dL/dU and dL/dgamma.
"""
from __future__ import annotations

from dataclasses import dataclass

import torch

from . import HardHydro, check, hard_hydro_steps, hard_hydro_steps_backward


@dataclass(frozen=True)
class Mesh:
    shape: tuple                    # (nz, ny, nx)
    bc: object = 0                  # one kind or six (x-, x+, y-, y+, z-, z+)
    extent: tuple = (1.0, 1.0, 1.0)


def _handle(mesh: Mesh, gamma: float, dtype):
    return HardHydro(mesh.shape, gamma, mesh.bc, dtype=dtype, extent=mesh.extent)


def schedule(U0, gamma, mesh: Mesh, nsteps: int, cfl: float):
    """The CFL time steps of a forward rollout (host list of floats)."""
    m = _handle(mesh, float(gamma), U0.dtype)
    U = U0.detach().clone()
    dts = []
    for _ in range(nsteps):
        dt = m.cfl_dt(U, cfl)
        dts.append(dt)
        U = m.step(U, dt)
    return dts


class _States:
    """Room for n states, each on a 16-byte boundary."""

    def __init__(self, n, like):
        step = (like.numel() + 31) // 32 * 32
        self.flat = torch.empty(n * step, dtype=like.dtype, device=like.device)
        self.size, self.step = like.numel(), step

    def __getitem__(self, i):
        return self.flat[i * self.step:i * self.step + self.size]

    def pointer(self, i):
        return self.flat.data_ptr() + i * self.step * self.flat.element_size()


class HydroRollout(torch.autograd.Function):
    """The steps of a segment go to the library in one call, and the handle's
    scratch comes from the caching allocator: 256^2 FP32, 20 steps and their
    gradient, 2.23 -> 1.39 ms, of which the kernels are ~0.9 (a call per step and
    buffer, and cudaMalloc / cudaFree per rollout, were the rest)."""

    @staticmethod
    def forward(ctx, U0, gamma, mesh: Mesh, dts, every: int = 20):
        m = _handle(mesh, float(gamma), U0.dtype)
        dts = list(dts)
        n = len(dts)
        U = U0.detach().contiguous().clone()
        # out[i], the state after step i: a checkpoint every `every` steps, else
        # one of two buffers in turn; the last in a tensor of its own
        marks = [i for i in range(n - 1) if (i + 1) % every == 0]
        ckpts = _States(len(marks), U)
        ctx.first, ctx.work = U, None
        if n:
            start = m._check(U)
            ctx.work = m.workspace(0, U.device)
            turn, last = _States(2 if n > 1 else 0, U), torch.empty_like(U)
            out = [turn.pointer(i & 1) for i in range(n - 1)] + [last.data_ptr()]
            for k, i in enumerate(marks):
                out[i] = ckpts.pointer(k)
            check(hard_hydro_steps(m.h, start, out, dts, m._stream()), "hard_hydro_steps")
            U = last
        else:
            U = U.clone()
        ctx.m, ctx.dts, ctx.every, ctx.ckpts, ctx.segments = m, dts, every, ckpts, len(marks) + 1
        ctx.gamma_dtype = gamma.dtype if torch.is_tensor(gamma) else torch.float64
        return U

    @staticmethod
    def backward(ctx, gU):
        m, dts, every = ctx.m, ctx.dts, ctx.every
        g = gU.contiguous().clone()
        g_gamma = torch.zeros((), dtype=torch.float64, device=gU.device)
        if dts:
            gp, s = m._check(g), m._stream()
            here = torch.cuda.current_stream(gU.device)
            for t in (ctx.first, ctx.ckpts.flat, ctx.work):
                t.record_stream(here)                 # the forward pass may have had another
            work = m.workspace(1, gU.device)
            states = _States(min(every, len(dts)) - 1, g)
            for seg in reversed(range(ctx.segments)):
                start = seg * every
                stop = min(len(dts), start + every)
                at = [ctx.first.data_ptr() if seg == 0 else ctx.ckpts.pointer(seg - 1)]
                at += [states.pointer(i) for i in range(stop - start - 1)]
                check(hard_hydro_steps(m.h, at[0], at[1:], dts[start:stop - 1], s), "hard_hydro_steps")
                check(hard_hydro_steps_backward(m.h, at, gp, dts[start:stop], g_gamma.data_ptr(), s),
                      "hard_hydro_steps_backward")
            ctx.adjoint_work = work                   # the handle's until the next call
        return g, g_gamma.to(ctx.gamma_dtype), None, None, None


def rollout(U0, gamma, mesh: Mesh, dts, every: int = 20):
    if not torch.is_tensor(gamma):
        gamma = torch.tensor(float(gamma), dtype=torch.float64, device=U0.device)
    return HydroRollout.apply(U0, gamma, mesh, dts, every)
