"""Differentiable potential energy over path frames (torch.autograd), marshalling only.

PotentialEnergy(X) -> U(X_t) per frame (scps_energy_forces). Its backward
returns g_t * grad U(X_t) through ForceGrad, whose own backward is the
Hessian-vector product H(X_t) v_t (scps_hvp). So second derivatives of path
functionals work, e.g. the gradient of sum_t |grad U(X_t)|^2 (a term of the
Onsager-Machlup action of Eq. (SOM)) is sum_t 2 H(X_t) grad U(X_t).
ForceNormSquared and ForceNormAction compute that action with one force launch forward
and one force + one HVP launch backward (force_norm_action).
All arithmetic runs in the CUDA kernels behind the C ABI.
"""
from __future__ import annotations

import torch


class ForceGrad(torch.autograd.Function):
    """grad U(X_t) for frames X (float32, (T, n, 3), CUDA); backward: H(X_t) v_t."""

    @staticmethod
    def forward(ctx, X, system, topo):
        X = X.contiguous()
        U = torch.empty(X.shape[0], dtype=torch.float64, device=X.device)
        F = torch.empty_like(X)
        system.energy_forces(topo, X, U, F)
        ctx.save_for_backward(X)
        ctx.system, ctx.topo = system, topo
        return -F

    @staticmethod
    def backward(ctx, v):
        (X,) = ctx.saved_tensors
        HV = torch.empty_like(X)
        ctx.system.hvp(ctx.topo, X, v.contiguous().to(X.dtype), HV)
        return HV, None, None


class PotentialEnergy(torch.autograd.Function):
    """U(X_t) per frame (float64); backward: g_t grad U(X_t), itself differentiable."""

    @staticmethod
    def forward(ctx, X, system, topo):
        X = X.contiguous()
        U = torch.empty(X.shape[0], dtype=torch.float64, device=X.device)
        system.energy_forces(topo, X, U, None)
        ctx.save_for_backward(X)
        ctx.system, ctx.topo = system, topo
        return U

    @staticmethod
    def backward(ctx, gU):
        (X,) = ctx.saved_tensors
        grad = ForceGrad.apply(X, ctx.system, ctx.topo)
        return gU.to(grad.dtype)[:, None, None] * grad, None, None


def potential_energy(system, X, topo=0):
    return PotentialEnergy.apply(X, system, topo)


class ForceNormSquared(torch.autograd.Function):
    """sum_t |grad U(X_t)|^2 over frames X (float64 scalar). The forces are not kept:
    the backward evaluates them again and returns g * 2 H(X_t) grad U(X_t) (one
    force launch and one HVP launch), which is activation checkpointing over the
    frames without the generic checkpoint machinery. First order only: for further
    derivatives compose ForceGrad instead."""

    @staticmethod
    def forward(ctx, X, system, topo):
        X = X.contiguous()
        U = torch.empty(X.shape[0], dtype=torch.float64, device=X.device)
        F = torch.empty_like(X)
        system.energy_forces(topo, X, U, F)
        ctx.save_for_backward(X)
        ctx.system, ctx.topo = system, topo
        return (F.double() ** 2).sum()

    @staticmethod
    def backward(ctx, g):
        (X,) = ctx.saved_tensors
        U = torch.empty(X.shape[0], dtype=torch.float64, device=X.device)
        F = torch.empty_like(X)
        ctx.system.energy_forces(ctx.topo, X, U, F)
        HV = torch.empty_like(X)
        ctx.system.hvp(ctx.topo, X, F.mul_(-2.0), HV)  # v = 2 grad U = -2 F
        return HV * g.to(HV.dtype), None, None


class ForceNormAction(torch.autograd.Function):
    """sum_t |grad U(X_t)|^2 over all frames X (float64 scalar). The forward evaluates every
    frame in one launch and keeps only the positions; the backward evaluates the forces
    again, straight into the gradient it returns, and applies 2 H(X_t) grad U(X_t) there in
    place, frame by frame: one force launch and one HVP launch, and no memory beyond the
    gradient (segments of frames with buffers of their own need more and, at 50 frames,
    leave a third of the GPU idle in 20 launches of each: 2.3 ms for 1000 x 560 atoms, forward
    and backward, against 1.1 ms). First order only, like ForceNormSquared."""

    @staticmethod
    def forward(ctx, X, system, topo, segment=50):
        X = X.contiguous()
        U = torch.empty(X.shape[0], dtype=torch.float64, device=X.device)
        F = torch.empty_like(X)
        system.energy_forces(topo, X, U, F)
        ctx.save_for_backward(X)
        ctx.system, ctx.topo, ctx.segment = system, topo, segment
        return (F.double() ** 2).sum()

    @staticmethod
    def backward(ctx, g):
        if ctx.segment < 1:
            raise ValueError("segment must be at least 1")
        (X,) = ctx.saved_tensors
        U = torch.empty(X.shape[0], dtype=torch.float64, device=X.device)
        G = torch.empty_like(X)
        ctx.system.energy_forces(ctx.topo, X, U, G)
        G.mul_(-2.0)  # v = 2 grad U
        ctx.system.hvp(ctx.topo, X, G, G)
        return G.mul_(g.to(G.dtype)), None, None, None


def force_norm_action(system, X, topo=0, segment=50):
    """sum_t |grad U(X_t)|^2 over the frames; the backward recomputes the forces (activation
    checkpointing over path frames). `segment` bounded the frames whose forces were live at a
    time; the backward needs no memory for them any more, so every value from 1 on gives the
    same (smaller ones are refused by the backward)."""
    return ForceNormAction.apply(X, system, topo, segment)
