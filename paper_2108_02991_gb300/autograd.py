"""The attraction-repulsion energy as a torch.autograd.Function.

forward  = sparkling_energy: F = F^a - F^r (paper eqs. global_minimization,
           attraction_term, repulsion_term), a float64 scalar on K's device;
backward = dL/dK = dL/dF * (A - R) / N (eqs. attraction_derivative_basic and
           Fr_grad).

Where K needs a gradient and the sums are direct, the forward computes A and
the energy of the attraction from the same reciprocal square roots
(sparkling_energy_and_grad: the SFU bounds both, so the pair costs about one)
and keeps (A - R) / N for the backward, 24 bytes a sample.  Otherwise the
backward is sparkling_energy_backward, with the per-pair distances recomputed.
Nothing of size N x N (or N x P) is ever stored.
"""
from __future__ import annotations

import torch


class SparklingEnergy(torch.autograd.Function):
    @staticmethod
    def forward(ctx_, K, rho, lo, hi, lib_ctx, acc):
        from . import make_grid, sparkling_energy, sparkling_energy_and_grad
        grid = make_grid(rho, lo, hi)
        dK = None
        if ctx_.needs_input_grad[0]:
            (F, _, _), dK = sparkling_energy_and_grad(lib_ctx, K, grid, acc)
        else:
            F, _, _ = sparkling_energy(lib_ctx, K, grid, acc)
        ctx_.save_for_backward(K, rho, dK)
        ctx_.lo, ctx_.hi, ctx_.lib_ctx, ctx_.acc = lo, hi, lib_ctx, acc
        return torch.tensor(F, dtype=torch.float64, device=K.device)

    @staticmethod
    def backward(ctx_, grad_out):
        from . import make_grid, sparkling_energy_backward
        K, rho, dK = ctx_.saved_tensors
        g = grad_out.detach().to(torch.float64).contiguous()
        if dK is not None:
            with torch.no_grad():          # no second derivative
                return (dK * g).to(K.dtype), None, None, None, None, None
        grid = make_grid(rho, ctx_.lo, ctx_.hi)
        dK = sparkling_energy_backward(ctx_.lib_ctx, K, grid, g=g, scale=1.0, acc=ctx_.acc)
        return dK, None, None, None, None, None


def sparkling_energy_fn(K, rho, lib_ctx, lo: float = -0.5, hi: float = 0.5, acc: int = 0):
    """F(K) differentiable with respect to K (CUDA tensor [N, 3])."""
    if not torch.is_grad_enabled():        # the value alone
        K = K.detach()
    return SparklingEnergy.apply(K, rho, lo, hi, lib_ctx, acc)
