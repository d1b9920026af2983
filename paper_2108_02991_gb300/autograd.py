"""Differentiable sampling-pattern energy on the GPU.

forward  = sparkling_energy: F = F^a - F^r (paper eqs. global_minimization,
           attraction_term, repulsion_term), a float64 scalar on K's device;
backward = dL/dK = dL/dF * (A - R) / N (eqs. attraction_derivative_basic and
           Fr_grad).

Where K needs a gradient and the sums are direct, the forward forms A from the
reciprocal square roots of the attraction's energy (sparkling_energy_keep: the
SFU bounds both, so the pair costs little more than one) and keeps it for the
backward, 24 bytes a sample; the backward is left with the repulsion.  In the
other modes, and with keep_attraction=False, the forward is the energy alone
and the backward sums both.  Nothing of size N x N (or N x P) is ever stored.

A forward that no backward follows (a logged loss, the trials of a line search)
costs least under torch.no_grad() or with keep_attraction=False; otherwise it
takes 4 to 9 % longer than sparkling_energy.
"""
from __future__ import annotations

import torch

from . import make_grid, sparkling_energy, sparkling_energy_backward_kept, sparkling_energy_keep


class SparklingEnergy(torch.autograd.Function):
    @staticmethod
    def forward(ctx_, K, rho, lo, hi, lib_ctx, acc, keep=True):
        grid = make_grid(rho, lo, hi)
        A, ctx_.eps = None, -1.0
        if keep and ctx_.needs_input_grad[0]:
            (F, _, _), A, ctx_.eps = sparkling_energy_keep(lib_ctx, K, grid, acc)
        else:
            F, _, _ = sparkling_energy(lib_ctx, K, grid, acc)
        ctx_.save_for_backward(K, rho, A)
        ctx_.lo, ctx_.hi, ctx_.lib_ctx, ctx_.acc = lo, hi, lib_ctx, acc
        return torch.tensor(F, dtype=torch.float64, device=K.device)

    @staticmethod
    def backward(ctx_, grad_out):
        K, rho, A = ctx_.saved_tensors
        grid = make_grid(rho, ctx_.lo, ctx_.hi)
        g = grad_out.to(torch.float64).contiguous()        # only its values are read
        dK = sparkling_energy_backward_kept(ctx_.lib_ctx, K, grid, A, ctx_.eps, g=g, scale=1.0,
                                            acc=ctx_.acc)
        return dK, None, None, None, None, None, None


def sparkling_energy_fn(K, rho, lib_ctx, lo: float = -0.5, hi: float = 0.5, acc: int = 0,
                        keep_attraction: bool = True):
    """F(K) differentiable with respect to K (CUDA tensor [N, 3]).

    keep_attraction=False: the forward computes the value alone and keeps
    nothing but K and rho, the backward sums the attraction as well."""
    if not torch.is_grad_enabled():        # the value alone
        K = K.detach()
    return SparklingEnergy.apply(K, rho, lo, hi, lib_ctx, acc, keep_attraction)
