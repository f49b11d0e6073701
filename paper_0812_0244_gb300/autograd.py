"""torch.autograd.Function for E_c^nl(n, grad n) on the CUDA library.

forward  : E_c^nl only (pointwise, plane and pencil transforms, contraction,
           FP64 energy); nothing of the Nq theta fields is kept.
backward : runs the pipeline again with the potential requested in its
           "gradient-output" form, which recomputes theta, and returns
             dE/dn_i         = dOmega v_loc,i
             dE/d(grad_c n)_i = dOmega w_c,i
           (Eq. Vi of the paper with the chain through grad n left to
           autograd), both scaled by the incoming gradient inside the
           assembly kernel (vdw_energy_gradients).

So when the caller builds grad n from n with its own differentiable
operator, autograd reproduces v_nl of Eq. (Vi) for that operator.
"""
from __future__ import annotations

import torch
from torch.autograd import forward_ad

from .vdwnl import VdwNL


def _memory_is_value(t):
    """Whether the bytes at t's address are all there is to t: not so for a
    batched tensor (vmap) and a zero tensor, which have no memory, for a lazily
    negated one and for a dual one, whose tangent is held elsewhere."""
    try:
        if t.data_ptr() == 0:
            return False
    except RuntimeError:
        return False
    return not t.is_neg() and forward_ad.unpack_dual(t).tangent is None


class VdwEnergy(torch.autograd.Function):
    @staticmethod
    def forward(ctx, n, grad, handle: VdwNL):
        E = torch.empty((), dtype=torch.float64, device=n.device)
        handle.energy_gradients(n.contiguous(), grad.contiguous(), E=E)
        ctx.save_for_backward(n, grad)
        ctx.handle = handle
        return E

    @staticmethod
    def backward(ctx, gE):
        n, grad = ctx.saved_tensors
        h = ctx.handle
        # create_graph, or a gE that the library cannot read by its address
        # (is_grads_batched, a negative bit, a tangent): the scaling by gE stays
        # a torch operation
        if torch.is_grad_enabled() or not _memory_is_value(gE):
            v = torch.empty_like(n, dtype=torch.float32).contiguous()
            w = torch.empty_like(grad, dtype=torch.float32).contiguous()
            h.energy_potential(n.contiguous(), grad.contiguous(), None, v, w)
            scale = (gE * h.dOmega).to(torch.float32)
            return (v * scale if ctx.needs_input_grad[0] else None,
                    w * scale if ctx.needs_input_grad[1] else None, None)
        n, grad = n.contiguous(), grad.contiguous()
        dn = torch.empty_like(n) if ctx.needs_input_grad[0] else None
        dg = torch.empty_like(grad) if ctx.needs_input_grad[1] else None
        h.energy_gradients(n, grad, gE, None, dn, dg)
        return dn, dg, None


def vdw_energy(n, grad, handle: VdwNL):
    """E_c^nl (FP64 scalar tensor) with gradients w.r.t. n and grad n."""
    return VdwEnergy.apply(n, grad, handle)
