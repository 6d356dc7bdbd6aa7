"""Differentiable out = D(V) psi for the staggered, Wilson and Brillouin operators.

forward:  out = D psi (dirac_apply)
backward: dL/dpsi = D^+ g (dirac_apply_dagger) and dL/dV = the link force
          (dirac_force; for Brillouin through the transporters W, which the
          backward pass rebuilds from V), both hand-written kernels of the library, with
          PyTorch's convention for real losses of complex tensors
          (grad = dL/dRe + i dL/dIm), so that for L = Re <g, D psi> the
          gradients are exactly D^+ g and F.

Loading the links into the handle (dirac_set_links: a conversion and, for
Brillouin, the build of W) is skipped where it would load what is
already there:
  - backward reloads V only if the handle was given other links after this
    node's forward pass (autograd itself rejects a V changed in place since);
  - forward, with reuse_links=True (the default), skips the load when V is
    the tensor object the handle last loaded and its version counter has not
    moved, so a training loop over fixed links loads them once.  Writes
    through V.data do not move the version counter: code that changes the
    links that way (torch.autograd.gradcheck does) passes reuse_links=False.
"""
from __future__ import annotations

import torch

from . import Dirac


class DiracApply(torch.autograd.Function):
    @staticmethod
    def forward(ctx, psi, V, D: Dirac, reuse_links: bool = True):
        if reuse_links:
            D.set_links_if_changed(V)
        else:
            D.set_links(V, remember=False)   # a later reuse_links=True call loads again
        ctx.links_generation = D.links_generation
        out = D.apply(psi.detach().to(D.canon_dtype).contiguous())
        ctx.D = D
        ctx.save_for_backward(psi, V)
        return out

    @staticmethod
    def backward(ctx, g):
        D = ctx.D
        psi, V = ctx.saved_tensors
        g = g.to(D.canon_dtype).contiguous()
        if D.links_generation != ctx.links_generation:
            D.set_links(V)   # the handle was given other links since the forward pass
        gpsi = gV = None
        if ctx.needs_input_grad[0] and ctx.needs_input_grad[1] and _own_calls(D):
            gpsi, gV = D.backward(psi.detach(), g)
            return gpsi.to(psi.dtype), gV.to(V.dtype), None, None
        if ctx.needs_input_grad[0]:
            gpsi = D.apply_dagger(g).to(psi.dtype)
        if ctx.needs_input_grad[1]:
            gV = D.force(psi.detach().to(D.canon_dtype).contiguous(), g).to(V.dtype)
        return gpsi, gV, None, None


def _own_calls(D) -> bool:
    """Whether D is a Dirac with the class's own calls, so that its fused backward gives what
    they give: not a subclass's or one handle's replacements, nor another object that has the
    calls."""
    return type(D) is Dirac and not {"apply", "apply_dagger", "force", "backward"} & D.__dict__.keys()


def dirac_apply(D: Dirac, psi: torch.Tensor, V: torch.Tensor, reuse_links: bool = True) -> torch.Tensor:
    """out = D(V) psi, differentiable in psi and V."""
    return DiracApply.apply(psi, V, D, reuse_links)
