"""torch.autograd.Function for the uniformity energy (hand-written backward).

E(y, verts) = sum over mobile particles of (rho_i - W0)^2 at positions
x = P(y): surface particles projected onto the plane of their current
(frozen) triangle built from ``verts``, all others x = y.  Forward and
backward are the library's CUDA kernels (``fppg_energy_forward``,
``fppg_energy_backward``); torch only holds the device buffers and the stream.
Where a backward may follow, the forward keeps its grid and kernel sums for it
in a tensor (about 50 bytes a particle and 4 a fine key), so that neither is
made twice, and a forward that is never differentiated costs no gradient.
"""
from __future__ import annotations

import torch

from . import Body


class UniformityEnergy(torch.autograd.Function):
    @staticmethod
    def forward(ctx, y: torch.Tensor, verts: torch.Tensor, body: Body, grad: bool = True):
        """grad: whether a backward may follow (with the inputs' own flags)."""
        if not (y.is_cuda and verts.is_cuda):
            raise ValueError("UniformityEnergy runs on the GPU only")
        y = y.detach().contiguous().float()
        verts = verts.detach().contiguous().float()
        body.set_stream(torch.cuda.current_stream())
        if not (grad and any(ctx.needs_input_grad[:2])):
            return torch.tensor(body.energy_ptr(y.data_ptr(), verts.data_ptr()), dtype=torch.float64, device=y.device)
        state = torch.empty(body.energy_state_bytes(body.n), dtype=torch.uint8, device=y.device)
        E = body.energy_forward_ptr(y.data_ptr(), verts.data_ptr(), state.data_ptr(), state.numel())
        ctx.save_for_backward(y, verts, state)
        ctx.body, ctx.n = body, body.n
        return torch.tensor(E, dtype=torch.float64, device=y.device)

    @staticmethod
    def backward(ctx, gE):
        y, verts, state = ctx.saved_tensors
        gy = torch.empty_like(y) if ctx.needs_input_grad[0] else None
        gV = torch.empty_like(verts) if ctx.needs_input_grad[1] else None
        ctx.body.set_stream(torch.cuda.current_stream())
        ctx.body.energy_backward_ptr(ctx.n, y.data_ptr(), verts.data_ptr(), state.data_ptr(), state.numel(),
                                     0 if gy is None else gy.data_ptr(), 0 if gV is None else gV.data_ptr())
        s = gE.to(torch.float32)
        return None if gy is None else gy * s, None if gV is None else gV * s, None, None


def uniformity_energy(y: torch.Tensor, verts: torch.Tensor, body: Body) -> torch.Tensor:
    return UniformityEnergy.apply(y, verts, body, torch.is_grad_enabled())
