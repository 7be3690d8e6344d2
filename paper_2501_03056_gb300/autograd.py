"""torch.autograd.Function for the uniformity energy (hand-written backward).

E(y, verts) = sum over mobile particles of (rho_i - W0)^2 at positions
x = P(y): surface particles projected onto the plane of their current
(frozen) triangle built from ``verts``, all others x = y.  Forward and
backward are the library's CUDA kernels (``fppg_energy``); torch only holds
the device buffers and the stream.  Where a gradient is wanted the forward
makes it too: it shares the grid, the kernel sums and the wait for the device
with the energy, which a backward of its own would do a second time (torus,
237 k particles: 737 -> 563 us for both).  An energy alone is for no_grad.
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
        gy = torch.empty_like(y) if grad and ctx.needs_input_grad[0] else None
        gV = torch.empty_like(verts) if grad and ctx.needs_input_grad[1] else None
        E = body.energy_ptr(y.data_ptr(), verts.data_ptr(), 0 if gy is None else gy.data_ptr(),
                            0 if gV is None else gV.data_ptr())
        # (y and verts so that a change in place before the backward is refused)
        ctx.save_for_backward(y, verts, gy, gV)
        return torch.tensor(E, dtype=torch.float64, device=y.device)

    @staticmethod
    def backward(ctx, gE):
        s = gE.to(torch.float32)
        _, _, gy, gV = ctx.saved_tensors
        return None if gy is None else gy * s, None if gV is None else gV * s, None, None


def uniformity_energy(y: torch.Tensor, verts: torch.Tensor, body: Body) -> torch.Tensor:
    return UniformityEnergy.apply(y, verts, body, torch.is_grad_enabled())
