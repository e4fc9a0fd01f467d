"""torch.autograd binding of the differentiable leapfrog.

``leapfrog(x0, v0, m, nsteps, dt, eps)`` runs nsteps kick-drift-kick steps
(paper Sec. 3.1) on the GPU through libnbody and returns (x(T), v(T)); the
backward pass calls the library's checkpointed adjoint, so gradients with
respect to x0, v0 and m come from the hand-written adjoint kernel, not from
torch's tracing.  Tensors are float32 on one CUDA device; torch provides
only the device memory and the stream.
"""
from __future__ import annotations

import torch

from . import _lib


def _scratch(n, device):
    """Memory for the pair-symmetric force, or None (small n, or no room: the
    one-sided force needs none)."""
    size = _lib.lf_scratch_bytes(n)
    if size == 0:
        return None
    try:
        return torch.empty(size, dtype=torch.uint8, device=device)
    except torch.OutOfMemoryError:
        return None


class LeapfrogFunction(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x0, v0, m, nsteps: int, dt: float, eps: float, G: float, ckpt_every: int):
        for t in (x0, v0, m):
            if t.dtype != torch.float32 or not t.is_cuda:
                raise TypeError("leapfrog needs float32 CUDA tensors")
        n = m.shape[0]
        stream = torch.cuda.current_stream(x0.device)
        x = x0.detach().contiguous().clone()
        v = v0.detach().contiguous().clone()
        mm = m.detach().contiguous()
        acc = torch.empty_like(x)
        ckpt = torch.empty(_lib.lf_ckpt_floats(n, nsteps, ckpt_every), dtype=torch.float32,
                           device=x.device)
        scratch = _scratch(n, x.device)
        _lib.lf_forward(n, mm, x, v, acc, nsteps, dt, ckpt, eps=eps, G=G, ckpt_every=ckpt_every,
                        stream=stream, scratch=scratch)
        ctx.save_for_backward(mm, ckpt)
        # the backward pass re-runs these steps: with the same force (should there
        # be no room for its scratch then, up to FP32 rounding)
        ctx.lent = scratch is not None
        ctx.cfg = (n, nsteps, dt, eps, G, ckpt_every)
        return x, v

    @staticmethod
    def backward(ctx, gx, gv):
        mm, ckpt = ctx.saved_tensors
        n, nsteps, dt, eps, G, ckpt_every = ctx.cfg
        dev = mm.device
        lx = (gx.detach().contiguous().clone() if gx is not None
              else torch.zeros((n, 3), dtype=torch.float32, device=dev))
        lv = (gv.detach().contiguous().clone() if gv is not None
              else torch.zeros((n, 3), dtype=torch.float32, device=dev))
        lm = torch.empty(n, dtype=torch.float32, device=dev)
        work = torch.empty(_lib.lf_work_floats(n, ckpt_every), dtype=torch.float32, device=dev)
        _lib.lf_backward(n, mm, ckpt, nsteps, dt, lx, lv, lm, work, eps=eps, G=G,
                         ckpt_every=ckpt_every, stream=torch.cuda.current_stream(dev),
                         scratch=_scratch(n, dev) if ctx.lent else None)
        return lx, lv, lm, None, None, None, None, None


def leapfrog(x0, v0, m, nsteps: int, dt: float, eps: float, G: float = 1.0, ckpt_every: int = 8):
    """Differentiable KDK leapfrog; returns (x(T), v(T))."""
    return LeapfrogFunction.apply(x0, v0, m, int(nsteps), float(dt), float(eps), float(G),
                                  int(ckpt_every))
