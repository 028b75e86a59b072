"""torch.autograd.Function around the CUDA adjoint of the forced FCLB update.

Forward: T steps of the D3Q27 FCLB update from a given state under a body
force F (lbm_adjoint_forward, checkpointing every `every` steps, 0 = the
library's choice); returns the final distributions f_T.  Backward: dL/dF
from dL/df_T by the hand-written adjoint stream-collide kernel
(lbm_adjoint_backward).  A context records one forward at a time: the node
keeps the generation of its forward and its backward refuses to run once
the context has recorded another (or its force was reset), instead of
returning the gradient of a different forward.  The distributions and
gradients move through the C ABI as float64 arrays: where F lives (the
library reads and writes device arrays of its own GPU in place), on the
host otherwise; all stepping, recomputation and adjoint sweeps run in the
CUDA library.  96^3, T = 128, F on the GPU: 177 ms through host arrays and
staged copies, 20 ms in place (forward, loss and backward).
"""
import ctypes

import numpy as np
import torch

from . import lbm


def _in_place(t):
    """Whether the library may take t's memory as it is: contexts live on the
    process's one visible GPU."""
    return t.is_cuda and torch.cuda.device_count() == 1


def _plain(t):
    """t as float64 values in a row of memory.  (A tensor may carry a pending
    sign, torch.Tensor.is_neg, that neither double() nor contiguous() resolves
    when type and layout are right already.)"""
    return t.detach().double().contiguous().resolve_neg()


def _call(fn, ctx, *args):
    """A C entry point on float64 device tensors.  The library works on the
    context's stream, so the current stream's work on them (their making, or
    what their memory held before) ends first; the calls themselves return
    when they are done."""
    torch.cuda.current_stream().synchronize()
    ptr = [ctypes.cast(a.data_ptr(), ctypes.POINTER(ctypes.c_double)) if torch.is_tensor(a) else a for a in args]
    lbm._check(ctx, getattr(lbm.load(), fn)(ctx.h, *ptr))


class ForcedFclb(torch.autograd.Function):
    @staticmethod
    def forward(fctx, F, ctx, f0, T, every):
        NX, NY, NZ = ctx.dims(0)
        if F.numel() < 3 * ctx.ncells(0):
            raise ValueError("F holds %d values, the grid needs %d" % (F.numel(), 3 * ctx.ncells(0)))
        lbm.lbm_set_state(ctx, 0, np.asarray(f0, dtype=np.float64))
        in_place = _in_place(F)
        if in_place:
            Fd = _plain(F)
            _call("lbm_set_force", ctx, Fd)
        else:
            lbm.lbm_set_force(ctx, F.detach().cpu().double().numpy())
        lbm.lbm_adjoint_forward(ctx, T, every)
        if in_place:
            fT = torch.empty((ctx.Q, NZ, NY, NX), dtype=torch.float64, device=F.device)
            _call("lbm_get_state", ctx, 0, fT, fT.numel())
        else:
            fT = torch.from_numpy(lbm.lbm_get_state(ctx, 0))
        fctx.lbm_ctx = ctx
        fctx.generation = lbm.lbm_adjoint_generation(ctx)[0]
        return fT.to(device=F.device, dtype=F.dtype)

    @staticmethod
    def backward(fctx, grad_fT):
        if lbm.lbm_adjoint_generation(fctx.lbm_ctx)[0] != fctx.generation:
            raise RuntimeError("the lbm context has recorded another adjoint forward (or its force "
                               "changed) since this node's forward; run each forward's backward "
                               "before the next forward on the same context")
        ctx = fctx.lbm_ctx
        if _in_place(grad_fT):
            NX, NY, NZ = ctx.dims(0)
            lam = _plain(grad_fT)
            g = torch.empty((3, NZ, NY, NX), dtype=torch.float64, device=grad_fT.device)
            _call("lbm_adjoint_backward", ctx, lam, g)
        else:
            g = torch.from_numpy(lbm.lbm_adjoint_backward(ctx, grad_fT.detach().cpu().double().numpy()))
        return g.to(device=grad_fT.device, dtype=grad_fT.dtype), None, None, None, None


def forced_fclb(F, ctx, f0, T, every):
    """f_T of T forced FCLB steps from f0, differentiable w.r.t. F."""
    return ForcedFclb.apply(F, ctx, f0, T, every)
