"""torch.autograd.Function over the C ABI: D = forward(R, m, S_age); backward = the
hand-written straight-through adjoint (App. B of the paper: gradients through the
unrolled day loop, with the Gumbel-softmax relaxation of the infection draw)."""
from __future__ import annotations

import torch

from . import capi


class GabmFunction(torch.autograd.Function):
    """``GabmFunction.apply(ctx, R, m, S_age, n_seed) -> D``.

    R, m: [I, T] float32 CUDA tensors; S_age: [I, 9] float32; n_seed: ints per instance.
    D: [I, T] float64 daily new deaths.  The backward runs ``gabm_backward`` on the
    same ctx, so a ctx serves one forward/backward pair at a time.
    """

    @staticmethod
    def forward(fctx, handle, R, m, S_age, n_seed):
        T = int(R.shape[-1])
        D, _ = capi.gabm_forward(handle, T, R.detach().contiguous(), m.detach().contiguous(),
                                 S_age.detach().contiguous(), n_seed)
        fctx.handle = handle
        fctx.dtypes = (R.dtype, m.dtype, S_age.dtype)
        return D

    @staticmethod
    def backward(fctx, gD):
        gD = gD.detach().to(torch.float64).contiguous()
        (I, T), A = gD.shape, capi.GABM_NUM_AGES
        # one buffer, so that one conversion serves the three gradients
        flat = torch.empty(I * (2 * T + A), dtype=torch.float64, device=gD.device)
        dR, dm, dS = flat.split((I * T, I * T, I * A))
        capi.gabm_backward(fctx.handle, gD, dR.view(I, T), dm.view(I, T), dS.view(I, A))
        if len(set(fctx.dtypes)) == 1:
            dR, dm, dS = flat.to(fctx.dtypes[0]).split((I * T, I * T, I * A))
        else:
            dR, dm, dS = (x.to(t) for x, t in zip((dR, dm, dS), fctx.dtypes))
        return None, dR.view(I, T), dm.view(I, T), dS.view(I, A), None
