"""torch.autograd.Function over the acoustic forward model.

``acoustic_modeling(m, src_wav, ...)`` returns the receiver traces of
``acoustic_forward``; its backward pass returns the vector-Jacobian products
with respect to the squared slowness ``m`` (``acoustic_gradient``, the
adjoint-state FWI gradient with forward-wavefield checkpointing) and with
respect to the source wavelets (``acoustic_adjoint``), or both in one reverse
sweep (C ABI ``acoustic_vjp``).  Everything runs in the
library's CUDA kernels; this module only wires the calls into autograd.
"""
from __future__ import annotations

import torch

from . import (_as_grid, _empty_like_kind, _native, _ptr, _stream_for, acoustic_adjoint,
               acoustic_forward, acoustic_gradient)


def _vjp(grid, so, dt, nt, m, src_xyz, src_wav, rec_xyz, rec_resid, damp, checkpoint_every):
    """Gradients with respect to m and to the source wavelets in one reverse sweep
    (C ABI ``acoustic_vjp``): what acoustic_gradient and acoustic_adjoint return."""
    g = _as_grid(grid)
    nshots, nsrc = int(src_xyz.shape[0]), int(src_xyz.shape[1])
    nrec = int(rec_xyz.shape[1])
    if tuple(rec_resid.shape) != (nshots, nt, nrec):
        raise ValueError("rec_resid must be [nshots][nt][nrec]")
    grad = _empty_like_kind(m, tuple(g.shape))
    src_grad = _empty_like_kind(m, (nshots, nt, nsrc))
    st = _native.load().acoustic_vjp(
        g.struct(), int(so), float(dt), int(nt), nshots, _ptr(m, "m"), _ptr(damp, "damp"), nsrc,
        _ptr(src_xyz, "src_xyz"), _ptr(src_wav, "src_wav"), nrec, _ptr(rec_xyz, "rec_xyz"),
        _ptr(rec_resid, "rec_resid"), int(checkpoint_every), _ptr(grad, "grad"),
        _ptr(src_grad, "src_grad"), _stream_for(m, grad))
    _native.check(st)
    return grad, src_grad


class AcousticModeling(torch.autograd.Function):
    @staticmethod
    def forward(ctx, m, src_wav, grid, so, dt, src_xyz, rec_xyz, damp, checkpoint_every):
        m = m.contiguous()
        src_wav = src_wav.contiguous()
        nt = int(src_wav.shape[1])
        rec, _ = acoustic_forward(grid, so, dt, nt, m, src_xyz, src_wav, rec_xyz, damp=damp,
                                  return_final=False)
        ctx.save_for_backward(m, src_wav)
        ctx.cfg = (grid, so, dt, nt, src_xyz, rec_xyz, damp, checkpoint_every)
        return rec

    @staticmethod
    def backward(ctx, grad_rec):
        m, src_wav = ctx.saved_tensors
        grid, so, dt, nt, src_xyz, rec_xyz, damp, ck = ctx.cfg
        grad_rec = grad_rec.contiguous()
        gm = gq = None
        if ctx.needs_input_grad[0] and ctx.needs_input_grad[1]:  # one reverse sweep
            gm, gq = _vjp(grid, so, dt, nt, m, src_xyz, src_wav, rec_xyz, grad_rec, damp, ck)
        elif ctx.needs_input_grad[0]:
            gm = acoustic_gradient(grid, so, dt, nt, m, src_xyz, src_wav, rec_xyz, grad_rec,
                                   damp=damp, checkpoint_every=ck)
        elif ctx.needs_input_grad[1]:
            gq = acoustic_adjoint(grid, so, dt, nt, m, src_xyz, rec_xyz, grad_rec, damp=damp)
        return gm, gq, None, None, None, None, None, None, None


def acoustic_modeling(m, src_wav, grid, so, dt, src_xyz, rec_xyz, damp=None, checkpoint_every=0):
    """Differentiable receiver traces d(m, q) [nshots][nt][nrec]."""
    return AcousticModeling.apply(m, src_wav, grid, so, dt, src_xyz, rec_xyz, damp,
                                  checkpoint_every)
