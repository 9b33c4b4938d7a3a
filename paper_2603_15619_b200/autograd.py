"""torch.autograd wrapper around the C ABI: one differentiable call per attention layer.

Plumbing only: forward and backward are single calls into the CUDA library (moda_attn_fwd_gqa /
moda_attn_bwd_gqa; plain multi-head attention is the H_kv == H case).  The depth cache is passed
and differentiated in cache layout: the gradient of ``depth_kv`` has the layout of the cache
(kv = 0 holds dKd, kv = 1 holds dVd, slots >= l are zero), so that a stack of layers can add it to
the gradients of the layers that wrote those slots (moda_depth_cache_unpack turns a slot back into
[B, T, H_kv, d] tensors).
"""
from __future__ import annotations

import torch

from . import binding


class _ModaAttention(torch.autograd.Function):
    @staticmethod
    def forward(ctx, Q, K, V, depth_kv, l, scale):
        Q, K, V = Q.contiguous(), K.contiguous(), V.contiguous()
        O, LSE = binding.moda_attn_fwd_gqa(Q, K, V, depth_kv if l > 0 else None, l, scale)
        ctx.save_for_backward(Q, K, V, depth_kv if l > 0 else None, O, LSE)
        ctx.l, ctx.scale = int(l), float(scale)
        ctx.mark_non_differentiable(LSE)
        ctx.set_materialize_grads(False)                       # nothing to fill for LSE
        return O, LSE

    @staticmethod
    def backward(ctx, dO, _dLSE):
        Q, K, V, depth_kv, O, LSE = ctx.saved_tensors
        B, T, H, d = Q.shape
        Hk = K.shape[2]
        l = ctx.l
        if dO is None:
            dO = torch.zeros_like(O)
        d_cache = None
        if l > 0:
            # the kernels write every element of slots < l; later slots of the caller's cache get no gradient
            d_cache = torch.empty_like(depth_kv)
            slots = binding.moda_depth_cache_bytes(B, T, Hk, d, l) // 2
            if slots < depth_kv.numel():
                d_cache.view(-1)[slots:].zero_()
        dQ, dK, dV, _ = binding.moda_attn_bwd_gqa(Q, K, V, depth_kv, O, dO.contiguous(), LSE, l, ctx.scale,
                                                  d_depth_kv=d_cache)
        return dQ, dK, dV, d_cache, None, None


def moda_attention(Q, K, V, depth_kv=None, l=0, scale=None):
    """Differentiable MoDA attention of one layer.

    Q [B,T,H,d]; K, V [B,T,H_kv,d] (H_kv divides H); ``depth_kv`` a depth cache with H_kv heads
    holding at least ``l`` slots (see alloc_depth_cache / moda_depth_cache_append).  Returns
    O [B,T,H,d] and LSE [B,H,T] (LSE is not differentiable)."""
    if scale is None:
        scale = Q.shape[-1] ** -0.5
    if l > 0 and depth_kv is None:
        raise ValueError("depth_kv is required when l > 0")
    # the same two calls and saved tensors as a C++ node; None for anything but plain tensors outside of transforms, modes and tracers
    out = binding.host().attention(Q, K, V, depth_kv, l, scale)
    if out is not None:
        return out
    if depth_kv is None:
        depth_kv = Q.new_empty(0)
    return _ModaAttention.apply(Q, K, V, depth_kv, int(l), float(scale))
