"""Depth stream of a stack of attention layers, differentiable end to end.

In a MoDA model (paper Sec. 2.2, the "write" step) every attention layer appends its own K, V to
the depth stream after attending, and layer l attends to the l slots written before it.  So K_i, V_i
of layer i receive gradient from layer i's own sequence attention and, as depth slot i, from every
later layer.  ``DepthStream`` owns the depth cache and wires those contributions together around the
C-ABI calls; it is plumbing: no arithmetic of the operator happens here.

    stream = DepthStream(B, T, H_kv, d, n_layers)
    for layer in layers:
        q, k, v = layer.project(x)               # [B,T,H,d], [B,T,H_kv,d], [B,T,H_kv,d]
        o = stream.attend(q, k, v)               # attends to the slots so far, then appends k, v
        x = layer.rest(x, o)

A token tensor chains the calls: the token behind slot l stands for the first l + 1 slots of the depth
cache, and its gradient is a gradient cache of that many slots.  Backward runs the layers in reverse.
The first layer of a pass writes its depth gradients into a new buffer, every layer below adds its own to
slots < l of that buffer in place and takes slot l, which by then holds the contributions of all later
layers, as part of the gradient of its own K, V (moda_attn_bwd_gqa_slot does both).  Because the buffer
travels as a gradient, passes over one stream do not see each other, also when one failed half way.
"""
from __future__ import annotations

import torch

from . import binding


class _Attend(torch.autograd.Function):
    @staticmethod
    def forward(ctx, Q, K, V, token, slots, l, scale):
        Q, K, V = Q.contiguous(), K.contiguous(), V.contiguous()
        # attention and the "write" step (slot l = this layer's K, V) in one launch
        O, LSE = binding.moda_attn_fwd_append(Q, K, V, slots.cache if l > 0 else None, l, scale, slots.cache, l)
        ctx.save_for_backward(Q, K, V, O, LSE)
        ctx.slots, ctx.l, ctx.scale = slots, l, scale
        ctx.set_materialize_grads(False)                       # a token without a gradient is the start of a pass
        return O, slots.token(l + 1)

    @staticmethod
    def backward(ctx, dO, dtoken):
        Q, K, V, O, LSE = ctx.saved_tensors
        slots, l = ctx.slots, ctx.l
        dO = torch.zeros_like(O) if dO is None else dO.contiguous()
        # slots < l of the gradient cache receive this layer's share
        grads, filled = slots.open(dtoken, l)
        args = (Q, K, V, slots.cache if l > 0 else None, O, dO, LSE, l, ctx.scale)
        if filled:                                             # later layers attended to slot l: added where dK, dV are stored
            dQ, dK, dV = binding.moda_attn_bwd_gqa_slot(*args, grads, l)
        else:
            dQ, dK, dV, _ = binding.moda_attn_bwd_gqa(*args, d_depth_kv=grads if l > 0 else None)
        return dQ, dK, dV, slots.close(grads, filled, l), None, None, None


class _Write(torch.autograd.Function):
    """A slot written without attending (the FFN-side depth K/V of Sec. 2.2): its gradient is the
    slot of the gradient cache that the later layers filled."""

    @staticmethod
    def forward(ctx, K, V, token, slots, slot):
        K, V = K.contiguous(), V.contiguous()
        binding.moda_depth_cache_append(slots.cache, slot, K, V)
        ctx.slots, ctx.slot = slots, slot
        ctx.save_for_backward(K, V)
        ctx.set_materialize_grads(False)
        return slots.token(slot + 1)

    @staticmethod
    def backward(ctx, dtoken):
        K, V = ctx.saved_tensors
        slots, slot = ctx.slots, ctx.slot
        dK, dV = torch.zeros_like(K), torch.zeros_like(V)
        grads, filled = slots.open(dtoken, slot)
        if filled:
            binding.moda_depth_cache_unpack(grads, slot, dK, dV)
        return dK, dV, slots.close(grads, filled, slot) if filled else None, None, None


class _ProjectWrite(torch.autograd.Function):
    """A slot produced by a key / value projection of X (Sec. 2.2: an FFN layer obtains its depth pair through a KV
    projection of its input) and written by the projection's own epilogue: one launch, K and V never stored.  Backward:
    the slot of the gradient cache is dK, dV; dX = dK Wk + dV Wv and dW = dK^T X are plain library GEMMs."""

    @staticmethod
    def forward(ctx, X, Wk, Wv, token, slots, slot):
        X, Wk, Wv = X.contiguous(), Wk.contiguous(), Wv.contiguous()
        binding.moda_kv_project_append(X, Wk, Wv, slots.shape[2], cache=slots.cache, slot=slot, store_kv=False)
        ctx.slots, ctx.slot = slots, slot
        ctx.save_for_backward(X, Wk, Wv)
        ctx.set_materialize_grads(False)
        return slots.token(slot + 1)

    @staticmethod
    def backward(ctx, dtoken):
        X, Wk, Wv = ctx.saved_tensors
        slots, slot = ctx.slots, ctx.slot
        B, T, Hk, d = slots.shape
        grads, filled = slots.open(dtoken, slot)
        if not filled:
            return torch.zeros_like(X), torch.zeros_like(Wk), torch.zeros_like(Wv), None, None, None
        dK = torch.empty((B, T, Hk, d), dtype=X.dtype, device=X.device)
        dV = torch.empty_like(dK)
        binding.moda_depth_cache_unpack(grads, slot, dK, dV)
        dK2, dV2, X2 = dK.view(B * T, Hk * d), dV.view(B * T, Hk * d), X.view(B * T, -1)
        dX = (dK2 @ Wk).addmm_(dV2, Wv).view_as(X)
        return dX, dK2.t() @ X2, dV2.t() @ X2, slots.close(grads, filled, slot), None, None


class _Slots:
    """What a stream's autograd nodes share: the depth cache, and the gradient cache of the latest pass.  Kept apart from the
    DepthStream, whose token leads back to the nodes: a node that held the stream itself would close a reference cycle,
    and the caches would then live until the garbage collector happens to run."""

    def __init__(self, B, T, H_kv, d, n_layers, device):
        self.shape = (B, T, H_kv, d)
        self.n_layers = n_layers
        self.slot_elems = binding.moda_depth_cache_bytes(B, T, H_kv, d, 1) // 2
        self.cache = binding.alloc_depth_cache(B, T, H_kv, d, n_layers, device)
        self.grads = None                                      # gradient cache of the latest pass
        self.grad_slots = 0                                    # slots of it that hold something
        self.seeded = False                                    # it is the caller's: the next pass adds to it

    def token(self, n):
        """A tensor of the first n slots' shape without their memory."""
        return torch.empty_strided((n * self.slot_elems,), (0,), dtype=self.cache.dtype, device=self.cache.device)

    def open(self, dtoken, slot):
        """(buffer, filled) for the node of slot ``slot``: a gradient cache that it may write in place, and whether slots
        0 .. ``slot`` of it hold gradients.  ``dtoken`` is what the nodes above passed down, None at the start of a pass."""
        if dtoken is None:
            if self.seeded:
                return self.grads, True
            self.grads, self.grad_slots = None, 0              # the previous pass's: its memory may serve this one
            return torch.empty_like(self.cache) if slot > 0 else None, False
        if self.grads is not None and dtoken.data_ptr() == self.grads.data_ptr():
            return self.grads, True
        grads = torch.empty_like(self.cache)                   # a gradient from elsewhere: not ours to write to
        grads[:dtoken.numel()].copy_(dtoken)
        return grads, True

    def close(self, grads, filled, slot):
        """The gradient of the token below slot ``slot``, once the node's own share is in ``grads``."""
        if grads is not self.grads:
            self.grads, self.grad_slots = grads, slot + 1 if filled else slot
        self.seeded = False
        return grads[:slot * self.slot_elems] if slot > 0 else None


class DepthStream:
    """Depth cache of one forward pass through a stack, and the gradient of its slots.

    ``cache`` may be replaced by another depth cache of the same size.  ``grad_cache`` is the gradient cache of the latest
    backward pass; before the first one it is zero, and what the caller adds to it then, or a gradient cache that the caller
    assigns, is where the next pass starts from."""

    def __init__(self, B, T, H_kv, d, n_layers, device="cuda"):
        self.shape = (B, T, H_kv, d)
        self.n_layers = int(n_layers)
        self._slots = _Slots(B, T, H_kv, d, self.n_layers, device)
        self.n_written = 0
        self.token = self._slots.token(0).requires_grad_()

    @property
    def cache(self):
        return self._slots.cache

    @cache.setter
    def cache(self, cache):
        self._slots.cache = cache

    @property
    def grad_cache(self):
        """Gradient cache of the latest backward pass, zero in the slots that it did not reach."""
        s = self._slots
        if s.grads is None:
            self.grad_cache = torch.zeros_like(s.cache)
        elif s.grad_slots < self.n_layers:
            s.grads[s.grad_slots * s.slot_elems:].zero_()
            s.grad_slots = self.n_layers
        return s.grads

    @grad_cache.setter
    def grad_cache(self, grads):
        s = self._slots
        s.grads, s.grad_slots, s.seeded = grads, self.n_layers, True

    def slot_has_grad(self, l):
        return l < self.n_written - 1

    def attend(self, Q, K, V, scale=None):
        """MoDA attention of the next layer: attends to the slots written so far, then appends K, V."""
        l = self.n_written
        if l >= self.n_layers:
            raise ValueError("more layers than the stream was sized for")
        if scale is None:
            scale = Q.shape[-1] ** -0.5
        O, self.token = _Attend.apply(Q, K, V, self.token, self._slots, l, float(scale))
        self.n_written = l + 1
        return O

    def write(self, K, V):
        """Appends K, V [B,T,H_kv,d] as the next slot without attending (e.g. an FFN layer's depth K/V)."""
        slot = self.n_written
        if slot >= self.n_layers:
            raise ValueError("more slots than the stream was sized for")
        self.token = _Write.apply(K, V, self.token, self._slots, slot)
        self.n_written = slot + 1

    def project_write(self, X, Wk, Wv):
        """Appends K = X Wk^T, V = X Wv^T (X [B,T,D_model], W [H_kv d, D_model]) as the next slot without attending:
        the projection kernel writes the slot from its epilogue."""
        slot = self.n_written
        if slot >= self.n_layers:
            raise ValueError("more slots than the stream was sized for")
        self.token = _ProjectWrite.apply(X, Wk, Wv, self.token, self._slots, slot)
        self.n_written = slot + 1
