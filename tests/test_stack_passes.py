"""Book-keeping of DepthStream's backward passes, without a GPU: the C-ABI calls are replaced by a small linear operator with
exact bf16 values (O = Q + K + V + sum_i c(l, i) (Kd_i + 2 Vd_i)) on a cache of plain [slot][K, V][B][T][H_kv][d] tensors, and
memory that the stream does not fill holds NaN.  What is checked is which calls write, add to and read which slots."""
import pytest
import torch

import paper_2603_15619_b200 as moda
from paper_2603_15619_b200 import binding

B, T, H, D, DM = 1, 3, 2, 4, 6
SLOT = 2 * B * T * H * D


def coef(l, i):
    return 1.0 + (l + i) % 3


def slots_of(cache):
    return cache.view(-1, 2, B, T, H, D)


class Operator:
    """The calls that stack.py makes.  ``fail_at``: number of the backward call that raises before it writes anything."""

    def __init__(self, monkeypatch):
        self.calls, self.fail_at, self.names = 0, None, []
        nan = lambda t, **kw: torch.full(t.shape, float("nan"), dtype=t.dtype)
        monkeypatch.setattr(torch, "empty_like", nan)
        monkeypatch.setattr(binding, "moda_depth_cache_bytes", lambda *a: 2 * SLOT * a[-1])
        monkeypatch.setattr(binding, "alloc_depth_cache", lambda *a: torch.full((SLOT * a[4],), float("nan"), dtype=torch.bfloat16))
        for name in ("moda_attn_fwd_append", "moda_attn_bwd_gqa", "moda_attn_bwd_gqa_slot", "moda_depth_cache_append", "moda_depth_cache_unpack",
                     "moda_kv_project_append"):
            monkeypatch.setattr(binding, name, getattr(self, name))

    def moda_attn_fwd_append(self, Q, K, V, depth, l, scale, cache, slot):
        O = Q + K + V
        for i in range(l):
            O = O + coef(l, i) * (slots_of(depth)[i, 0] + 2 * slots_of(depth)[i, 1])
        self.moda_depth_cache_append(cache, slot, K, V)
        return O, torch.zeros(B, H, T)

    def backward_call(self, name):
        self.calls += 1
        self.names.append(name)
        if self.calls == self.fail_at:
            raise moda.ModaError(-2, name)

    def moda_attn_bwd_gqa(self, Q, K, V, depth, O, dO, LSE, l, scale, d_depth_kv=None):
        self.backward_call("moda_attn_bwd_gqa")
        for i in range(l):
            slots_of(d_depth_kv)[i].copy_(torch.stack([coef(l, i) * dO, 2 * coef(l, i) * dO]))
        return dO.clone(), dO.clone(), dO.clone(), d_depth_kv

    def moda_attn_bwd_gqa_slot(self, Q, K, V, depth, O, dO, LSE, l, scale, d_depth_kv, slot):
        self.backward_call("moda_attn_bwd_gqa_slot")
        assert slot >= l
        for i in range(l):
            slots_of(d_depth_kv)[i].add_(torch.stack([coef(l, i) * dO, 2 * coef(l, i) * dO]))
        left = slots_of(d_depth_kv)[slot]
        return dO.clone(), dO + left[0], dO + left[1]

    def moda_depth_cache_append(self, cache, slot, K, V):
        slots_of(cache)[slot] = torch.stack([K, V]).detach()

    def moda_depth_cache_unpack(self, cache, slot, K, V):
        K.copy_(slots_of(cache[:SLOT * (slot + 1)])[slot, 0])
        V.copy_(slots_of(cache[:SLOT * (slot + 1)])[slot, 1])

    def moda_kv_project_append(self, X, Wk, Wv, H_kv, cache, slot, store_kv):
        self.moda_depth_cache_append(cache, slot, (X @ Wk.t()).view(B, T, H, D), (X @ Wv.t()).view(B, T, H, D))


KINDS = ("attend", "write", "attend", "project", "attend", "write")


class Stack:
    """attend, write, attend, project_write, attend, and a last slot that nothing attends to."""

    def __init__(self):
        g = torch.Generator().manual_seed(3)
        new = lambda *s: torch.randint(-1, 2, s, generator=g).to(torch.bfloat16).requires_grad_()
        shapes = {"attend": [(B, T, H, D)] * 3, "write": [(B, T, H, D)] * 2, "project": [(B, T, DM), (H * D, DM), (H * D, DM)]}
        self.inputs = [[new(*s) for s in shapes[kind]] for kind in KINDS]
        self.dO = [new(B, T, H, D).detach() for kind in KINDS if kind == "attend"]
        self.leaves = [x for group in self.inputs[:-1] for x in group]

    def run(self):
        stream = moda.DepthStream(B, T, H, D, len(KINDS), device="cpu")
        outs = []
        for kind, x in zip(KINDS, self.inputs):
            out = {"attend": stream.attend, "write": stream.write, "project": stream.project_write}[kind](*x)
            if kind == "attend":
                outs.append(out)
        return stream, outs

    def reference(self):
        """The same outputs from plain torch operations."""
        slots, outs = [], []
        for kind, x in zip(KINDS, self.inputs):
            if kind == "attend":
                Q, K, V = (t.float() for t in x)
                l = len(slots)
                outs.append(Q + K + V + sum(coef(l, i) * (k + 2 * v) for i, (k, v) in enumerate(slots)))
            elif kind == "write":
                K, V = (t.float() for t in x)
            else:
                X, Wk, Wv = (t.float() for t in x)
                K, V = ((X @ W.t()).view(B, T, H, D) for W in (Wk, Wv))
            slots.append((K, V))
        return outs

    def grads(self, which, leaves=None):
        return torch.autograd.grad([self.reference()[i] for i in which], leaves or self.leaves, [self.dO[i].float() for i in which],
                                   allow_unused=True)


def check(got, want):
    for a, b in zip(got, want, strict=True):
        b = torch.zeros_like(a, dtype=torch.float32, memory_format=torch.preserve_format) if b is None else b
        assert torch.equal(torch.zeros(a.shape) if a is None else a.float(), b)


@pytest.fixture
def op(monkeypatch):
    return Operator(monkeypatch)


def run_pass(stack, outs, which, **kw):
    return torch.autograd.grad([outs[i] for i in which], stack.leaves, [stack.dO[i] for i in which], allow_unused=True, **kw)


def test_forward_is_the_reference(op):
    stack = Stack()
    check(stack.run()[1], stack.reference())


@pytest.mark.parametrize("order", [[(0, 1, 2)], [(0, 1, 2), (0, 1, 2)], [(1,), (0, 1, 2)], [(2,), (1,), (0,)], [(1,), (2,)], [(0,), (1, 2), (0, 2)]])
def test_passes_over_one_stream_do_not_see_each_other(op, order):
    stack = Stack()
    _, outs = stack.run()
    for which in order:
        want = [torch.zeros(x.shape) if w is None else w for x, w in zip(stack.leaves, stack.grads(which))]
        got = [torch.zeros(x.shape) if g is None else g for x, g in zip(stack.leaves, run_pass(stack, outs, which, retain_graph=True))]
        check(got, want)


def test_layers_below_the_first_take_up_their_slot_in_their_backward_call(op):
    stack = Stack()
    _, outs = stack.run()
    run_pass(stack, outs, (0, 1, 2))
    assert op.names == ["moda_attn_bwd_gqa", "moda_attn_bwd_gqa_slot", "moda_attn_bwd_gqa_slot"]


@pytest.mark.parametrize("fail_at", [1, 2, 3])
def test_a_pass_after_one_that_failed(op, fail_at):
    stack = Stack()
    _, outs = stack.run()
    op.fail_at = fail_at
    with pytest.raises(moda.ModaError):
        run_pass(stack, outs, (0, 1, 2), retain_graph=True)
    check(run_pass(stack, outs, (0, 1, 2)), stack.grads((0, 1, 2)))


def test_a_pass_inside_another(op):
    """A hook in the middle of a pass runs a pass of its own over the same stream."""
    stack = Stack()
    _, outs = stack.run()
    inner, entered = [], []

    def hook(_):
        if not entered:
            entered.append(True)
            inner.extend(run_pass(stack, outs, (1, 2), retain_graph=True))
    handle = stack.inputs[4][0].register_hook(hook)
    outer = run_pass(stack, outs, (0, 1, 2), retain_graph=True)
    handle.remove()
    check(outer, stack.grads((0, 1, 2)))
    assert inner
    want = [torch.zeros(x.shape) if w is None else w for x, w in zip(stack.leaves, stack.grads((1, 2)))]
    check([torch.zeros(x.shape) if g is None else g for x, g in zip(stack.leaves, inner)], want)


def test_caches_that_the_caller_reads_replaces_or_fills(op):
    stack = Stack()
    stream, outs = stack.run()
    n = len(KINDS)
    mine = stream.cache.clone()
    stream.cache = mine                                    # the nodes use it from now on
    assert stream._slots.cache is mine and stream.cache is mine
    assert torch.equal(stream.grad_cache, torch.zeros(n * SLOT))
    slots_of(stream.grad_cache)[1].fill_(3.0)              # a gradient from elsewhere for the slot of the first write
    got = run_pass(stack, outs, (0, 1, 2), retain_graph=True)
    want = [w.clone() for w in stack.grads((0, 1, 2))]
    for i in (3, 4):
        want[i] += 3.0
    check(got, want)
    check(run_pass(stack, outs, (0, 1, 2), retain_graph=True), stack.grads((0, 1, 2)))
    full = slots_of(stream.grad_cache)
    assert bool((full[4:] == 0).all()) and torch.equal(full[3, 0].float(), coef(4, 3) * stack.dO[2].float())
    assert stream.slot_has_grad(n - 2) and not stream.slot_has_grad(n - 1)
    seed = torch.zeros(n * SLOT, dtype=torch.bfloat16)
    slots_of(seed)[1].fill_(-2.0)
    stream.grad_cache = seed
    want = [w.clone() for w in stack.grads((0, 1, 2))]
    for i in (3, 4):
        want[i] -= 2.0
    check(run_pass(stack, outs, (0, 1, 2)), want)
    assert stream.grad_cache is seed


def test_one_layer_alone(op):
    stream = moda.DepthStream(B, T, H, D, 1, device="cpu")
    x = [torch.ones(B, T, H, D, dtype=torch.bfloat16, requires_grad=True) for _ in range(3)]
    stream.attend(*x).sum().backward()
    assert all(torch.equal(t.grad, torch.ones_like(t.detach()).fill_(1.0)) for t in x)
    assert bool((stream.grad_cache == 0).all())
