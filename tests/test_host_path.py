"""The host path of the hot calls (csrc/moda_host.cpp): what it does not serve it hands back, and where it serves a call (GPU) the
results and the autograd behaviour are those of the general path."""
import pytest
import torch

import paper_2603_15619_b200 as moda
from paper_2603_15619_b200 import autograd, binding

gpu = pytest.mark.gpu
BF16 = torch.bfloat16


class _Refuses:
    """Stands in for the extension: every call takes the general path."""

    def __getattr__(self, name):
        return lambda *a: None


@pytest.fixture
def general(monkeypatch):
    """Runs a function on the general path."""
    def run(f, *a, **k):
        with monkeypatch.context() as m:
            m.setattr(binding, "host", lambda: _Refuses())
            return f(*a, **k)
    return run


def test_what_is_not_plain_is_handed_back():
    host = binding.host()
    x = torch.zeros(1, 4, 2, 64, dtype=BF16)
    m = torch.empty(1, 4, 2, 64, dtype=BF16, device="meta")
    for t in (x, m, None, 3):
        assert host.attention(t, t, t, None, 0, 0.1) is None
        assert host.attn_fwd(t, t, t, None, 0, 0.1, None, 0, None, None) is None
        assert host.attn_bwd(t, t, t, None, t, t, t, 0, 0.1, None, None, None, None, None, None) is None
        assert host.decode(t, t, t, None, None, None, 4, 0, 0.1, None, None, None) is None
    assert host.decode() is None and host.attention() is None


def _qkv(B, T, H, Hk, d, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    new = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=BF16)
    return new(B, T, H, d), new(B, T, Hk, d), new(B, T, Hk, d), new(B, T, H, d)


def _cache(B, T, Hk, d, l, slots=None):
    cache = moda.alloc_depth_cache(B, T, Hk, d, slots or max(l, 1))
    for i in range(l):
        _, K, V, _ = _qkv(B, T, Hk, Hk, d, 10 + i)
        moda.moda_depth_cache_append(cache, i, K, V)
    return cache


def _same(a, b, loose=()):
    assert len(a) == len(b)
    for i, (x, y) in enumerate(zip(a, b)):
        if x is None or y is None:
            assert x is None and y is None
        elif i in loose:                                   # dQ: the order of its fp32 additions is not fixed
            assert (x.float() - y.float()).norm() <= 1e-3 * y.float().norm() + 1e-6
        else:
            assert torch.equal(x, y), i


@gpu
@pytest.mark.parametrize("B,T,H,Hk,d,l", [(1, 1, 1, 1, 64, 0), (2, 129, 4, 2, 64, 3), (1, 300, 2, 2, 128, 5)])
def test_layer_calls_agree_with_the_general_path(general, B, T, H, Hk, d, l):
    Q, K, V, dO = _qkv(B, T, H, Hk, d)
    cache = _cache(B, T, Hk, d, l, l + 1)
    other = cache.clone()
    O, LSE = moda.moda_attn_fwd_append(Q, K, V, cache, l, 0.125, cache, l)
    _same((O, LSE), general(moda.moda_attn_fwd_append, Q, K, V, other, l, 0.125, other, l))
    assert torch.equal(cache[:other.numel()], other)
    _same(moda.moda_attn_fwd_gqa(Q, K, V, cache, l, 0.125), (O, LSE))
    given = torch.empty_like(O), torch.empty_like(LSE)
    got = moda.moda_attn_fwd_gqa(Q, K, V, cache, l, 0.125, O=given[0], LSE=given[1])
    assert got[0] is given[0] and got[1] is given[1] and torch.equal(given[0], O)
    for stages in (None, moda.MODA_BWD_ALL_STAGES, moda.MODA_BWD_ALL_STAGES | moda.MODA_BWD_DETERMINISTIC):
        a = moda.moda_attn_bwd_gqa(Q, K, V, cache, O, dO, LSE, l, 0.125, stages=stages)
        b = general(moda.moda_attn_bwd_gqa, Q, K, V, cache, O, dO, LSE, l, 0.125, stages=stages)
        _same(a, b, loose=(0,))
    assert moda.moda_last_status() == 0


@gpu
@pytest.mark.parametrize("form", ["plain", "varlen", "paged"])
def test_decode_agrees_with_the_general_path(general, form):
    B, T, H, Hk, d, l = 3, 200, 4, 2, 64, 2
    g = torch.Generator(device="cuda").manual_seed(1)
    new = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=BF16)
    q, depth, lens = new(B, H, d), new(l, B, Hk, 2, d), torch.tensor([1, 77, 200], dtype=torch.int32, device="cuda")
    if form == "paged":
        args = (moda.moda_attn_decode_paged, q, new(12, 64, Hk, d), new(12, 64, Hk, d), torch.arange(12, dtype=torch.int32, device="cuda").view(3, 4), lens)
    elif form == "varlen":
        args = (moda.moda_attn_decode_varlen, q, new(B, T, Hk, d), new(B, T, Hk, d), lens)
    else:
        args = (moda.moda_attn_decode, q, new(B, T, Hk, d), new(B, T, Hk, d))
    f, rest = args[0], (*args[1:], depth, T, l, 0.125)
    _same(f(*rest), general(f, *rest))
    with pytest.raises(moda.ModaError) as here:             # errors of the C call come as they did
        f(*rest[:-1], -1.0)
    with pytest.raises(moda.ModaError) as there:
        general(f, *rest[:-1], -1.0)
    assert here.value.code == there.value.code and str(here.value) == str(there.value)


def _errors(f):
    try:
        f()
    except Exception as e:
        return type(e)
    return None


@gpu
def test_wrong_arguments_are_refused_as_before(general):
    Q, K, V, dO = _qkv(1, 64, 2, 2, 64)
    bad = [lambda: moda.moda_attn_fwd_gqa(Q.float(), K, V, None, 0, 0.1), lambda: moda.moda_attn_fwd_gqa(Q.transpose(1, 2), K, V, None, 0, 0.1),
           lambda: moda.moda_attn_fwd_gqa(Q, K[:, :32], V, None, 0, 0.1), lambda: moda.moda_attn_fwd_gqa(Q, K, V, None, 3, 0.1),
           lambda: moda.moda_attn_fwd_gqa(Q, K.cpu(), V, None, 0, 0.1), lambda: moda.moda_attn_fwd_gqa(Q, K, V, None, 0, 0.0),
           lambda: moda.moda_attn_fwd_gqa(Q.transpose(2, 3), K, V, None, 0, 0.1), lambda: moda.moda_attn_fwd_gqa(Q[..., :32], K[..., :32], V[..., :32], None, 0, 0.1),
           lambda: moda.moda_attention(Q, K, V, None, 2), lambda: moda.moda_attention(Q, K.float(), V), lambda: moda.moda_attn_fwd_gqa(Q, K, V, None, -1, 0.1),
           lambda: moda.moda_attn_fwd_append(Q, K, V, None, 0, 0.1, None, 0), lambda: moda.moda_attn_decode(Q[:, 0], K, V, None, 65, 0, 0.1)]
    # backward: no gradient cache for 257 slots or 32 features, a scale, a stage mask, tensors that are missing or of another type or strides
    LSE, cache = torch.zeros(1, 2, 64, device="cuda"), _cache(1, 64, 2, 64, 2, 3)
    narrow = [t[..., :32].contiguous() for t in (Q, K, V)]
    bwd = lambda q=Q, k=K, v=V, depth=cache, O=dO, g=dO, lse=LSE, l=1, scale=0.1, **kw: moda.moda_attn_bwd_gqa(q, k, v, depth, O, g, lse, l, scale, **kw)
    slot = lambda g=dO, l=1, grads=cache, at=2, **kw: moda.moda_attn_bwd_gqa_slot(Q, K, V, cache, dO, g, LSE, l, 0.1, grads, at, **kw)
    bad += [lambda: bwd(l=257), lambda: bwd(*narrow, O=narrow[0], g=narrow[0]), lambda: bwd(l=-1), lambda: bwd(scale=-1.0), lambda: bwd(stages=0),
            lambda: bwd(stages=64), lambda: bwd(depth=None), lambda: bwd(O=None), lambda: bwd(g=dO.cpu()), lambda: bwd(g=dO.transpose(1, 2)),
            lambda: bwd(q=Q.float()), lambda: bwd(k=K[:, :32]), lambda: bwd(l=257, d_depth_kv=cache), lambda: bwd(workspace=LSE),
            lambda: slot(at=0), lambda: slot(at=-1), lambda: slot(at=256), lambda: slot(grads=None), lambda: slot(l=257), lambda: slot(g=dO.cpu()),
            lambda: slot(workspace=LSE)]
    for i, f in enumerate(bad):
        want = general(_errors, f)
        assert want is not None and _errors(f) is want, (i, want, _errors(f))


def _short(t):
    return t.flatten()[:-1]


def test_buffers_are_looked_at_before_their_address_is_taken():
    """In host memory the check of the size and the type comes before the one of the device."""
    x = torch.zeros(8, dtype=BF16)
    for f, text in ((lambda: binding._bf16(x, 9), "9 elements"), (lambda: binding._bf16(x.float(), 8), "torch.bfloat16"), (lambda: binding._f32(x, 8), "torch.float32"),
                    (lambda: binding._bf16(x, 8), "CUDA"), (lambda: binding._slots(x, 1, 1, 64, 2, 64), "65536 bytes"),
                    (lambda: binding._slots(x, 257, 1, 64, 2, 64), "CUDA"), (lambda: binding._slots(x, -3, 1, 64, 2, 64), "CUDA"),
                    (lambda: binding._slots(x, 1, 1, 64, 2, 64, e4m3=True), "bytes"), (lambda: binding._token(x, 2, 3, 2, 64), "1536 elements")):
        with pytest.raises(ValueError, match=text):
            f()
    assert binding._bf16(None, 9) is None and binding._slots(None, 1, 1, 64, 2, 64) is None
    for B, T, H, d, n in ((1, 1, 1, 64, 1), (2, 128, 3, 128, 4), (3, 129, 2, 64, 256), (1, 1000, 16, 128, 7)):
        for e4m3, size in ((False, moda.moda_depth_cache_bytes(B, T, H, d, n)), (True, moda.moda_depth_cache_e4m3_bytes(B, T, H, d, n))):
            for short, text in ((1, "take"), (0, "CUDA")):
                with pytest.raises(ValueError, match=text):
                    binding._slots(torch.empty(size - short, dtype=torch.uint8, device="meta"), n, B, T, H, d, e4m3=e4m3)


@gpu
def test_buffers_that_are_too_small_or_of_another_type_are_refused(general):
    Q, K, V, dO = _qkv(1, 64, 2, 2, 64)
    O, LSE, cache = torch.empty_like(Q), torch.zeros(1, 2, 64, device="cuda"), _cache(1, 64, 2, 64, 2, 3)
    cache8 = torch.zeros(moda.moda_depth_cache_e4m3_bytes(1, 64, 2, 64, 3), dtype=torch.uint8, device="cuda")
    two = cache[:cache.numel() // 3 * 2]
    q, tok, lens = Q[:, 0], torch.zeros(2, 1, 2, 2, 64, device="cuda", dtype=BF16), torch.tensor([9], dtype=torch.int32, device="cuda")
    table = torch.zeros(1, 1, dtype=torch.int32, device="cuda")
    scale = 0.125
    for wrong in (_short, lambda t: t.double()):
        few = _short if wrong is _short else lambda t: t[:t.numel() // 4]     # caches: any type, enough bytes
        calls = [lambda: moda.moda_attention(Q, K, V, few(two), 2),
                 lambda: moda.moda_attn_decode(q, K, V, tok, 64, 2, scale, O=wrong(q)), lambda: moda.moda_attn_decode(q, K, V, tok, 64, 2, scale, LSE=wrong(LSE[:, :, 0])),
                 lambda: moda.moda_attn_decode_varlen(q, K, V, lens, wrong(tok), 64, 2, scale), lambda: moda.moda_attn_decode_varlen(q, K, wrong(V), lens, tok, 64, 2, scale),
                 lambda: moda.moda_attn_decode_paged(q, K, wrong(V), table, lens, tok, 64, 2, scale), lambda: moda.moda_attn_decode_paged(q, K, V, table, lens, wrong(tok), 64, 2, scale),
                 lambda: moda.moda_depth_cache_append(few(two), 1, K, V), lambda: moda.moda_depth_cache_unpack(few(two), 1, O, O.clone()),
                 lambda: moda.moda_depth_cache_unpack_add(cache, 1, O, wrong(V)), lambda: moda.moda_depth_cache_append_e4m3(few(cache8), 2, K, V),
                 lambda: moda.moda_depth_slot_mass(Q, few(two), LSE, 2, scale), lambda: moda.moda_depth_slot_mass(Q, cache, wrong(LSE), 2, scale),
                 lambda: moda.moda_kv_project_append(K.view(1, 64, 128), torch.zeros(128, 128, device="cuda", dtype=BF16), torch.zeros(128, 128, device="cuda", dtype=BF16), 2,
                                                     cache=few(two), slot=1)]
        for f, depth in ((moda.moda_attn_fwd_gqa, two), (moda.moda_attn_fwd, two), (moda.moda_attn_fwd_prefill, two), (moda.moda_attn_fwd_e4m3, cache8)):
            l = 3 if depth is cache8 else 2
            calls += [lambda f=f, depth=depth, l=l: f(Q, K, V, few(depth), l, scale), lambda f=f, depth=depth, l=l: f(Q, K, V, depth, l, scale, O=wrong(O)),
                      lambda f=f, depth=depth, l=l: f(Q, K, V, depth, l, scale, LSE=wrong(LSE))]
        calls += [lambda: moda.moda_attn_fwd_append(Q, K, V, None, 0, scale, few(two), 1), lambda: moda.moda_attn_fwd_append_e4m3(Q, K, V, None, 0, scale, few(cache8), 2)]
        for f, depth in ((moda.moda_attn_bwd_gqa, two), (moda.moda_attn_bwd, two), (moda.moda_attn_bwd_e4m3, cache8)):
            l = 3 if depth is cache8 else 2
            calls += [lambda f=f, depth=depth, l=l: f(Q, K, V, few(depth), O, dO, LSE, l, scale), lambda f=f, depth=depth, l=l: f(Q, K, V, depth, wrong(O), dO, LSE, l, scale),
                      lambda f=f, depth=depth, l=l: f(Q, K, V, depth, O, wrong(dO), LSE, l, scale), lambda f=f, depth=depth, l=l: f(Q, K, V, depth, O, dO, wrong(LSE), l, scale),
                      lambda f=f, depth=depth, l=l: f(Q, K, V, depth, O, dO, LSE, l, scale, d_depth_kv=few(two))]
            calls += [lambda f=f, depth=depth, l=l, n=n: f(Q, K, V, depth, O, dO, LSE, l, scale, **{n: wrong(O)}) for n in ("dQ", "dK", "dV")]
        calls += [lambda: moda.moda_attn_bwd_gqa_slot(Q, K, V, two, O, dO, LSE, 1, scale, few(two), 1), lambda: moda.moda_attn_bwd_gqa_slot(Q, K, V, two, O, wrong(dO), LSE, 1, scale, two, 1)]
        for i, f in enumerate(calls):
            assert general(_errors, f) is ValueError and _errors(f) is ValueError, (wrong, i)
    torch.cuda.synchronize()
    assert moda.moda_last_status() == 0


@gpu
@pytest.mark.parametrize("l", [0, 2])
def test_differentiable_call_behaves_as_the_general_one(general, l):
    """Gradients, unused outputs, saved-tensor hooks, in-place changes, retained graphs, no_grad, inference mode, non-contiguous inputs,
    second derivatives, transforms."""
    def leaves():
        Q, K, V, dO = _qkv(1, 130, 4, 2, 64)
        x = [t.requires_grad_() for t in (Q, K, V)]
        cache = _cache(1, 130, 2, 64, 2, 3).requires_grad_() if l else None
        return x, cache, dO

    def grads():
        x, cache, dO = leaves()
        O, LSE = moda.moda_attention(*x, cache, l)
        assert O.requires_grad and not LSE.requires_grad
        wrt = x + ([cache] if l else [])
        first = torch.autograd.grad(O, wrt, dO, retain_graph=True)
        again = torch.autograd.grad(O, wrt, dO)
        with pytest.raises(RuntimeError, match="backward through the graph a second time"):
            torch.autograd.grad(O, wrt, dO)
        _same(first, again, loose=(0,))
        return [O, LSE, *first]

    _same(grads(), general(grads), loose=(2,))

    def hooks():
        x, cache, dO = leaves()
        seen = []
        with torch.autograd.graph.saved_tensors_hooks(lambda t: (seen.append(tuple(t.shape)), t.clone())[1], lambda t: t):
            O, _ = moda.moda_attention(*x, cache, l)
        O.backward(dO)
        return sorted(seen), [t.grad for t in x]

    a, b = hooks(), general(hooks)
    assert a[0] == b[0] and len(a[0]) == (6 if l else 5)
    _same(a[1], b[1], loose=(0,))

    def changed():
        x, cache, dO = leaves()
        y = [t * 1 for t in x]
        O, _ = moda.moda_attention(*y, cache, l)
        y[1].add_(1)
        O.backward(dO)

    assert general(_errors, changed) is RuntimeError and _errors(changed) is RuntimeError

    def others():
        x, cache, dO = leaves()
        with torch.no_grad():
            assert not moda.moda_attention(*x, cache, l)[0].requires_grad
        with torch.inference_mode():
            a = moda.moda_attention(*x, cache, l)[0]
            assert a.is_inference()
        t = [u.transpose(1, 2).contiguous().transpose(1, 2) for u in x]       # not contiguous
        b = moda.moda_attention(*t, cache, l)[0]
        assert torch.equal(a, b)
        g = torch.autograd.grad(moda.moda_attention(*x, cache, l)[0], x, dO, create_graph=True)
        return [b, *g], [u.requires_grad for u in g]

    a, b = others(), general(others)
    _same(a[0], b[0], loose=(1,))
    assert a[1] == b[1]

    def mapped():
        x, cache, dO = leaves()
        torch.func.vmap(lambda q: moda.moda_attention(q, x[1], x[2], cache, l)[0])(x[0][None])

    def dual():
        x, cache, dO = leaves()
        with torch.autograd.forward_ad.dual_level():
            moda.moda_attention(torch.autograd.forward_ad.make_dual(x[0], dO), x[1], x[2], cache, l)

    for f in (mapped, dual):
        assert _errors(f) is general(_errors, f) and _errors(f) is not None

    class Sub(torch.Tensor):
        pass

    def subclass():
        x, cache, dO = leaves()
        q = x[0].detach().as_subclass(Sub)
        return [type(t) for t in moda.moda_attn_fwd_gqa(q, x[1].detach(), x[2].detach(), cache, l, 0.1)]

    assert subclass() == general(subclass)
    assert moda.moda_last_status() == 0


UNPACKED = {"host memory": lambda t: t.cpu(), "strides": lambda t: t.repeat_interleave(2, -1)[..., ::2], "type": lambda t: t.double(),
            "size": lambda t: t.flatten()[:t.numel() // 2], "shape": lambda t: t.flatten()[:64]}


@gpu
@pytest.mark.parametrize("how", UNPACKED)
def test_what_a_saved_tensor_hook_hands_back_is_looked_at(how):
    """Refused before anything is launched, whichever of the six saved tensors it is."""
    for which in range(6):
        x, cache = [t.requires_grad_() for t in _qkv(1, 130, 4, 2, 64)[:3]], _cache(1, 130, 2, 64, 2, 3)
        seen = []
        pack = lambda t: (seen.append(t), len(seen) - 1)[1]
        unpack = lambda i: UNPACKED[how](seen[i].detach()) if i == which else seen[i]
        with torch.autograd.graph.saved_tensors_hooks(pack, unpack):
            O, _ = moda.moda_attention(*x, cache, 2)
        assert len(seen) == 6
        with pytest.raises(ValueError):
            O.backward(torch.ones_like(O))
    assert moda.moda_last_status() == 0


@gpu
def test_streams_and_threads():
    """A call follows the current stream, in threads of their own too, and outputs belong to it."""
    import threading
    Q, K, V, dO = _qkv(1, 256, 2, 2, 64)
    want = moda.moda_attn_fwd_gqa(Q, K, V, None, 0, 0.125)
    torch.cuda.synchronize()
    out, errors = {}, []

    def work(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                leaves = [t.clone().requires_grad_() for t in (Q, K, V)]
                for _ in range(20):
                    O, LSE = moda.moda_attention(*leaves, None, 0, 0.125)
                    g = torch.autograd.grad(O, leaves, dO)
            s.synchronize()
            out[i] = [O, LSE, *g]
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(4):
        _same(out[i][:2], want)
        _same(out[i], out[0], loose=(2,))


@pytest.fixture
def other_host(monkeypatch, tmp_path):
    """The binding as another Python or torch finds it: the extension's file has another name."""
    monkeypatch.setattr(binding, "_host", None)
    monkeypatch.setattr(binding, "HOST_PATH", str(tmp_path / "_host.so"))


def test_without_the_extension_calls_take_the_python_form(other_host):
    x = torch.zeros(1, 4, 2, 64, dtype=BF16)
    for f in (lambda: moda.moda_attn_fwd_gqa(x, x, x, None, 0, 0.1), lambda: moda.moda_attention(x, x, x),
              lambda: moda.moda_attn_bwd_gqa(x, x, x, None, x, x, x, 0, 0.1), lambda: moda.moda_attn_decode(x[:, 0], x, x, None, 4, 0, 0.1)):
        with pytest.raises(ValueError, match="CUDA"):       # the Python form's own refusal
            f()


@gpu
def test_results_without_the_extension(other_host):
    Q, K, V, dO = _qkv(1, 130, 2, 2, 64)
    O, LSE = moda.moda_attn_fwd_gqa(Q, K, V, None, 0, 0.125)
    assert type(binding.host()).__name__ == "_NoHost"
    x = [t.requires_grad_() for t in (Q, K, V)]
    torch.autograd.grad(moda.moda_attention(*x, None, 0, 0.125)[0], x, dO)
    _same((O, LSE), moda.moda_attention(*x, None, 0, 0.125))


def test_a_build_is_for_one_python_and_one_torch():
    import sysconfig
    from paper_2603_15619_b200 import build
    assert build.HOST == binding.HOST_PATH and torch.__version__ in build.HOST and sysconfig.get_config_var("SOABI") in build.HOST


def test_a_build_is_taken_up_by_the_process_that_makes_it(monkeypatch):
    from paper_2603_15619_b200 import build
    monkeypatch.setattr(binding, "_host", binding._NoHost())
    build.build_host()
    assert binding.host().__spec__.origin == binding.HOST_PATH


class _Calls(torch.overrides.TorchFunctionMode):
    """Names of the torch functions that pass a torch-function mode."""

    def __init__(self):
        super().__init__()
        self.names = []

    def __torch_function__(self, func, types, args=(), kwargs=None):
        self.names.append(getattr(func, "__name__", str(func)))
        return func(*args, **(kwargs or {}))


@gpu
def test_torch_function_modes_see_the_calls_they_saw(general):
    Q, K, V, dO = _qkv(1, 64, 2, 2, 64)
    O, LSE = moda.moda_attn_fwd_gqa(Q, K, V, None, 0, 0.125)

    def seen(f):
        with _Calls() as mode:
            f()
        return mode.names

    for f in (lambda: moda.moda_attn_fwd_gqa(Q, K, V, None, 0, 0.125), lambda: moda.moda_attn_bwd_gqa(Q, K, V, None, O, dO, LSE, 0, 0.125),
              lambda: moda.moda_attn_decode(Q[:, 0], K, V, None, 64, 0, 0.125), lambda: moda.moda_attention(Q, K, V)):
        assert seen(f) == general(seen, f) and "empty_like" in seen(f)


@gpu
def test_a_default_device_does_not_cost_the_extension():
    Q, K, V, _ = _qkv(1, 64, 2, 2, 64)
    want = moda.moda_attn_fwd_gqa(Q, K, V, None, 0, 0.125)
    with torch.device("cpu"):
        got = binding.host().attn_fwd(Q, K, V, None, 0, 0.125, None, 0, None, None)
        assert got is not None and got[0].is_cuda
        with _Calls():
            assert binding.host().attn_fwd(Q, K, V, None, 0, 0.125, None, 0, None, None) is None
    _same(got, want)
