"""What a user of the MoDA operator has it do, as cases that can be timed and compared.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges; ``prepare`` makes what a program has in hand
before the call, ``run`` is one pass through the package's public entry points.  Values are seeded Gaussians with the
shapes of the workloads in ``paper_2603_15619_b200.synthetic`` and of the sweeps in ``bench.py``; attention cost does not
depend on the values.

Kinds of case:

    attend   one differentiable call, ``moda_attention``, and its backward pass
    stack    a training step through ``DepthStream``: every layer attends and appends its K, V, every second slot is an
             FFN-side projection written by ``project_write``; gradients of every input and weight
    layer    one layer of a training stack through the operator's own calls: forward that appends the layer's K, V,
             and backward; depth cache in bf16, in e4m3, or position-major for grouped heads
    prefill  a chunk of new positions over a longer KV cache (serving, forward only)
    decode   one token per sequence: contiguous cache, lengths per sequence, or pages
    project  key / value projection whose epilogue writes the depth slot
"""
from __future__ import annotations

import math

import torch

import paper_2603_15619_b200 as moda
from paper_2603_15619_b200 import flops

DEV = "cuda"
BF16 = torch.bfloat16


def listed():
    return [
        # the smallest differentiable call (workload c1): latency and launches
        dict(name="attend_tiny", kind="attend", B=1, T=256, H=2, Hk=2, d=64, l=4),
        # one optimisation step of a short, ragged batch through a whole stack (8 slots, half of them FFN-side)
        dict(name="stack_short", kind="stack", B=2, T=1000, H=16, Hk=16, d=128, n=4, Dm=2048),
        # last layer of the 1.5B-shaped model at its training length (workload c2)
        dict(name="layer_1p5b", kind="layer", cache="bf16", B=4, T=4096, H=16, Hk=16, d=128, l=23),
        # middle of the depth sweep (workload c3)
        dict(name="layer_8k", kind="layer", cache="bf16", B=2, T=8192, H=16, Hk=16, d=128, l=16),
        # long context (workload c4), the largest
        dict(name="layer_64k", kind="layer", cache="bf16", B=1, T=65536, H=16, Hk=16, d=128, l=24),
        # narrow heads, deep stack (workload c5, one sequence)
        dict(name="layer_narrow", kind="layer", cache="bf16", B=1, T=32768, H=32, Hk=32, d=64, l=32),
        # grouped heads with the position-major cache (a row of the paper's kernel table)
        dict(name="layer_grouped", kind="layer", cache="pm", B=1, T=16384, H=64, Hk=8, d=64, l=64),
        # a ragged length with the depth cache held in e4m3
        dict(name="layer_e4m3", kind="layer", cache="e4m3", B=2, T=5000, H=16, Hk=16, d=128, l=23),
        # serving: a chunk of a prompt over what is cached already
        dict(name="prefill_chunk", kind="prefill", B=4, Tq=2000, T=15000, H=16, Hk=8, d=128, l=24),
        # serving: one sequence, one token (latency)
        dict(name="decode_one", kind="decode", form="plain", B=1, T=8192, H=16, Hk=8, d=128, l=24),
        # serving: a batch of sequences of different lengths over a paged cache
        dict(name="decode_paged", kind="decode", form="paged", B=32, T=8192, H=32, Hk=8, d=128, l=24),
        # projection of a layer's K, V with the slot written beside them
        dict(name="kv_project", kind="project", cache="bf16", B=2, T=8192, Dm=2048, Hk=16, d=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fits(case):
    """No dearer than the largest listed case, and a few tens of GB at most."""
    w, top = work(case), work(next(c for c in listed() if c["name"] == "layer_64k"))
    slot = 4 * case["B"] * (case.get("Tq") or case["T"]) * case["Hk"] * case["d"]
    slots = 2 * (case.get("l", 2 * case.get("n", 1)) + 1)
    return w["flops"] <= top["flops"] and w["bytes"] <= top["bytes"] and slot * slots <= 30e9


def draw(rng):
    while True:
        kind = rng.choice(["attend", "stack", "layer", "layer", "layer", "prefill", "decode", "decode", "project"])
        d = rng.choice([64, 128])
        if kind == "attend":
            G = rng.choice([1, 1, 2, 4])
            Hk = rng.choice([1, 2, 4, 8])
            case = dict(kind=kind, B=rng.randint(1, 4), T=_log_int(rng, 65, 2048), H=Hk * G, Hk=Hk, d=d, l=rng.randint(0, 16))
        elif kind == "stack":
            G = rng.choice([1, 1, 2, 4])
            Hk = rng.choice([4, 8, 16])
            case = dict(kind=kind, B=rng.randint(1, 4), T=_log_int(rng, 200, 4096), H=Hk * G, Hk=Hk, d=d, n=rng.randint(2, 6),
                        Dm=rng.choice([1024, 2048]))
        elif kind == "layer":
            cache = rng.choice(["bf16", "bf16", "e4m3", "pm"])
            G = rng.choice([2, 4, 8]) if cache == "pm" else rng.choice([1, 1, 1, 2, 4]) if cache == "bf16" else 1
            Hk = rng.choice([4, 8, 16]) if G > 1 else rng.choice([8, 16, 32])
            case = dict(kind=kind, cache=cache, B=rng.randint(1, 4), T=_log_int(rng, 1024, 65536), H=Hk * G, Hk=Hk, d=d,
                        l=rng.randint(1, 64 if cache == "pm" else 32))
        elif kind == "prefill":
            G, Hk, T = rng.choice([1, 2, 4, 8]), rng.choice([4, 8, 16]), _log_int(rng, 2048, 65536)
            case = dict(kind=kind, B=rng.randint(1, 8), Tq=min(T, _log_int(rng, 128, 8192)), T=T, H=Hk * G, Hk=Hk, d=d, l=rng.randint(1, 32))
        elif kind == "decode":
            G, Hk = rng.choice([1, 2, 4, 8]), rng.choice([4, 8, 16])
            case = dict(kind=kind, form=rng.choice(["plain", "varlen", "paged"]), B=_log_int(rng, 1, 128), T=_log_int(rng, 300, 32768),
                        H=Hk * G, Hk=Hk, d=d, l=rng.randint(1, 32))
            if 4 * case["B"] * case["T"] * Hk * d > 8e9:
                continue
        else:
            case = dict(kind=kind, cache=rng.choice(["bf16", "e4m3"]), B=rng.randint(1, 4), T=_log_int(rng, 300, 32768),
                        Dm=rng.choice([1024, 2048, 4096]), Hk=rng.choice([4, 8, 16, 32]), d=d)
        if _fits(case):
            return case


# ---------------------------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 7919 + 17)
    return g


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=BF16)


def _fill_cache(g, kind, B, T, Hk, d, l, slots):
    """A depth cache of `slots` slots of which the first `l` have been written by the layers below."""
    cache = (moda.alloc_depth_cache_e4m3 if kind == "e4m3" else moda.alloc_depth_cache)(B, T, Hk, d, slots, DEV)
    append = {"bf16": moda.moda_depth_cache_append, "e4m3": moda.moda_depth_cache_append_e4m3,
              "pm": moda.moda_depth_cache_append_pm}[kind]
    for i in range(l):
        append(cache, i, _normal(g, B, T, Hk, d), _normal(g, B, T, Hk, d))
    return cache


def prepare(case, seed):
    c, g = case, _gen(seed)
    B, T, Hk, d = c["B"], c["T"], c["Hk"], c["d"]
    s = dict(case)
    if c["kind"] == "attend":
        H, l = c["H"], c["l"]
        s.update(Q=_normal(g, B, T, H, d), K=_normal(g, B, T, Hk, d), V=_normal(g, B, T, Hk, d), dO=_normal(g, B, T, H, d))
        s["depth"] = _fill_cache(g, "bf16", B, T, Hk, d, l, l) if l else None
        s["leaves"] = [s[k].requires_grad_(True) for k in ("Q", "K", "V", "depth") if s[k] is not None]
    elif c["kind"] == "stack":
        H, n, Dm = c["H"], c["n"], c["Dm"]
        s["qkv"] = [[_normal(g, B, T, h, d).requires_grad_(True) for h in (H, Hk, Hk)] for _ in range(n)]
        s["ffn"] = [[x.requires_grad_(True) for x in (_normal(g, B, T, Dm), _normal(g, Hk * d, Dm) * Dm ** -0.5, _normal(g, Hk * d, Dm) * Dm ** -0.5)]
                    for _ in range(n - 1)]                      # nothing attends to a slot behind the last layer
        s["dO"] = [_normal(g, B, T, H, d) for _ in range(n)]
    elif c["kind"] == "layer":
        H, l = c["H"], c["l"]
        s.update(Q=_normal(g, B, T, H, d), K=_normal(g, B, T, Hk, d), V=_normal(g, B, T, Hk, d), dO=_normal(g, B, T, H, d))
        s["depth"] = _fill_cache(g, c["cache"], B, T, Hk, d, l, l + 1)
        s["grad"] = moda.alloc_depth_cache(B, T, Hk, d, l, DEV)  # a stack keeps one gradient cache for all its layers
    elif c["kind"] == "prefill":
        H, l, Tq = c["H"], c["l"], c["Tq"]
        s.update(Q=_normal(g, B, Tq, H, d), K=_normal(g, B, T, Hk, d), V=_normal(g, B, T, Hk, d))
        s["depth"] = _fill_cache(g, "bf16", B, Tq, Hk, d, l, l)
    elif c["kind"] == "decode":
        H, l = c["H"], c["l"]
        s.update(q=_normal(g, B, H, d), depth=_normal(g, l, B, Hk, 2, d))
        # a server keeps its scratch from step to step
        s["workspace"] = torch.empty(moda.moda_decode_workspace_bytes(B, H, d), dtype=torch.uint8, device=DEV)
        if c["form"] == "paged":
            blocks = (T + 63) // 64
            s.update(K=_normal(g, B * blocks, 64, Hk, d), V=_normal(g, B * blocks, 64, Hk, d))
            s["table"] = torch.randperm(B * blocks, generator=g, device=DEV).to(torch.int32).view(B, blocks)
        else:
            s.update(K=_normal(g, B, T, Hk, d), V=_normal(g, B, T, Hk, d))
        if c["form"] != "plain":
            s["lens"] = torch.randint(1, T + 1, (B,), generator=g, device=DEV, dtype=torch.int32)
    else:
        Dm = c["Dm"]
        s.update(X=_normal(g, B, T, Dm), Wk=_normal(g, Hk * d, Dm) * Dm ** -0.5, Wv=_normal(g, Hk * d, Dm) * Dm ** -0.5)
        s["depth"] = _fill_cache(g, c["cache"], B, T, Hk, d, 0, 1)
    return s


def _parts(cache, slots):
    """A cache as up to 32 runs of whole slots (views; the largest caches are handled piece by piece)."""
    slots_of = cache.view(slots, -1)
    return list(slots_of.split(-(-slots // 32)))


def run(state):
    s = state
    kind, d = s["kind"], s["d"]
    scale = d ** -0.5
    if kind == "attend":
        O, LSE = moda.moda_attention(s["Q"], s["K"], s["V"], s["depth"], s["l"], scale)
        return [O, LSE, *torch.autograd.grad(O, s["leaves"], s["dO"])]
    if kind == "stack":
        n = s["n"]
        stream = moda.DepthStream(s["B"], s["T"], s["Hk"], d, 2 * n - 1, DEV)
        outs = []
        for i in range(n):
            outs.append(stream.attend(*s["qkv"][i], scale))
            if i < n - 1:
                stream.project_write(*s["ffn"][i])
        leaves = [x for group in s["qkv"] + s["ffn"] for x in group]
        return [*outs, *torch.autograd.grad(outs, leaves, s["dO"])]
    if kind == "layer":
        Q, K, V, depth, l = s["Q"], s["K"], s["V"], s["depth"], s["l"]
        if s["cache"] == "bf16":
            O, LSE = moda.moda_attn_fwd_append(Q, K, V, depth, l, scale, depth, l)
            grads = moda.moda_attn_bwd_gqa(Q, K, V, depth, O, s["dO"], LSE, l, scale, d_depth_kv=s["grad"])
        elif s["cache"] == "e4m3":
            O, LSE = moda.moda_attn_fwd_append_e4m3(Q, K, V, depth, l, scale, depth, l)
            grads = moda.moda_attn_bwd_e4m3(Q, K, V, depth, O, s["dO"], LSE, l, scale, d_depth_kv=s["grad"])
        else:
            O, LSE = moda.moda_attn_fwd_gqa_pm(Q, K, V, depth, l, scale)
            moda.moda_depth_cache_append_pm(depth, l, K, V)
            grads = moda.moda_attn_bwd_gqa_pm(Q, K, V, depth, O, s["dO"], LSE, l, scale, d_depth_kv_pm=s["grad"])
        return [O, LSE, depth.view(l + 1, -1)[l], *grads[:3], *_parts(grads[3], l)]
    if kind == "prefill":
        return moda.moda_attn_fwd_prefill(s["Q"], s["K"], s["V"], s["depth"], s["l"], scale)
    if kind == "decode":
        if s["form"] == "plain":
            return moda.moda_attn_decode(s["q"], s["K"], s["V"], s["depth"], s["T"], s["l"], scale, workspace=s["workspace"])
        if s["form"] == "varlen":
            return moda.moda_attn_decode_varlen(s["q"], s["K"], s["V"], s["lens"], s["depth"], s["T"], s["l"], scale, workspace=s["workspace"])
        return moda.moda_attn_decode_paged(s["q"], s["K"], s["V"], s["table"], s["lens"], s["depth"], s["T"], s["l"], scale,
                                           workspace=s["workspace"])
    K, V = moda.moda_kv_project_append(s["X"], s["Wk"], s["Wv"], s["Hk"], cache=s["depth"], slot=0, e4m3=s["cache"] == "e4m3")
    return [K, V, s["depth"]]


# ---------------------------------------------------------------------------------------------------------------------
def _layer_work(B, T, H, Hk, d, l, slot_bytes_per_value=2.0):
    """Forward (with the write of a slot) and backward of one layer: the conventions of ``flops``, K, V and slots with Hk heads."""
    q, kv = B * T * H * d, B * T * Hk * d
    fwd = 2 * (2 * q + 2 * kv) + slot_bytes_per_value * 2 * (l + 1) * kv + 4 * B * H * T
    bwd = 2 * (4 * q + 4 * kv) + (slot_bytes_per_value + 2) * 2 * l * kv + 4 * B * H * T
    return fwd + bwd, flops.fwd_bwd_flops(B, T, H, d, l)


def work(case):
    c = case
    B, T, Hk, d = c["B"], c["T"], c["Hk"], c["d"]
    if c["kind"] == "attend":
        by, fl = _layer_work(B, T, c["H"], Hk, d, c["l"])
    elif c["kind"] == "stack":
        by = fl = 0.0
        for i in range(c["n"]):
            b, f = _layer_work(B, T, c["H"], Hk, d, 2 * i)
            by, fl = by + b, fl + f
        x, kv, w = B * T * c["Dm"], B * T * Hk * d, 2 * Hk * d * c["Dm"]
        # projection, dX and dW; X, the weights, the slot and their gradients once each way
        fl += (c["n"] - 1) * 3 * 2.0 * B * T * c["Dm"] * 2 * Hk * d
        by += (c["n"] - 1) * 2.0 * (3 * x + 3 * w + 4 * kv)
    elif c["kind"] == "layer":
        by, fl = _layer_work(B, T, c["H"], Hk, d, c["l"], 1.0 + 4.0 / d if c["cache"] == "e4m3" else 2.0)
    elif c["kind"] == "prefill":
        Tq, H, l = c["Tq"], c["H"], c["l"]
        pairs = Tq * (T - Tq) + Tq * (Tq + 1) / 2 + Tq * l
        fl = 4.0 * B * H * d * pairs
        by = 2.0 * (2 * B * Tq * H * d + 2 * B * T * Hk * d + 2 * l * B * Tq * Hk * d) + 4.0 * B * H * Tq
    elif c["kind"] == "decode":
        H, l = c["H"], c["l"]
        rows = B * (T if c["form"] == "plain" else (T + 1) / 2) + l * B          # lengths are uniform in [1, T]
        by = 2.0 * (2 * rows * Hk * d + 2 * B * H * d)
        fl = 4.0 * rows * H * d
    else:
        x, kv, w = B * T * c["Dm"], B * T * Hk * d, 2 * Hk * d * c["Dm"]
        fl = 2.0 * B * T * c["Dm"] * 2 * Hk * d
        by = 2.0 * (x + w + 2 * kv) + (1.0 + 4.0 / d if c["cache"] == "e4m3" else 2.0) * 2 * kv
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    # bf16 storage with fp32 sums: outputs sit about 2e-3 (O, K, V) to 3.5e-3 (gradients) from the fp64 oracle, so two correct
    # implementations may differ by twice that; LSE (fp32) is far inside.
    t = {"rel": 1e-2}
    if case["kind"] == "project" and case["cache"] == "e4m3":
        t["differ"] = 0.02               # codes of values that round to another bf16: ties of the fp32 sums
    return t


# ---------------------------------------------------------------------------------------------------------------------
# The same in 64 bits and plain torch.  Depth slots as plain tensors: [slots, B, T, Hk, d], for K and for V.
def _read_cache(kind, cache, B, T, Hk, d, slots):
    Tp = -(-T // 128) * 128
    if kind == "pm":
        x = cache.view(slots, B, Hk, Tp, 2, d).permute(4, 0, 1, 3, 2, 5)
    elif kind == "bf16":
        x = cache.view(slots, B, Hk, Tp // 128, 2, d // 8, 128, 8).permute(4, 0, 1, 3, 6, 2, 5, 7).reshape(2, slots, B, Tp, Hk, d)
    else:
        blocks = cache.view(slots, B, Hk, Tp // 128, 2, 128 * d + 512)
        codes = blocks[..., :128 * d].contiguous().view(torch.float8_e4m3fn).float()
        codes = codes.view(slots, B, Hk, Tp // 128, 2, d // 16, 128, 16).permute(4, 0, 1, 3, 6, 2, 5, 7)
        row_scale = blocks[..., 128 * d:].contiguous().view(torch.float32).permute(4, 0, 1, 3, 5, 2)
        x = (codes.double() * row_scale[..., None, None].double()).reshape(2, slots, B, Tp, Hk, d)
    return x[0][:, :, :T], x[1][:, :, :T]


def _as_cache(kind, Kd, Vd):
    slots, B, T, Hk, d = Kd.shape
    Tp = -(-T // 128) * 128
    x = torch.zeros(2, slots, B, Tp, Hk, d, dtype=Kd.dtype, device=Kd.device)
    x[0, :, :, :T], x[1, :, :, :T] = Kd, Vd
    if kind == "pm":
        return x.permute(1, 2, 4, 3, 0, 5).reshape(-1)
    return x.view(2, slots, B, Tp // 128, 128, Hk, d // 8, 8).permute(1, 2, 5, 3, 0, 6, 4, 7).reshape(-1)


def _attend64(Q, K, V, Kd, Vd, scale, dO=None):
    """(O, LSE), and with dO (O, LSE, dQ, dK, dV, dKd, dVd), head by head over blocks of queries; the last query sees every key."""
    (B, Tq, H, d), T, Hk = Q.shape, K.shape[1], K.shape[2]
    new = lambda x: torch.zeros(x.shape, dtype=torch.float64, device=x.device)
    O, LSE = new(Q), torch.zeros(B, H, Tq, dtype=torch.float64, device=Q.device)
    if dO is not None:
        dQ, dK, dV, dKd, dVd = new(Q), new(K), new(V), new(Kd), new(Vd)
    rows = max(128, min(2048, (1 << 27) // T))
    for b in range(B):
        for h in range(H):
            j = h // (H // Hk)
            k, v = K[b, :, j].double(), V[b, :, j].double()
            for t in range(0, Tq, rows):
                u = min(Tq, t + rows)
                n = u + T - Tq                                             # keys that the block's last query sees
                q, kd, vd = Q[b, t:u, h].double(), Kd[:, b, t:u, j].double(), Vd[:, b, t:u, j].double()
                s = (q @ k[:n].t()).mul_(scale)
                s.masked_fill_(torch.ones(u - t, n, dtype=torch.bool, device=s.device).triu_(n - (u - t) + 1), -math.inf)
                sd = (q * kd).sum(-1).t() * scale
                lse = torch.logsumexp(torch.cat([torch.logsumexp(s, 1, keepdim=True), sd], 1), 1, keepdim=True)
                p, pd = s.sub_(lse).exp_(), (sd - lse).exp()
                o = p @ v[:n] + (pd.t()[..., None] * vd).sum(0)
                O[b, t:u, h], LSE[b, h, t:u] = o, lse[:, 0]
                if dO is None:
                    continue
                g = dO[b, t:u, h].double()
                D = (g * o).sum(-1, keepdim=True)
                dV[b, :n, j] += p.t() @ g
                ds = (g @ v[:n].t()).sub_(D).mul_(p)
                dsd = (((g * vd).sum(-1).t() - D) * pd).t()[..., None] * scale
                dQ[b, t:u, h] = (ds @ k[:n]).mul_(scale) + (dsd * kd).sum(0)
                dK[b, :n, j] += (ds.t() @ q).mul_(scale)
                dKd[:, b, t:u, j] += dsd * q
                dVd[:, b, t:u, j] += pd.t()[..., None] * g
    return (O, LSE) if dO is None else (O, LSE, dQ, dK, dV, dKd, dVd)


@torch.no_grad()
def exact(case, seed):
    s = prepare(case, seed)
    kind, B, T, Hk, d = s["kind"], s["B"], s["T"], s["Hk"], s["d"]
    scale = d ** -0.5
    if kind in ("attend", "layer"):
        l, form = s["l"], s.get("cache", "bf16")
        if l:
            Kd, Vd = _read_cache(form, s["depth"].detach(), B, T, Hk, d, s["l"] + (kind == "layer"))
        else:
            Kd = Vd = s["K"].detach()[None][:0]
        O, LSE, dQ, dK, dV, dKd, dVd = _attend64(s["Q"].detach(), s["K"].detach(), s["V"].detach(), Kd[:l], Vd[:l], scale, s["dO"])
        # the gradients of the largest caches would not fit the card in 64 bits and in the order of the cache
        parts = -(-l // -(-l // 32)) if l else 0
        grad = _as_cache("pm" if form == "pm" else "bf16", dKd, dVd) if l and dKd.numel() < 2.5e9 else None
        if kind == "attend":
            return [O, LSE, dQ, dK, dV] + ([grad] if l else [])
        slot = None if form == "e4m3" else _as_cache(form, s["K"][None].double(), s["V"][None].double())
        return [O, LSE, slot, dQ, dK, dV, *([None] * parts if grad is None else _parts(grad, l))]
    if kind == "stack":
        n = s["n"]
        Ks, Vs = [], []                                                    # what the slots hold, in their order
        for i in range(n):
            Ks.append(s["qkv"][i][1].detach().double())
            Vs.append(s["qkv"][i][2].detach().double())
            if i < n - 1:
                X, Wk, Wv = (x.detach().double() for x in s["ffn"][i])
                Ks.append((X @ Wk.t()).view(B, T, Hk, d))
                Vs.append((X @ Wv.t()).view(B, T, Hk, d))
        Ks, Vs = torch.stack(Ks), torch.stack(Vs)
        gK, gV, outs, dQs = torch.zeros_like(Ks), torch.zeros_like(Vs), [], []
        for i in range(n):
            O, _, dQ, dK, dV, dKd, dVd = _attend64(s["qkv"][i][0].detach(), Ks[2 * i], Vs[2 * i], Ks[:2 * i], Vs[:2 * i], scale, s["dO"][i])
            outs.append(O)
            dQs.append(dQ)
            gK[:2 * i] += dKd
            gV[:2 * i] += dVd
            gK[2 * i] += dK
            gV[2 * i] += dV
        grads = [x for i in range(n) for x in (dQs[i], gK[2 * i], gV[2 * i])]
        for i in range(n - 1):
            X, Wk, Wv = (x.detach().double() for x in s["ffn"][i])
            k, v, x = gK[2 * i + 1].reshape(B * T, -1), gV[2 * i + 1].reshape(B * T, -1), X.view(B * T, -1)
            grads += [(k @ Wk + v @ Wv).view_as(X), k.t() @ x, v.t() @ x]
        return [*outs, *grads]
    if kind == "prefill":
        Kd, Vd = _read_cache("bf16", s["depth"], B, s["Tq"], Hk, d, s["l"])
        return list(_attend64(s["Q"], s["K"], s["V"], Kd, Vd, scale))
    if kind == "decode":
        O, LSE = [], []
        for b in range(B):
            n = int(s["lens"][b]) if "lens" in s else T
            if s["form"] == "paged":
                K, V = (s[x][s["table"][b].long()].reshape(-1, Hk, d)[None, :n] for x in ("K", "V"))
            else:
                K, V = s["K"][b:b + 1, :n], s["V"][b:b + 1, :n]
            pair = s["depth"][:, b:b + 1, None]                            # [l, 1, 1, Hk, 2, d]
            o, lse = _attend64(s["q"][b:b + 1, None], K, V, pair[..., 0, :], pair[..., 1, :], scale)
            O.append(o[:, 0])
            LSE.append(lse[..., 0])
        return [torch.cat(O), torch.cat(LSE)]
    X = s["X"].double()
    K, V = ((X @ s[w].double().t()).view(B, T, Hk, d) for w in ("Wk", "Wv"))
    return [K, V, _as_cache("bf16", K[None], V[None]) if s["cache"] == "bf16" else None]
