"""The work a user of libmikv has it do, as measurable cases: decode steps, decode attention, a whole token over all
layers, the cache build from a prefill, and the prefill importance.

Every case goes through the package's public entry points (`MixedPrecisionLayer`, `mikv_decode_attention`,
`mikv_prefill_scores`) on seeded tensors shaped like the caches of Llama-2-7B, Llama-2-13B and Mistral-7B: K, V and
queries ~ N(0, 1) in bf16 with four outlier channels per KV head scaled by 10 in keys and queries, importance scores
~ LogNormal(0, 1). `exact` evaluates the same inputs in plain torch, the quantizer in IEEE fp32 as the method defines
it and everything after it in 64 bits.
"""
from __future__ import annotations

import math

import torch

import paper_2402_18096_gb300 as mikv
from paper_2402_18096_gb300.layer import MixedPrecisionLayer, workspace

D = mikv.HEAD_DIM
SCALE = 1.0 / math.sqrt(D)
STEPS_ROOM = 64  # decode steps a cache has room for beyond its prefill


def _case(kind, batch, heads_q, heads_kv, context, bits=2, group=32, ratio=0.2, hi_bits=16, k_channel=False, layers=1):
    return dict(kind=kind, batch=batch, heads_q=heads_q, heads_kv=heads_kv, context=context, bits=bits, group=group,
                ratio=ratio, hi_bits=hi_bits, k_channel=k_channel, layers=layers)


def listed():
    cases = {
        # one request on a short prompt: the smallest call, where launches and latency count
        "step-tiny": _case("step", 1, 32, 32, 512, 4, 32, 0.20),
        # three chat requests on a grouped-query model, an odd context length
        "step-gqa-b3-t1999": _case("step", 3, 32, 8, 1999, 2, 64, 0.20),
        # an ordinary serving batch: one layer's decode step on the Llama-2-7B shape
        "step-llama2-7b": _case("step", 8, 32, 32, 4096, 2, 32, 0.20),
        # INT3, 40 heads, 10 % important: the Llama-2-13B shape
        "step-llama2-13b": _case("step", 16, 40, 40, 8192, 3, 64, 0.10),
        # the largest: a long-context batch on the Mistral-7B shape
        "step-mistral-7b": _case("step", 32, 32, 8, 32768, 2, 32, 0.20),
        # the important set at reduced precision too (Table 3: INT8 important, INT2 retained)
        "step-mistral-hi8": _case("step", 32, 32, 8, 32768, 2, 64, 0.20, hi_bits=8),
        # per-channel retained keys with token buffering (App. C)
        "step-mistral-kch": _case("step", 32, 32, 8, 32768, 2, 64, 0.20, k_channel=True),
        # attention alone, for an engine with its own policy: a wide batch, nearly everything retained in INT3
        "attend-int3-b64": _case("attend", 64, 32, 32, 4096, 3, 128, 0.05),
        # a whole token: the decode step of all 32 layers of the Llama-2-7B shape, one after another
        "token-llama2-7b": _case("token", 8, 32, 32, 4096, 2, 32, 0.20, layers=32),
        # end of a long prefill: balancer, selection, gather and quantization of one layer's cache
        "build-mistral-7b": _case("build", 32, 32, 8, 32768, 2, 32, 0.20),
        # the prefill's accumulated attention: a batch of medium prompts, and one long prompt
        "scores-llama2-7b": _case("scores", 8, 32, 32, 4096),
        "scores-mistral-7b": _case("scores", 1, 32, 8, 32768),
    }
    return [dict(name=n, **c) for n, c in cases.items()]


def draw(rng):
    """One more case of the listed ranges: contexts of 300 to 32768 tokens (odd ones too), batches of 1 to 64, every
    head grouping, code width, group size, importance ratio and important-set precision the entry points are used with."""
    while True:
        kind = rng.choice(["step"] * 5 + ["attend", "token", "build", "build", "scores", "scores"])
        heads_q, heads_kv = rng.choice([(32, 32), (32, 32), (40, 40), (32, 8), (32, 8), (32, 16), (32, 4)])
        batch = int(round(math.exp(rng.uniform(0.0, math.log(64.0)))))
        context = int(round(math.exp(rng.uniform(math.log(300.0), math.log(32768.0)))))
        bits = rng.choice([2, 2, 3, 4])
        group = rng.choice([32, 64, 128])
        ratio = rng.choice([0.0, 0.05, 0.10, 0.20, 0.25, 0.50])
        variant = rng.choice(["bf16"] * 4 + ["coded", "channel", "evict"])
        c = _case(kind, batch, heads_q, heads_kv, context, bits, group, ratio)
        if kind == "scores":
            c.update(bits=2, group=32, ratio=0.2)
        elif kind == "token":
            c["layers"] = rng.choice([16, 24, 32])
        elif variant == "coded":
            c["hi_bits"] = rng.choice([8, 4, 2])
        elif variant == "channel":
            c["k_channel"] = True
        elif variant == "evict":
            c.update(bits=0, group=32, ratio=rng.choice([0.20, 0.50]))
        if kind in ("attend", "build") and c["bits"] == 0 and c["ratio"] == 0.0:
            continue
        prefill = batch * (heads_q + 2 * heads_kv) * context * D * 2 * c["layers"]
        most = 1.4e10 if kind != "token" else 4e10  # bytes of prefill tensors behind the largest listed caches
        if prefill <= most and work(c)["bytes"] <= (1.6e9 if kind in ("step", "attend") else 6.5e9 if kind == "token"
                                                    else 1.6e10) and work(c)["flops"] <= 4.5e12:
            return c


# ---------------------------------------------------------------------------------------------------- inputs

def _shape(c):
    return mikv.shape_for_context(c["batch"], c["heads_q"], c["heads_kv"], c["bits"], c["group"], c["context"],
                                  c["ratio"], STEPS_ROOM, hi_bits=c["hi_bits"],
                                  k_channel_group=64 if c["k_channel"] else 0)


def _gen(seed, layer, kind):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + layer * 101 + kind) & 0x7FFFFFFFFFFF)


def _normal(seed, layer, kind, *shape):
    return torch.randn(*shape, generator=_gen(seed, layer, kind), device="cuda", dtype=torch.bfloat16)


def _channel_scale(c, seed, layer):
    """bf16 [Hkv, 1, D]: 10 on two channels of the first half of each KV head and on their rotary partners."""
    pick = torch.rand(c["heads_kv"], D // 2, generator=_gen(seed, layer, 0), device="cuda").topk(2, dim=1).indices
    scale = torch.ones(c["heads_kv"], D, device="cuda", dtype=torch.bfloat16)
    return scale.scatter_(1, torch.cat([pick, pick + D // 2], 1), 10.0).unsqueeze(1)


def _prefill(c, seed, layer=0):
    """(q_pre [B, Hq, T, D], k, v [B, Hkv, T, D]) of one layer's prefill, bf16."""
    B, Hq, H, T = c["batch"], c["heads_q"], c["heads_kv"], c["context"]
    sc = _channel_scale(c, seed, layer)
    q = _normal(seed, layer, 1, B, Hq, T, D).mul_(sc.repeat_interleave(Hq // H, 0))
    return q, _normal(seed, layer, 2, B, H, T, D).mul_(sc), _normal(seed, layer, 3, B, H, T, D)


def _scores(c, seed, layer=0):
    return torch.randn(c["batch"], c["heads_kv"], c["context"], generator=_gen(seed, layer, 4), device="cuda").exp_()


def _token(c, seed, layer=0):
    """(q [B, Hq, D], k_new, v_new [B, Hkv, D]) of the decoded token, bf16."""
    B, Hq, H = c["batch"], c["heads_q"], c["heads_kv"]
    k = _normal(seed, layer, 6, B, H, D).mul_(_channel_scale(c, seed, layer)[:, 0])
    return _normal(seed, layer, 5, B, Hq, D), k, _normal(seed, layer, 7, B, H, D)


CACHE_ARRAYS = ("k_hi", "v_hi", "hi_tok", "acc", "k_codes", "v_codes", "k_params", "v_params", "lo_tok",
                "k_hi_params", "v_hi_params")


def _cache_outputs(cache):
    got = {n: getattr(cache, n) for n in CACHE_ARRAYS}
    return {n: t for n, t in got.items() if t is not None and t.numel()}


def prepare(case, seed):
    c, shape = case, _shape(case)
    if c["kind"] == "scores":
        q, k, _ = _prefill(c, seed)
        ws = workspace(mikv.mikv_workspace_bytes(shape, mikv.WS_PREFILL, c["context"]))
        scores = torch.zeros(c["batch"], c["heads_kv"], c["context"], device="cuda")
        return dict(kind="scores", shape=shape, q=q, k=k, scores=scores, ws=ws)
    if c["kind"] == "build":
        q, k, v = _prefill(c, seed)
        return dict(kind="build", shape=shape, q=q, k=k, v=v, scores=_scores(c, seed))
    layers, inputs = [], []
    for li in range(c["layers"]):
        q, k, v = _prefill(c, seed, li)
        layers.append(MixedPrecisionLayer.from_prefill(shape, k, v, _scores(c, seed, li), q))
        del q, k, v
        inputs.append(_token(c, seed, li))
    out = torch.zeros(c["layers"], c["batch"], c["heads_q"], D, dtype=torch.bfloat16, device="cuda")
    state = dict(kind=c["kind"], layers=layers, inputs=inputs, out=out, n_lo=layers[0].n_lo, pos=layers[0].pos)
    if c["kind"] == "attend":
        layer = layers[0]  # the slot of the next token holds this one, so that every attended slot holds a token
        mikv.mikv_insert_token(layer.cache, inputs[0][1], inputs[0][2], layer.pos, layer.slots)
        layer.ws = workspace(mikv.mikv_workspace_bytes(shape, mikv.WS_ATTENTION, layer.n_lo))
        state["outputs"] = {"out": out[0]}
    elif c["kind"] == "step":
        state["outputs"] = dict(_cache_outputs(layers[0].cache), out=out[0], slots=layers[0].slots)
    else:  # a model keeps each kind of cache array of all its layers in one allocation
        pool = {n: torch.stack([getattr(layer.cache, n) for layer in layers]) for n in _cache_outputs(layers[0].cache)}
        slots = torch.stack([layer.slots for layer in layers])
        for li, layer in enumerate(layers):
            for n, t in pool.items():
                setattr(layer.cache, n, t[li])
            layer.slots = slots[li]
        state["outputs"] = dict(pool, out=out, slots=slots)
    return state


def run(state):
    """One pass. A decode step's retained length is put back first, so that every pass is the step of that length."""
    kind = state["kind"]
    if kind == "scores":
        mikv.mikv_prefill_scores(state["shape"], state["q"], state["k"], state["scores"], state["ws"])
        return state["scores"]
    if kind == "build":
        layer = MixedPrecisionLayer.from_prefill(state["shape"], state["k"], state["v"], state["scores"], state["q"])
        out = _cache_outputs(layer.cache)
        out["slots"] = layer.slots
        if layer.cache.balancer is not None:
            out["balancer"] = layer.cache.balancer
        return out
    if kind == "attend":
        layer = state["layers"][0]
        mikv.mikv_decode_attention(layer.cache, layer.n_lo, state["inputs"][0][0], layer.sm_scale, state["out"][0],
                                   layer.ws)
        return state["outputs"]
    for layer, (q, k, v), out in zip(state["layers"], state["inputs"], state["out"]):
        layer.n_lo, layer.pos = state["n_lo"], state["pos"]
        layer.step(q, k, v, out)
    return state["outputs"]


# ------------------------------------------------------------------------------------------------------ work

def _row(bits, group):
    return D * bits / 8 + 4 * (D / group)


def _sizes(c):
    k = mikv.mikv_budget(c["context"], c["ratio"])
    return k, (c["context"] - k if c["bits"] else 0)


def work(case):
    c = case
    B, Hq, H, T = c["batch"], c["heads_q"], c["heads_kv"], c["context"]
    if c["kind"] == "scores":  # the causal triangle of Q K^T, once
        return {"bytes": 2.0 * B * (Hq + H) * T * D + 4.0 * B * H * T, "flops": 2.0 * D * B * Hq * T * (T + 1) / 2}
    k, n_lo = _sizes(c)
    hi_row = 4.0 * D if c["hi_bits"] == 16 else 2 * _row(c["hi_bits"], 64)
    if not c["bits"]:
        lo = 0.0
    elif c["k_channel"]:  # the incomplete last group of 64 waits in bf16
        whole = n_lo // 64 * 64
        lo = whole * (D * c["bits"] / 8 + 4.0 * D / 64 + _row(c["bits"], c["group"])) + (n_lo - whole) * 4.0 * D
    else:
        lo = n_lo * 2.0 * _row(c["bits"], c["group"])
    if c["kind"] == "build":  # q, k, v and the scores in; both sets, the token ids, the scores and the balancer out
        read = 2.0 * B * (Hq + 2 * H) * T * D + 4.0 * B * H * T
        return {"bytes": read + B * H * (k * (hi_row + 8) + lo + 4.0 * n_lo) + 4.0 * H * D, "flops": 0.0}
    hi_cap = k + 1
    cache = B * H * (hi_cap * hi_row + lo)
    small = 4.0 * B * Hq * D
    if c["kind"] != "attend":  # the new token, its slot, the scores in and out, the token ids, the demoted row
        small += B * H * (4.0 * D + hi_cap * 12.0 + 8 + (2 * _row(c["bits"], c["group"]) + 4 if c["bits"] else 0))
    return {"bytes": c["layers"] * (cache + small), "flops": c["layers"] * 4.0 * D * B * Hq * (hi_cap + n_lo)}


# ----------------------------------------------------------------------------------------------------- exact

def _half_toward(x, up):
    """fp32 -> fp16 rounded up or down."""
    h = x.half()
    off = h.float() < x if up else h.float() > x
    bits = h.view(torch.int16).int() & 0xFFFF
    away = (bits >= 0x8000) ^ up  # the magnitude grows
    zero = (bits & 0x7FFF) == 0
    moved = torch.where(zero, torch.full_like(bits, 1 if up else 0x8001), torch.where(away, bits + 1, bits - 1))
    bits = torch.where(off, moved, bits)
    return torch.where(bits >= 0x8000, bits - 0x10000, bits).to(torch.int16).view(torch.float16)


def _eq1(x, bits):
    """fp32 [..., n] quantized over its last dimension (Eq. 1) and dequantized in 64 bits."""
    qmax = (1 << bits) - 1
    beta = _half_toward(x.amin(-1, keepdim=True), False).float()
    span = x.amax(-1, keepdim=True) - beta
    alpha = torch.where(span == 0, torch.ones_like(span), _half_toward(span / qmax, True).float())
    code = torch.round((x - beta) / alpha).clamp_(0, qmax)
    return code.double() * alpha.double() + beta.double()


def _eq1_rows(x, bits, group):
    return _eq1(x.unflatten(-1, (D // group, group)), bits).flatten(-2)


def _balancer(q, k):
    H = k.shape[1]
    mq = q.abs().amax((0, 2)).float().view(H, -1, D).amax(1)
    mk = k.abs().amax((0, 2)).float()
    return torch.where((mq == 0) | (mk == 0), torch.ones_like(mq), torch.sqrt(mq / mk))


def _exact_layer(c, seed, layer, attend_only):
    """(out [B, Hq, D], acc [B, Hkv, hi_stride]) of one layer's step, in 64 bits."""
    B, Hq, H, T = c["batch"], c["heads_q"], c["heads_kv"], c["context"]
    G, shape = Hq // H, _shape(c)
    n_hi, n_lo = _sizes(c)
    q_pre, k, v = _prefill(c, seed, layer)
    bal = torch.ones(H, D, device="cuda") if c["k_channel"] else _balancer(q_pre, k)
    del q_pre
    scores = _scores(c, seed, layer)
    q, k_new, v_new = _token(c, seed, layer)
    out = torch.zeros(B, Hq, D, dtype=torch.float64, device="cuda")
    acc = torch.zeros(B, H, shape.hi_stride, dtype=torch.float64, device="cuda")
    for b in range(B):
        order = scores[b].sort(dim=1, stable=True).indices
        kept, gone = order[:, T - n_hi:].sort(dim=1).values, order[:, :T - n_hi].sort(dim=1).values
        rows = lambda x, i: x.gather(1, i.unsqueeze(-1).expand(-1, -1, D))  # noqa: E731
        kh = torch.cat([rows(k[b], kept), k_new[b].unsqueeze(1)], 1).float()
        vh = torch.cat([rows(v[b], kept), v_new[b].unsqueeze(1)], 1).float()
        qf = q[b].double().view(H, G, D)
        qb = qf / bal.double().unsqueeze(1)
        if c["hi_bits"] == 16:
            keys, vals, logits = kh.double(), vh.double(), None
            logits = qf @ keys.transpose(1, 2)
        else:
            keys = _eq1_rows(kh * bal.unsqueeze(1), c["hi_bits"], 64)
            vals = _eq1_rows(vh, c["hi_bits"], 64)
            logits = qb @ keys.transpose(1, 2)
        if n_lo:
            kl, vl = rows(k[b], gone).float(), rows(v[b], gone).float()
            if c["k_channel"]:
                whole = n_lo // 64 * 64
                groups = kl[:, :whole].unflatten(1, (whole // 64, 64)).transpose(2, 3)
                kd = _eq1(groups, c["bits"]).transpose(2, 3).flatten(1, 2) if whole else kl[:, :0].double()
                vd = _eq1_rows(vl[:, :whole], c["bits"], c["group"])
                kl, vl = torch.cat([kd, kl[:, whole:].double()], 1), torch.cat([vd, vl[:, whole:].double()], 1)
            else:
                kl = _eq1_rows(kl * bal.unsqueeze(1), c["bits"], c["group"])
                vl = _eq1_rows(vl, c["bits"], c["group"])
            logits = torch.cat([logits, qb @ kl.transpose(1, 2)], 2)
            vals = torch.cat([vals, vl], 1)
        p = torch.softmax(logits * SCALE, -1)
        out[b] = (p @ vals).view(Hq, D)
        acc[b, :, :n_hi] = scores[b].double().gather(1, kept)
        if not attend_only:
            acc[b, :, :n_hi + 1] += p[:, :, :n_hi + 1].sum(1)
    return out, acc


def exact(case, seed):
    c = case
    B, Hq, H, T = c["batch"], c["heads_q"], c["heads_kv"], c["context"]
    if c["kind"] == "scores":
        q, k, _ = _prefill(c, seed)
        out = torch.zeros(B, H, T, dtype=torch.float64, device="cuda")
        n = 2048
        for b in range(B):
            for j in range(Hq):
                h = j // (Hq // H)
                kd = k[b, h].double()
                for i in range(0, T, n):
                    e = min(T, i + n)
                    s = (q[b, j, i:e].double() @ kd[:e].T).mul_(SCALE)
                    s[:, i:].masked_fill_(torch.ones(e - i, e - i, dtype=torch.bool, device="cuda").triu_(1), -math.inf)
                    out[b, h, :e] += torch.softmax(s, -1).sum(0)
        return out
    if c["kind"] == "build":  # codes and rows are whole numbers and copies; the balancer is what is computed
        if c["k_channel"]:
            return None
        q, k, _ = _prefill(c, seed)
        mq = q.abs().amax((0, 2)).double().view(H, -1, D).amax(1)
        return {"balancer": torch.sqrt(mq / k.abs().amax((0, 2)).double())}
    got = [_exact_layer(c, seed, li, c["kind"] == "attend") for li in range(c["layers"])]
    out, acc = (torch.stack([g[i] for g in got]) for i in (0, 1))
    if c["kind"] == "attend":
        return {"out": out[0]}
    return {"out": out[0], "acc": acc[0]} if c["kind"] == "step" else {"out": out, "acc": acc}
