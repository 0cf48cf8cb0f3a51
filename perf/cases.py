"""The calls whose speed is measured: what a program that deploys a W4/W2-GateUp
model has the library do, over the range of sizes it meets.

A case is one of
  gateup   the fused gate/up projection of one layer (2-, 3- or 4-bit codes,
           unmerged adapters with 2 and 3 bits), as an engine that schedules
           the MLP's matrices itself calls it;
  down     the 4-bit down projection of one layer (bf16 or fp32 output, with or
           without residual), which is also the projection call of attention;
  dense    the bf16 down projection of the BF16/W2-GateUp configuration;
  stack    a stack of gated-MLP layers through one call: decode steps of one to
           a few sequences, batched decode, prefill chunks;
  decoder  whole decoder layers, one decode step over a KV cache;
  moe      mixture-of-experts blocks, one decode step;
  pack     quantizing and packing a weight matrix, once per checkpoint.
Shapes are those of the package's configurations (4B, 8B and 14B class dense
models, a GPT-OSS-20B-shaped MoE) and generic ones; weights, adapters and
activations follow the distributions the package's synthetic workloads use.
Stacks have more packed weights than the L2 cache holds wherever the model has.
"""
import math

import torch

from paper_2606_04238_gb300 import wq

DEV = "cuda"
SHAPES = {"small": (256, 768), "4b": (2560, 9728), "8b": (4096, 14336), "14b": (5120, 17408)}
EPS = 1e-6


def listed():
    return [
        # one layer's gate/up of a small model, one token: the smallest call, all latency
        dict(name="gateup_small_m1", kind="gateup", d=256, inter=768, bits=2, group=64, r=8, m=1, prenorm=True),
        # a decode step of one sequence through 12 of the 4B-class model's 36 MLP layers (the headline workload's
        # layers; deeper stacks only add rounding differences between implementations)
        dict(name="stack_4b_m1", kind="stack", d=2560, inter=9728, layers=12, bits=2, group=128, group_down=128,
             down_bits=4, r=16, m=1),
        # a speculative-decoding verify step (5 tokens) of the 8B-class model with groups of 32
        dict(name="stack_8b_g32_m5", kind="stack", d=4096, inter=14336, layers=8, bits=2, group=32, group_down=32,
             down_bits=4, r=32, m=5),
        # batched decode, 24 sequences, 8B-class model
        dict(name="stack_8b_m24", kind="stack", d=4096, inter=14336, layers=8, bits=2, group=128, group_down=128,
             down_bits=4, r=32, m=24),
        # batched decode, 64 sequences, uniform 4-bit (the configuration the 2-bit one is compared with)
        dict(name="stack_4b_w4_m64", kind="stack", d=2560, inter=9728, layers=10, bits=4, group=128, group_down=128,
             down_bits=4, r=0, m=64),
        # a prefill chunk of 512 tokens, 14B-class model
        dict(name="stack_14b_m512", kind="stack", d=5120, inter=17408, layers=2, bits=2, group=128, group_down=128,
             down_bits=4, r=32, m=512),
        # a whole long prompt in one call (a ragged token count), 4B-class model
        dict(name="stack_4b_m3001", kind="stack", d=2560, inter=9728, layers=2, bits=2, group=128, group_down=128,
             down_bits=4, r=16, m=3001),
        # whole decoder layers, one sequence with an 8k context
        dict(name="decoder_4b_b1", kind="decoder", d=2560, inter=9728, layers=6, bits=2, group=128, r=16, heads=32,
             kv=8, hd=128, m=1, ctx=8192),
        # whole decoder layers, 16 sequences of different lengths up to 2k
        dict(name="decoder_4b_b16", kind="decoder", d=2560, inter=9728, layers=4, bits=2, group=128, r=16, heads=32,
             kv=8, hd=128, m=16, ctx=2048),
        # mixture of experts, one sequence
        dict(name="moe_m1", kind="moe", d=2880, inter=2880, layers=6, experts=32, top_k=4, bits=2, group=64, r=16, m=1),
        # mixture of experts, batched decode of 32 sequences
        dict(name="moe_m32", kind="moe", d=2880, inter=2880, layers=3, experts=32, top_k=4, bits=2, group=64, r=16,
             m=32),
        # quantizing and packing one gate matrix of the 8B-class model while a checkpoint is loaded
        dict(name="pack_w2_8b", kind="pack", d=4096, inter=14336, bits=2, group=128),
    ]


MOST_FLOPS = 4.0e11  # below the largest listed case's 5.5e11
MOST_BYTES = 1.0e9   # below the largest listed case's


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _shape(rng):
    """(d, inter, group): a model's shape, or a generic one."""
    if rng.random() < 0.5:
        d, inter = SHAPES[rng.choice(["4b", "4b", "8b", "14b"])]
        return d, inter, rng.choice([32, 64, 128, 128])
    d, inter = 64 * _log_int(rng, 4, 80), 64 * _log_int(rng, 8, 272)
    fits = [g for g in (32, 64, 128) if d % g == 0 and inter % g == 0]
    return d, inter, rng.choice(fits)


def draw(rng):
    for _ in range(200):
        kind = rng.choice(["gateup", "down", "dense", "stack", "stack", "stack", "stack", "decoder", "moe", "pack"])
        d, inter, group = _shape(rng)
        if kind == "gateup":
            bits = rng.choice([2, 2, 3, 4])
            c = dict(kind=kind, d=d, inter=inter, bits=bits, group=group, r=0 if bits == 4 else rng.choice([0, 8, 16, 32]),
                     m=_log_int(rng, 1, 64 if bits == 3 else 1024), prenorm=rng.random() < 0.7)
        elif kind == "down":
            c = dict(kind=kind, d=d, inter=inter, group=group, m=_log_int(rng, 1, 1024), f32=rng.random() < 0.4,
                     residual=rng.random() < 0.6)
        elif kind == "dense":
            c = dict(kind=kind, d=d, inter=inter, m=_log_int(rng, 1, 64), f32=rng.random() < 0.4,
                     residual=rng.random() < 0.6)
        elif kind == "stack":
            bits = rng.choice([2, 2, 2, 3, 4])
            down_bits = rng.choice([4, 4, 4, 4, 16])
            c = dict(kind=kind, d=d, inter=inter, layers=_log_int(rng, 1, 8), bits=bits, group=group, group_down=group,
                     down_bits=down_bits, r=0 if bits == 4 else rng.choice([0, 8, 16, 32]),
                     m=_log_int(rng, 1, 64 if bits == 3 or down_bits == 16 else 4096))
        elif kind == "decoder":
            heads, kv, hd = rng.choice([(32, 8, 128), (32, 8, 128), (16, 4, 64), (40, 8, 128)])
            if d % 128 or d < 512 or inter % 128:
                continue
            c = dict(kind=kind, d=d, inter=inter, layers=_log_int(rng, 1, 6), bits=rng.choice([2, 2, 4]), group=group,
                     r=16, heads=heads, kv=kv, hd=hd, m=_log_int(rng, 1, 32), ctx=_log_int(rng, 64, 16384))
            c["r"] = 0 if c["bits"] == 4 else c["r"]
            if c["m"] * c["ctx"] > 65536:
                continue
        elif kind == "moe":
            d, inter = rng.choice([(2880, 2880), (64 * _log_int(rng, 8, 45), 64 * _log_int(rng, 8, 45))])
            e = rng.choice([8, 16, 32])
            c = dict(kind=kind, d=d, inter=inter, layers=rng.randint(1, 4), experts=e, top_k=rng.choice([1, 2, 4]),
                     bits=rng.choice([2, 2, 4]), group=rng.choice([32, 64]), r=16, m=_log_int(rng, 1, 64))
            c["r"] = 0 if c["bits"] == 4 else c["r"]
        else:
            c = dict(kind=kind, d=d, inter=inter, bits=rng.choice([2, 2, 3, 4]), group=group)
        w = work(c)
        if w["flops"] <= MOST_FLOPS and w["bytes"] <= MOST_BYTES:
            return c
    raise RuntimeError("no case drawn")


# ---- inputs -----------------------------------------------------------------

class _Rand:
    """Draws of one case: every tensor has a seed of its own, made from the case's."""

    def __init__(self, seed):
        self.seed = int(seed)

    def normal(self, shape, key, std=1.0):
        g = torch.Generator(device=DEV)
        g.manual_seed((self.seed * 1_000_003 + key) % (1 << 62))
        return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32) * std

    def bf16(self, shape, key, std=1.0):
        return self.normal(shape, key, std).to(torch.bfloat16)

    def lens(self, n, hi, key):
        g = torch.Generator(device=DEV)
        g.manual_seed((self.seed * 1_000_003 + key) % (1 << 62))
        if n == 1:
            return torch.full((1,), hi - 1, dtype=torch.int32, device=DEV)
        return torch.randint(hi // 4, hi, (n,), generator=g, device=DEV, dtype=torch.int32)


def _mlp_draws(c, rnd, layer, experts=1):
    """fp32 weights and bf16 adapters of layer `layer` (of `experts` stacked experts)."""
    d, inter, r, k = c["d"], c["inter"], c.get("r", 0), 16 * (layer + 1)
    wg = rnd.normal((experts * inter, d), k, 0.02)
    wu = rnd.normal((experts * inter, d), k + 1, 0.02)
    wd = rnd.normal((experts * d, inter), k + 2, 0.02)
    lora = None
    if r:
        lora = (rnd.bf16((experts * 2 * r, d), k + 3, 0.01), rnd.bf16((experts * inter, r), k + 4, 0.01),
                rnd.bf16((experts * inter, r), k + 5, 0.01))
    return wg, wu, wd, lora


def _mlp_layer(c, rnd, layer, experts=1):
    wg, wu, wd, lora = _mlp_draws(c, rnd, layer, experts)
    gd = c.get("group_down", c["group"])
    down = wq.dense_weight(wd.to(torch.bfloat16)) if c.get("down_bits", 4) == 16 else wq.pack(wd, gd, 4)
    kw = {}
    if lora:
        kw = dict(lora_a=lora[0], lora_b_gate=lora[1], lora_b_up=lora[2], lora_scale=_scale(c))
    return wq.MLPLayer(wq.pack(wg, c["group"], c["bits"]), wq.pack(wu, c["group"], c["bits"]), down, **kw)


def _scale(c):
    return 2.0  # alpha / r with the alpha = 2r of the package's configurations


def prepare(case, seed):
    c, rnd = case, _Rand(seed)
    d, inter, kind, m = c["d"], c["inter"], c["kind"], c.get("m", 0)
    s = dict(c=c)
    if kind == "gateup":
        ly = _mlp_layer(dict(c, down_bits=16), rnd, 0)
        s.update(layer=ly, x=rnd.bf16((m, d), 1), h=torch.empty((m, inter), dtype=torch.bfloat16, device=DEV),
                 ws=wq.workspace(m, d, inter, c["r"]))
    elif kind in ("down", "dense"):
        w = rnd.normal((d, inter), 18, 0.02)
        s.update(w=w.to(torch.bfloat16) if kind == "dense" else wq.pack(w, c["group"], 4),
                 h=rnd.bf16((m, inter), 1, 0.5), res=rnd.bf16((m, d), 2) if c["residual"] else None,
                 y=torch.empty((m, d), dtype=torch.float32 if c["f32"] else torch.bfloat16, device=DEV))
        if kind == "down":
            s["ws"] = wq.workspace(m, d, inter, 0)
    elif kind == "stack":
        layers = [_mlp_layer(c, rnd, i) for i in range(c["layers"])]
        s.update(layers=layers, table=wq.LayerTable(layers), x=rnd.bf16((m, d), 1),
                 y=torch.empty((m, d), dtype=torch.bfloat16, device=DEV), ws=wq.workspace(m, d, inter, c["r"]))
    elif kind == "decoder":
        h, kv, hd, n = c["heads"], c["kv"], c["hd"], c["layers"]
        layers, caches = [], []
        for i in range(n):
            k = 16 * (i + 1)
            wqkv, wo = rnd.normal(((h + 2 * kv) * hd, d), k + 8, 0.02), rnd.normal((d, h * hd), k + 9, 0.02)
            layers.append(wq.DecoderLayer(wq.pack(wqkv, 128, 4), wq.pack(wo, 64, 4), _mlp_layer(c, rnd, i), h, kv, hd))
            caches.append((rnd.bf16((m, kv, c["ctx"], hd), k + 10), rnd.bf16((m, kv, c["ctx"], hd), k + 11)))
        s.update(layers=layers, caches=caches, cl=[ly.c() for ly in layers], x=rnd.bf16((m, d), 1),
                 lens=rnd.lens(m, c["ctx"], 2), ws=wq.decoder_workspace(m, layers[0], c["ctx"]),
                 y=[torch.empty((m, d), dtype=torch.bfloat16, device=DEV) for _ in range(n)])
    elif kind == "moe":
        e = c["experts"]
        layers = [wq.MoELayer(_mlp_layer(c, rnd, i, e), e, c["top_k"]) for i in range(c["layers"])]
        s.update(layers=layers, cl=[ly.c() for ly in layers], x=rnd.bf16((m, d), 1),
                 logits=[rnd.normal((m, e), 16 * (i + 1) + 8) for i in range(c["layers"])],
                 ws=wq.moe_workspace(m, layers[0]),
                 y=[torch.empty((m, d), dtype=torch.bfloat16, device=DEV) for _ in range(c["layers"])])
    else:
        s.update(w=rnd.normal((inter, d), 16, 0.02), out=wq.empty_qweight(inter, d, c["group"], c["bits"]))
    return s


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "gateup":
        ly = s["layer"]
        if c["bits"] == 4:
            return wq.gateup_w4(s["x"], ly.gate, ly.up, prenorm=c["prenorm"], h=s["h"], ws=s["ws"])
        fn = wq.gateup_w2_lora if c["bits"] == 2 else wq.gateup_w3_lora
        return fn(s["x"], ly.gate, ly.up, ly.lora_a, ly.lora_b_gate, ly.lora_b_up, lora_scale=ly.lora_scale,
                  prenorm=c["prenorm"], h=s["h"], ws=s["ws"])
    if kind == "down":
        return wq.down_w4(s["h"], s["w"], residual=s["res"], out_f32=c["f32"], y=s["y"], ws=s["ws"])
    if kind == "dense":
        return wq.down_bf16(s["h"], s["w"], residual=s["res"], out_f32=c["f32"], y=s["y"])
    if kind == "stack":
        return wq.mlp_forward(s["x"], s["layers"], prenorm=True, y=s["y"], ws=s["ws"], table=s["table"])
    if kind == "decoder":
        cur = s["x"]
        for i, ly in enumerate(s["layers"]):
            kc, vc = s["caches"][i]
            cur = wq.decoder_layer_forward(cur, s["lens"], ly, kc, vc, y=s["y"][i], ws=s["ws"], c_layer=s["cl"][i])
        return {"y": cur, "caches": s["caches"]}
    if kind == "moe":
        cur = s["x"]
        for i, ly in enumerate(s["layers"]):
            cur = wq.moe_forward(cur, s["logits"][i], ly, y=s["y"][i], ws=s["ws"], c_layer=s["cl"][i])
        return cur
    q = wq.pack(s["w"], c["group"], c["bits"], out=s["out"])
    return {"codes": q.codes, "meta": q.meta}


# ---- what a pass cannot do without ------------------------------------------

def _packed(n, k, bits, group):
    if bits == 16:
        return 2.0 * n * k
    return n * k * bits / 8.0 + n * (k / group) * 4.0


def work(case):
    c = case
    d, inter, kind, m = c["d"], c["inter"], c["kind"], c.get("m", 0)
    n, r = c.get("layers", 1), c.get("r", 0)
    if kind == "pack":
        return {"bytes": 4.0 * d * inter + _packed(inter, d, c["bits"], c["group"]), "flops": 0.0}
    if kind == "dense" or kind == "down":
        b = _packed(d, inter, 16 if kind == "dense" else 4, c.get("group", 128))
        b += 2.0 * m * inter + m * d * ((4 if c["f32"] else 2) + (2 if c["residual"] else 0))
        return {"bytes": b, "flops": 2.0 * m * d * inter}
    gu = 2 * _packed(inter, d, c["bits"], c["group"]) + 2.0 * r * (2 * d + 2 * inter)
    gu_flops = 2.0 * m * (2 * d * inter + 2 * r * (d + inter))
    if kind == "gateup":
        return {"bytes": gu + 2.0 * m * (d + inter), "flops": gu_flops}
    layer = gu + _packed(d, inter, c.get("down_bits", 4), c.get("group_down", c["group"]))
    flops = gu_flops + 2.0 * m * d * inter
    if kind == "moe":
        e, k = c["experts"], c["top_k"]
        used = e * (1.0 - (1.0 - k / e) ** m)  # experts that m tokens pick, on average
        return {"bytes": n * (used * layer + 4.0 * m * e) + 4.0 * m * d, "flops": n * k * flops}
    if kind == "decoder":
        h, kv, hd, ctx = c["heads"], c["kv"], c["hd"], c["ctx"]
        mean = ctx if m == 1 else 0.625 * ctx
        attn = _packed((h + 2 * kv) * hd, d, 4, 128) + _packed(d, h * hd, 4, 64) + 4.0 * m * kv * hd * mean
        aflops = 2.0 * m * d * (2 * h + 2 * kv) * hd + 4.0 * m * h * hd * mean
        return {"bytes": n * (layer + attn) + 4.0 * m * d, "flops": n * (flops + aflops)}
    return {"bytes": n * layer + 4.0 * m * d, "flops": n * flops}


# About four times the error measured against `exact`: one bf16 store gives 1.7e-3, each further layer of a stack
# 1.1e-3 more (rounding flips travel on: 2 layers 2.5e-3, 8 layers 8e-3 to 9e-3); fp32 output 2.9e-6.
def tolerance(case):
    kind = case["kind"]
    if kind == "pack":
        return "exact"
    if case.get("f32"):
        return {"rel": 1.2e-5}
    return {"rel": min(0.03, 0.003 + 0.0045 * case.get("layers", 1))}


# ---- the same in 64 bits ------------------------------------------------------

def _quantized(w, bits, group):
    """fp64 values of the group-quantized matrix: asymmetric min-max round-to-nearest in fp32, fp16 scales."""
    n, k = w.shape
    g = w.view(n, k // group, group)
    lo, hi = g.amin(2, keepdim=True), g.amax(2, keepdim=True)
    qmax = float((1 << bits) - 1)
    s = ((hi - lo) / qmax).to(torch.float16).to(torch.float32)
    s = torch.where(s == 0, torch.ones_like(s), s)
    z = torch.clamp(torch.round(-lo / s), 0.0, qmax)
    q = torch.clamp(torch.round(g / s) + z, 0.0, qmax)
    return ((q.double() - z.double()) * s.double()).view(n, k)


def _bf16(t):
    return t.to(torch.bfloat16).double()


def _rms(x):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + EPS)


def _gateup64(x, wg, wu, lora, scale, prenorm=True):
    xin = _rms(x) if prenorm else x
    g, u = xin @ wg.T, xin @ wu.T
    if lora is not None:
        a, bg, bu = (t.double() for t in lora)
        r = bg.shape[1]
        g = g + scale * (xin @ a[:r].T) @ bg.T
        u = u + scale * (xin @ a[r:].T) @ bu.T
    return g * torch.sigmoid(g) * u


def _mlp64(c, rnd, i, x):
    wg, wu, wd, lora = _mlp_draws(c, rnd, i)
    h = _bf16(_gateup64(x, _quantized(wg, c["bits"], c["group"]), _quantized(wu, c["bits"], c["group"]), lora, _scale(c)))
    wd = wd.to(torch.bfloat16).double() if c.get("down_bits", 4) == 16 else \
        _quantized(wd, 4, c.get("group_down", c["group"]))
    return x + h @ wd.T


def _rope64(v, pos, theta=1e6):
    """v [B, heads, hd] at positions pos [B]: element i pairs with i + hd/2."""
    hd = v.shape[-1]
    inv = theta ** (-2.0 * torch.arange(hd // 2, device=v.device, dtype=torch.float64) / hd)
    a = pos.double()[:, None, None] * inv
    lo, hi = v[..., :hd // 2], v[..., hd // 2:]
    return torch.cat([lo * torch.cos(a) - hi * torch.sin(a), hi * torch.cos(a) + lo * torch.sin(a)], -1)


def _decoder64(c, rnd):
    m, d, h, kv, hd = c["m"], c["d"], c["heads"], c["kv"], c["hd"]
    x, lens, caches = rnd.bf16((m, d), 1).double(), rnd.lens(m, c["ctx"], 2).long(), []
    rows = torch.arange(m, device=DEV)
    for i in range(c["layers"]):
        k = 16 * (i + 1)
        wqkv = _quantized(rnd.normal(((h + 2 * kv) * hd, d), k + 8, 0.02), 4, 128)
        wo = _quantized(rnd.normal((d, h * hd), k + 9, 0.02), 4, 64)
        kc, vc = rnd.bf16((m, kv, c["ctx"], hd), k + 10), rnd.bf16((m, kv, c["ctx"], hd), k + 11)
        qkv = (_rms(x) @ wqkv.T).view(m, h + 2 * kv, hd)
        q, kn, vn = qkv[:, :h], qkv[:, h:h + kv], qkv[:, h + kv:]
        q, kn = _rope64(_rms(q), lens), _rope64(_rms(kn), lens)
        kc[rows, :, lens] = kn.to(torch.bfloat16)
        vc[rows, :, lens] = vn.to(torch.bfloat16)
        o = torch.empty((m, h, hd), dtype=torch.float64, device=DEV)
        for b in range(m):
            n = int(lens[b]) + 1
            kb, vb = kc[b, :, :n].double(), vc[b, :, :n].double()
            p = torch.softmax(q[b].view(kv, h // kv, hd) @ kb.transpose(1, 2) / math.sqrt(hd), -1)
            o[b] = (p @ vb).view(h, hd)
        x1 = _bf16(x + _bf16(o.view(m, h * hd)) @ wo.T)
        y = _mlp64(c, rnd, i, x1)
        caches.append((kc.double(), vc.double()))
        x = _bf16(y)
    return {"y": y, "caches": caches}


def _moe64(c, rnd):
    m, d, inter, e, k, r = c["m"], c["d"], c["inter"], c["experts"], c["top_k"], c["r"]
    x = rnd.bf16((m, d), 1).double()
    for i in range(c["layers"]):
        wg, wu, wd, lora = _mlp_draws(c, rnd, i, e)
        top, idx = rnd.normal((m, e), 16 * (i + 1) + 8).double().topk(k, 1)
        p = torch.softmax(top, 1)
        y = x.clone()
        for j in range(e):
            t, slot = (idx == j).nonzero(as_tuple=True)
            if not len(t):
                continue
            own = slice(j * inter, (j + 1) * inter)
            la = None if lora is None else (lora[0][j * 2 * r:(j + 1) * 2 * r], lora[1][own], lora[2][own])
            h = _bf16(_gateup64(x[t], _quantized(wg[own], c["bits"], c["group"]),
                                _quantized(wu[own], c["bits"], c["group"]), la, _scale(c)))
            y.index_add_(0, t, p[t, slot][:, None] * (h @ _quantized(wd[j * d:(j + 1) * d], 4, c["group"]).T))
        x = _bf16(y)
    return y


def exact(case, seed):
    c, rnd = case, _Rand(seed)
    d, inter, kind, m = c["d"], c["inter"], c["kind"], c.get("m", 0)
    if kind == "pack":
        return None  # whole numbers
    if kind == "decoder":
        return _decoder64(c, rnd)
    if kind == "moe":
        return _moe64(c, rnd)
    if kind in ("down", "dense"):
        w = rnd.normal((d, inter), 18, 0.02)
        w = w.to(torch.bfloat16).double() if kind == "dense" else _quantized(w, 4, c["group"])
        y = rnd.bf16((m, inter), 1, 0.5).double() @ w.T
        return y + rnd.bf16((m, d), 2).double() if c["residual"] else y
    x = rnd.bf16((m, d), 1).double()
    if kind == "gateup":
        wg, wu, _, lora = _mlp_draws(c, rnd, 0)
        return _gateup64(x, _quantized(wg, c["bits"], c["group"]), _quantized(wu, c["bits"], c["group"]), lora,
                         _scale(c), c["prenorm"])
    for i in range(c["layers"]):
        y = _mlp64(c, rnd, i, x)
        x = _bf16(y)
    return y
