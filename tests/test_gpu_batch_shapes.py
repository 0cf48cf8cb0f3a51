"""The batched-decode launches at more shapes and counts of 9 to 64 tokens vs the
fp64 oracle.

Covers token counts at the edges of the 8-token tiles (9, 12, 16, 17, 24, 33, 40,
48, 64), ragged row blocks and feature blocks, every group size, the adapter, the
RMSNorm, row blocks in few and in many parts (a row block of 64 feature blocks is
spread over up to 32 CTAs), 4-bit gate/up, down with a residual in bf16 and fp32,
and a stack of two 8B-shaped layers at 16 tokens.  Products are exact and sums
fp32: the bound and the share of bit-equal outputs are check_bf16's defaults.
"""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2606_04238_gb300 import synth
from tests.gpu_util import check_bf16, check_f32, upload_packed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wq():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_04238_gb300 import wq as mod
    return mod


def _q(shape, group, bits, seed):
    w = (np.random.default_rng(seed).standard_normal(shape) * 0.02).astype(np.float32)
    return orc.quantize(w, group, bits)[:3]


GATEUP_CASES = [
    # d, inter, group, r, token counts
    (4096, 256, 128, 16, (9, 16, 33, 64)),   # 2 row blocks of 32 units each
    (4096, 200, 64, 8, (12, 48)),            # ragged rows, 2 row blocks
    (512, 1024, 32, 0, (17, 64)),            # 8 row blocks of 4 units, no adapter
    (384, 640, 128, 32, (17, 40)),           # 5 row blocks of 3 units
]


@pytest.mark.parametrize("d,inter,group,r,ms", GATEUP_CASES)
@pytest.mark.parametrize("prenorm", [False, True])
def test_batch_gateup(wq, d, inter, group, r, ms, prenorm):
    qg, qu = _q((inter, d), group, 2, d + inter), _q((inter, d), group, 2, d + inter + 1)
    g, u = upload_packed(*qg, group, 2), upload_packed(*qu, group, 2)
    kw, okw = {}, {}
    if r:
        a, bg, bu = synth.lora(d, inter, r, d + r)
        kw = dict(lora_a=a.cuda(), lora_b_gate=bg.cuda(), lora_b_up=bu.cuda())
        okw = dict(lora_a=synth.bf16_bits(a), lora_b_gate=synth.bf16_bits(bg), lora_b_up=synth.bf16_bits(bu))
    for m in ms:
        x = synth.activations((m, d), 10 + m)
        h = wq.gateup_w2_lora(x.cuda(), g, u, lora_scale=2.0, prenorm=prenorm, **kw)
        torch.cuda.synchronize()
        assert wq.device_status() == 0
        ref, _ = orc.gateup(synth.bf16_bits(x), qg, qu, group, okw.get("lora_a"), okw.get("lora_b_gate"),
                            okw.get("lora_b_up"), lora_scale=2.0, prenorm=prenorm)
        check_bf16(h, ref, f"batch h d={d} I={inter} g={group} r={r} m={m} prenorm={prenorm}")


@pytest.mark.parametrize("m", [17, 64])
def test_batch_gateup_w4(wq, m):
    d, inter, group = 512, 384, 64
    qg, qu = _q((inter, d), group, 4, 15), _q((inter, d), group, 4, 16)
    x = synth.activations((m, d), 17 + m)
    h = wq.gateup_w4(x.cuda(), upload_packed(*qg, group, 4), upload_packed(*qu, group, 4), prenorm=True)
    torch.cuda.synchronize()
    assert wq.device_status() == 0
    ref, _ = orc.gateup(synth.bf16_bits(x), qg, qu, group, None, None, None, lora_scale=0.0, prenorm=True)
    check_bf16(h, ref, f"batch W4 h m={m}")


DOWN_CASES = [
    # d (output rows), inter (features), group, token counts
    (384, 8192, 128, (17, 33, 64)),   # 3 row blocks of 64 units, 2 a CTA
    (4096, 512, 64, (9, 16)),         # 32 row blocks of 4 units
    (200, 1024, 32, (24,)),           # ragged rows
]


@pytest.mark.parametrize("d,inter,group,ms", DOWN_CASES)
def test_batch_down(wq, d, inter, group, ms):
    qd = _q((d, inter), group, 4, d * 3 + inter)
    dn = upload_packed(*qd, group, 4)
    for m in ms:
        h = (synth.activations((m, inter), 20 + m) * 0.5).to(torch.bfloat16)
        res = synth.activations((m, d), 30 + m)
        y = wq.down_w4(h.cuda(), dn, residual=res.cuda())
        y0 = wq.down_w4(h.cuda(), dn)
        y32 = wq.down_w4(h.cuda(), dn, residual=res.cuda(), out_f32=True)
        torch.cuda.synchronize()
        assert wq.device_status() == 0
        ref, _ = orc.down(synth.bf16_bits(h), qd, group, synth.bf16_bits(res))
        ref0, _ = orc.down(synth.bf16_bits(h), qd, group, None)
        check_bf16(y, ref, f"batch y d={d} I={inter} g={group} m={m}")
        check_bf16(y0, ref0, f"batch y (no residual) d={d} m={m}")
        check_f32(y32, ref, f"batch y fp32 d={d} m={m}")


def test_batch_is_deterministic(wq):
    d, inter, group = 384, 8192, 128
    qd = _q((d, inter), group, 4, 7)
    dn = upload_packed(*qd, group, 4)
    h = synth.activations((33, inter), 8).cuda()
    ys = [wq.down_w4(h, dn) for _ in range(3)]
    torch.cuda.synchronize()
    assert all(torch.equal(ys[0].view(torch.int16), y.view(torch.int16)) for y in ys[1:])


def test_batch_stack_8b_16_tokens(wq):
    """Two 8B-shaped layers at 16 tokens through wq_mlp_forward (the batched
    chain), each kernel teacher-forced on sampled tokens."""
    cfg = synth.CONFIGS["dense_8b"]
    m = 16
    layers, ents = [], []
    for l in range(2):
        wg, wu, wd = synth.layer_weights(cfg, l)
        qg = orc.quantize(wg.numpy(), cfg.group_gu, 2)[:3]
        qu = orc.quantize(wu.numpy(), cfg.group_gu, 2)[:3]
        qd = orc.quantize(wd.numpy(), cfg.group_down, 4)[:3]
        a, bg, bu = synth.lora(cfg.d, cfg.inter, cfg.r, 300 + l)
        layers.append(wq.MLPLayer(upload_packed(*qg, cfg.group_gu, 2), upload_packed(*qu, cfg.group_gu, 2),
                                  upload_packed(*qd, cfg.group_down, 4), lora_a=a.cuda(), lora_b_gate=bg.cuda(),
                                  lora_b_up=bu.cuda(), lora_scale=cfg.lora_scale))
        ents.append(dict(g=qg, u=qu, d=qd, a=synth.bf16_bits(a), bg=synth.bf16_bits(bg), bu=synth.bf16_bits(bu)))
    assert wq.mlp_forward_info(m, layers, prenorm=True)["route"] == wq.ROUTE_GEMM_CHAIN
    x = synth.activations((m, cfg.d), 310).cuda()
    _, states, h_states = wq.mlp_forward_states(x, layers, prenorm=True, with_h=True)
    torch.cuda.synchronize()
    assert wq.device_status() == 0
    rows = np.array([0, 5, 15])
    prev = synth.bf16_bits(x.cpu())
    for l, e in enumerate(ents):
        h_ref, _ = orc.gateup(prev[rows], e["g"], e["u"], cfg.group_gu, e["a"], e["bg"], e["bu"],
                              lora_scale=cfg.lora_scale, prenorm=True)
        check_bf16(h_states[l][rows], h_ref, f"8B m=16 layer {l} h")
        y_ref, _ = orc.down(synth.bf16_bits(h_states[l][rows].cpu()), e["d"], cfg.group_down, prev[rows])
        check_bf16(states[l][rows], y_ref, f"8B m=16 layer {l} y")
        prev = synth.bf16_bits(states[l].cpu())
