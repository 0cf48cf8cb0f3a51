"""The batched-decode kernels (9 to 64 tokens, fewer for large matrices) vs the fp64 oracle at the sizes
where their split can go wrong: every count of 8-token tiles and its edges,
ragged row blocks and feature blocks, one unit to many parts a row block,
adapter ranks that are no multiple of 16, every code width and group, rows
that are no multiple of 4 (scalar stores), the panel gate/up hands down, and
the slots of a mixture of experts grouped by expert.

Products are exact and sums fp32, so the bound and the share of bit-equal
bf16 outputs are those of the other decode kernels (check_bf16's defaults).
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


GATEUP = [
    # bits, d, inter, group, r, token counts
    (2, 128, 16, 128, 0, (9, 64)),             # one unit in all
    (2, 2048, 130, 64, 24, (10, 17, 25)),      # two row blocks, the second with 2 rows; rank 24
    (2, 96, 1000, 32, 8, (33, 41, 49)),        # less than a feature block; rank 8
    (3, 640, 384, 32, 16, (9, 31, 57)),
    (3, 512, 200, 128, 64, (16, 48)),
    (4, 1152, 264, 64, 0, (24, 40, 64)),
    (2, 2560, 6144, 128, 16, (2, 8)),          # few tokens: launches of 30M weights and more
]


@pytest.mark.parametrize("bits,d,inter,group,r,ms", GATEUP)
def test_batch_gateup(wq, bits, d, inter, group, r, ms):
    qg, qu = _q((inter, d), group, bits, d + inter), _q((inter, d), group, bits, d + inter + 1)
    g, u = upload_packed(*qg, group, bits), upload_packed(*qu, group, bits)
    kw, bl = {}, (None, None, None)
    if r:
        a, bg, bu = synth.lora(d, inter, r, d + r)
        kw = dict(lora_a=a.cuda(), lora_b_gate=bg.cuda(), lora_b_up=bu.cuda())
        bl = tuple(synth.bf16_bits(t) for t in (a, bg, bu))
    for m in ms:
        x = synth.activations((m, d), 10 + m)
        for prenorm in (True, False):
            if bits == 4:
                h = wq.gateup_w4(x.cuda(), g, u, prenorm=prenorm)
            else:
                fn = wq.gateup_w2_lora if bits == 2 else wq.gateup_w3_lora
                h = fn(x.cuda(), g, u, lora_scale=2.0, prenorm=prenorm, **kw)
            torch.cuda.synchronize()
            assert wq.device_status() == 0
            ref, _ = orc.gateup(synth.bf16_bits(x), qg, qu, group, *bl, lora_scale=2.0 if r else 0.0, prenorm=prenorm)
            check_bf16(h, ref, f"batch h bits={bits} d={d} I={inter} g={group} r={r} m={m} prenorm={prenorm}")


DOWN = [
    # d, inter, group, token counts
    (16, 128, 128, (9, 13)),
    (202, 1056, 32, (12, 64)),        # rows no multiple of 4; ragged feature block
    (130, 20480, 128, (17, 63)),      # 2 row blocks, 160 blocks: about 76 parts each
    (2560, 704, 64, (32, 33)),
    (4096, 20480, 128, (1, 3)),       # few tokens: 80M weights and more
]


@pytest.mark.parametrize("d,inter,group,ms", DOWN)
def test_batch_down(wq, d, inter, group, ms):
    qd = _q((d, inter), group, 4, d * 3 + inter)
    dn = upload_packed(*qd, group, 4)
    for m in ms:
        h = (synth.activations((m, inter), 20 + m) * 0.5).to(torch.bfloat16)
        res = synth.activations((m, d), 30 + m)
        y = wq.down_w4(h.cuda(), dn, residual=res.cuda())
        y32 = wq.down_w4(h.cuda(), dn, out_f32=True)
        torch.cuda.synchronize()
        assert wq.device_status() == 0
        ref, _ = orc.down(synth.bf16_bits(h), qd, group, synth.bf16_bits(res))
        ref0, _ = orc.down(synth.bf16_bits(h), qd, group, None)
        check_bf16(y, ref, f"batch y d={d} I={inter} g={group} m={m}")
        check_f32(y32, ref0, f"batch y fp32 d={d} m={m}")


@pytest.mark.parametrize("bits,group,group_down,r", [(2, 64, 32, 8), (3, 32, 128, 16), (4, 128, 64, 0)])
@pytest.mark.parametrize("m", [9, 40])
def test_batch_stack_hands_down_the_panel(wq, bits, group, group_down, r, m):
    """Two layers through wq_mlp_forward, each kernel teacher-forced; the run that
    keeps h and the run that only hands on its panel give the same y."""
    d, inter = 384, 896
    layers, ents = [], []
    for l in range(2):
        qg, qu = _q((inter, d), group, bits, 70 + l), _q((inter, d), group, bits, 80 + l)
        qd = _q((d, inter), group_down, 4, 90 + l)
        kw, bl = {}, (None, None, None)
        if r:
            a, bg, bu = synth.lora(d, inter, r, 50 + l)
            kw = dict(lora_a=a.cuda(), lora_b_gate=bg.cuda(), lora_b_up=bu.cuda(), lora_scale=2.0)
            bl = tuple(synth.bf16_bits(t) for t in (a, bg, bu))
        layers.append(wq.MLPLayer(upload_packed(*qg, group, bits), upload_packed(*qu, group, bits),
                                  upload_packed(*qd, group_down, 4), **kw))
        ents.append((qg, qu, qd, bl))
    x = synth.activations((m, d), 7).cuda()
    ws = wq.workspace(m, d, inter, r)
    y, states, h_states = wq.mlp_forward_states(x, layers, prenorm=True, ws=ws, with_h=True)
    y_plain = wq.mlp_forward(x, layers, prenorm=True, ws=ws)
    torch.cuda.synchronize()
    assert wq.device_status() == 0
    assert torch.equal(y.view(torch.int16), y_plain.view(torch.int16))
    prev = synth.bf16_bits(x.cpu())
    for l, (qg, qu, qd, bl) in enumerate(ents):
        ref, _ = orc.gateup(prev, qg, qu, group, *bl, lora_scale=2.0 if r else 0.0, prenorm=True)
        check_bf16(h_states[l], ref, f"batch stack bits={bits} m={m} layer {l} h")
        ref, _ = orc.down(synth.bf16_bits(h_states[l].cpu()), qd, group_down, prev)
        check_bf16(states[l], ref, f"batch stack bits={bits} m={m} layer {l} y")
        prev = synth.bf16_bits(states[l].cpu())


@pytest.mark.parametrize("m,E,k,r,skew", [
    (30, 16, 2, 8, 0.0),    # 60 slots, segments of up to 8
    (33, 8, 2, 24, 0.0),    # 66 slots, segments of up to 16; rank 24
    (64, 4, 3, 0, 0.0),     # 192 slots, segments of up to 32
    (64, 32, 1, 8, 9.0),    # every token takes expert 0: eight segments, 31 experts unread
])
def test_routed_batch(wq, m, E, k, r, skew):
    from tests.test_gpu_moe import _build, _check_block
    d, inter, group = 1120, 992, 32  # ragged feature blocks and row blocks
    layer, ents = _build(wq, d, inter, E, k, group, r, 300 + m)
    x = synth.activations((m, d), 11 + m)
    lg = np.random.default_rng(5 + m).standard_normal((m, E)).astype(np.float32)
    lg[:, 0] += skew
    _check_block(wq, layer, ents, x, torch.from_numpy(lg), group, f"routed m={m} E={E} k={k}", 2.0 if r else 0.0)


@pytest.mark.parametrize("bits,m", [(2, 2), (3, 1)])
def test_batch_stack_of_a_large_layer(wq, bits, m):
    """One layer of 50M weights a matrix takes the batched chain at a few tokens."""
    d, inter, group, r = 4096, 12800, 128, 8
    qg, qu, qd = _q((inter, d), group, bits, 1), _q((inter, d), group, bits, 2), _q((d, inter), group, 4, 3)
    a, bg, bu = synth.lora(d, inter, r, 4)
    layer = wq.MLPLayer(upload_packed(*qg, group, bits), upload_packed(*qu, group, bits), upload_packed(*qd, group, 4),
                        lora_a=a.cuda(), lora_b_gate=bg.cuda(), lora_b_up=bu.cuda(), lora_scale=2.0)
    assert wq.mlp_forward_info(m, [layer])["route"] == wq.ROUTE_GEMM_CHAIN
    x = synth.activations((m, d), 5).cuda()
    y, _, h = wq.mlp_forward_states(x, [layer], prenorm=True, with_h=True)
    torch.cuda.synchronize()
    assert wq.device_status() == 0
    bl = tuple(synth.bf16_bits(t) for t in (a, bg, bu))
    ref, _ = orc.gateup(synth.bf16_bits(x.cpu()), qg, qu, group, *bl, lora_scale=2.0, prenorm=True)
    check_bf16(h[0], ref, f"large layer h bits={bits} m={m}")
    ref, _ = orc.down(synth.bf16_bits(h[0].cpu()), qd, group, synth.bf16_bits(x.cpu()))
    check_bf16(y, ref, f"large layer y bits={bits} m={m}")


@pytest.mark.parametrize("m", [3, 8, 12])
def test_fp32_down_of_activations_of_one_sign(wq, m):
    """Activations of mean 0.5: a group's code sum and its zero-point term are many times
    their difference.  The error against 64 bits stays below 9e-7 of the result (6e-7
    measured, 7.5e-7 on the GEMV kernels); the two terms added to the total one after
    the other, the first from one chain of 8 MMAs, make it 1.8e-6 to 2.0e-6."""
    d, inter, group = 2560, 20480, 128
    gen = torch.Generator("cuda").manual_seed(m)
    w = torch.randn((d, inter), device="cuda", generator=gen) * 0.02
    q = wq.pack(w, group, 4)
    g = w.view(d, -1, group)
    lo, hi = g.amin(2, keepdim=True), g.amax(2, keepdim=True)
    s = ((hi - lo) / torch.full_like(hi, 15)).half().float()
    z = (-lo / s).round().clamp(0, 15)
    deq = ((((g / s).round() + z).clamp(0, 15) - z).double() * s.double()).view(d, inter)
    h = (torch.randn((m, inter), device="cuda", generator=gen) * 0.5 + 0.5).to(torch.bfloat16)
    ref = h.double() @ deq.T
    y = wq.down_w4(h, q, out_f32=True)
    assert float((y.double() - ref).norm() / ref.norm()) < 9e-7


def _cancelling_adapter(d, inter, r, gen):
    """Weights of value zero and an adapter whose large products cancel: the rows of A
    come in pairs whose products with x differ by x[0] (x and A are integers, so every
    fp32 sum is exact), and B subtracts one from the other.  Returns (gate, up, A, Bg, Bu)."""
    pairs = gen.integers(1, 128, (r, d)).astype(np.float32)  # row 2 i of gate, then of up
    a = np.repeat(pairs.reshape(r, 1, d), 2, 1).reshape(2 * r, d)
    a[1::2, 0] += 1
    b = [np.tile(np.array([-1, 1], np.float32) * (1 + i), (inter, r // 2)) / 16 for i in range(2)]
    z = (np.zeros((inter, d), np.uint8), np.full((inter, d // 64), 0x3C00, np.uint16), np.zeros((inter, d // 64), np.uint16))
    return z, *(torch.from_numpy(v).to(torch.bfloat16) for v in (a, *b))


@pytest.mark.parametrize("bits,d,inter,r,m", [(2, 256, 144, 8, 9), (2, 512, 768, 32, 24), (3, 256, 200, 64, 33),
                                              (2, 1024, 400, 16, 64)])
def test_adapter_products_are_kept_in_fp32(wq, bits, d, inter, r, m):
    """t = x A^T of 2^20 and more whose differences are 1 to 64: with fewer than 24 bits
    in t the difference is lost.  Exact sums, so h is the exact value rounded twice at
    most (fp32 SiLU, bf16)."""
    gen = np.random.default_rng(d + r)
    z, a, bg, bu = _cancelling_adapter(d, inter, r, gen)
    q = upload_packed(*z, 64, bits)
    x = gen.integers(64, 128, (m, d)).astype(np.float32)
    x[:, 0] = gen.integers(1, 65, m)
    fn = wq.gateup_w2_lora if bits == 2 else wq.gateup_w3_lora
    h = fn(torch.from_numpy(x).to(torch.bfloat16).cuda(), q, q, a.cuda(), bg.cuda(), bu.cuda(), lora_scale=0.25)
    g = x[:, :1].astype(np.float64) * 0.25 * (r / 2) / 16  # r / 2 pairs of weight 1 / 16
    ref = np.broadcast_to(g / (1 + np.exp(-g)) * (2 * g), (m, inter))
    got = h.float().cpu().numpy().astype(np.float64)
    # half a bf16 unit and 16 fp32 ones for the SiLU's exponential and quotient
    assert (np.abs(got - ref) <= np.abs(ref) * (2.0 ** -8 + 2.0 ** -20)).all(), np.abs(got / ref - 1).max()


@pytest.mark.parametrize("m,E,k,r", [(16, 4, 2, 8), (40, 8, 4, 24)])
def test_grouped_expert_adapter_products_are_kept_in_fp32(wq, m, E, k, r):
    d, inter = 2048, 1024
    gen = np.random.default_rng(m + E)
    z, a, bg, bu = _cancelling_adapter(d, inter, r, gen)
    st = lambda t: torch.cat([t] * E).contiguous().cuda()
    zz = upload_packed(*(np.concatenate([v] * E) for v in z), 64, 2)
    down = wq.pack(torch.randn((E * d, inter), device="cuda", generator=torch.Generator("cuda").manual_seed(1)) * 0.02, 64, 4)
    layer = wq.MoELayer(wq.MLPLayer(zz, zz, down, lora_a=st(a), lora_b_gate=st(bg), lora_b_up=st(bu), lora_scale=0.25),
                        E, k)
    x = gen.integers(8, 16, (m, d)).astype(np.float32)
    x[:, 0] = gen.integers(1, 65, m)
    lg = torch.from_numpy(gen.standard_normal((m, E)).astype(np.float32)).cuda()
    _, _, _, hs, _ = wq.moe_forward(torch.from_numpy(x).to(torch.bfloat16).cuda(), lg, layer, prenorm=False,
                                    with_slots=True)
    g = np.repeat(x[:, :1].astype(np.float64), k, 0) * 0.25 * (r / 2) / 16
    ref = np.broadcast_to(g / (1 + np.exp(-g)) * (2 * g), hs.shape)
    got = hs.float().cpu().numpy().astype(np.float64)
    assert (np.abs(got - ref) <= np.abs(ref) * (2.0 ** -8 + 2.0 ** -20)).all(), np.abs(got / ref - 1).max()


def test_moe_workspace_of_several_token_counts(wq):
    """One workspace for the largest token count serves smaller ones in between,
    on the slots' and the grouped launches."""
    from tests.test_gpu_moe import _build
    d, inter, E, k, group = 1024, 512, 8, 2, 64
    layer, _ = _build(wq, d, inter, E, k, group, 8, 900)
    ws = wq.moe_workspace(64, layer)
    for i, m in enumerate((64, 1, 7, 6, 33, 2, 64, 12)):
        x = synth.activations((m, d), 60 + i).cuda()
        lg = torch.from_numpy(np.random.default_rng(70 + i).standard_normal((m, E)).astype(np.float32)).cuda()
        y, y0 = wq.moe_forward(x, lg, layer, ws=ws).clone(), wq.moe_forward(x, lg, layer)
        assert torch.equal(y.view(torch.int16), y0.view(torch.int16)), m
    assert wq.device_status() == 0


def test_decoder_workspace_of_several_batches(wq):
    """One workspace for the largest batch serves smaller ones in between."""
    d, inter, H, kv, hd, max_len = 512, 896, 4, 2, 128, 64
    mk = lambda n, kk, bits, s: upload_packed(*_q((n, kk), 64, bits, s), 64, bits)
    layer = wq.DecoderLayer(mk((H + 2 * kv) * hd, d, 4, 1), mk(d, H * hd, 4, 2),
                            wq.MLPLayer(mk(inter, d, 2, 3), mk(inter, d, 2, 4), mk(d, inter, 4, 5)), H, kv, hd, 1e6)
    ws = wq.decoder_workspace(24, layer, max_len)
    for i, b in enumerate((24, 12, 1, 17, 9, 24)):
        x = synth.activations((b, d), 80 + i).cuda()
        lens = torch.full((b,), 10 + i, dtype=torch.int32, device="cuda")
        kc, vc = (synth.activations((b, kv, max_len, hd), 90 + j).cuda() for j in range(2))
        y = wq.decoder_layer_forward(x, lens, layer, kc, vc, ws=ws).clone()
        y0 = wq.decoder_layer_forward(x, lens, layer, kc, vc)
        assert torch.equal(y.view(torch.int16), y0.view(torch.int16)), b
    assert wq.device_status() == 0


@pytest.mark.parametrize("d,inter,H,group,big,split", [
    (5120, 17408, 40, 32, 25, (8, 7)),  # q/k/v and output projection of a batch of 8 and 7
    (1024, 8192, 40, 64, 17, (12, 11)),  # output projection of a batch of 12 and 11
])
def test_decoder_workspace_of_several_batches_with_split_projections(wq, d, inter, H, group, big, split):
    """The same where a GEMV launch of the projections splits its rows over feature
    panels, whose arrival counters have to be zero when it starts: a larger batch
    fills the workspace's buffers before."""
    kv, hd, max_len = 8, 128, 64
    nqkv = (H + 2 * kv) * hd
    for b in split:
        assert wq.plan_info(wq.KIND_DOWN_W4, d, H * hd, b, group)["panels"] > 1
    gen = torch.Generator("cuda").manual_seed(5)
    mk = lambda n, kk, bits: wq.pack(torch.randn((n, kk), device="cuda", generator=gen) * 0.02, group, bits)
    layer = wq.DecoderLayer(mk(nqkv, d, 4), mk(d, H * hd, 4),
                            wq.MLPLayer(mk(inter, d, 2), mk(inter, d, 2), mk(d, inter, 4)), H, kv, hd, 1e6)
    ws = wq.decoder_workspace(big, layer, max_len)
    for i, b in enumerate((big, split[0], big, split[1])):
        x = synth.activations((b, d), 180 + i).cuda()
        lens = torch.full((b,), 10 + i, dtype=torch.int32, device="cuda")
        kc, vc = (synth.activations((b, kv, max_len, hd), 190 + j).cuda() for j in range(2))
        y = wq.decoder_layer_forward(x, lens, layer, kc, vc, ws=ws).clone()
        y0 = wq.decoder_layer_forward(x, lens, layer, kc, vc)
        assert torch.equal(y.view(torch.int16), y0.view(torch.int16)), b
    assert wq.device_status() == 0


@pytest.mark.parametrize("m,E,k", [(1, 256, 12), (3, 33, 4), (12, 2, 1)])
def test_slots_find_their_experts(wq, m, E, k):
    """At most 12 slots: the gate/up launch and the routing launch rank the experts
    alike -- ties, signed zeros, negative and extreme logits."""
    from tests.test_gpu_moe import _build, _check_block
    d, inter, group = 64, 32, 32
    layer, ents = _build(wq, d, inter, E, k, group, 8, 700 + E)
    x = synth.activations((m, d), 17 + m)
    lg = np.random.default_rng(40 + E).integers(-3, 2, (m, E)).astype(np.float32)  # many ties
    lg[:, ::3] *= -0.0
    lg[0, E // 2], lg[0, -1], lg[0, 0] = 3e38, 1e-40, -3e38
    _check_block(wq, layer, ents, x, torch.from_numpy(lg), group, f"slots m={m} E={E} k={k}", 2.0)


@pytest.mark.parametrize("m,k", [(40, 3), (64, 6)])
def test_routed_batch_of_two_ctas_an_sm(wq, m, k):
    """Row blocks enough for two CTAs an SM (of 128 rows: 27 gate/up and 28 down ones an
    expert), with one and two token tiles a segment; sampled slots."""
    d, inter, E, group, r = 3488, 3424, 33, 32, 8
    n = lambda rows, cols, bits, s: wq.pack(torch.randn((rows, cols), device="cuda",
                                                        generator=torch.Generator("cuda").manual_seed(s)) * 0.02, group, bits)
    _, bg, bu = synth.lora(d, E * inter, r, 5)
    a_all = synth.weights((E * 2 * r, d), 6, std=0.01).to(torch.bfloat16)
    g, u, dn = n(E * inter, d, 2, 1), n(E * inter, d, 2, 2), n(E * d, inter, 4, 3)
    layer = wq.MoELayer(wq.MLPLayer(g, u, dn, lora_a=a_all.cuda(), lora_b_gate=bg.cuda(), lora_b_up=bu.cuda(),
                                    lora_scale=2.0), E, k)
    x = synth.activations((m, d), 8).cuda()
    lg = torch.from_numpy(np.random.default_rng(9).standard_normal((m, E)).astype(np.float32)).cuda()
    y, idx, wt, hs, ys = wq.moe_forward(x, lg, layer, with_slots=True)
    # the slots one by one on the single-expert calls
    sub = lambda q, e, rows: wq.QWeight(q.codes.view(E, -1)[e].contiguous(), q.meta.view(E, -1)[e].contiguous(),
                                        rows, q.k, q.group, q.bits)
    for s in range(0, m * k, 17):
        e, t = int(idx.view(-1)[s]), s // k
        h1 = wq.gateup_w2_lora(x[t:t + 1], sub(g, e, inter), sub(u, e, inter),
                               a_all.cuda()[e * 2 * r:(e + 1) * 2 * r].contiguous(),
                               bg.cuda()[e * inter:(e + 1) * inter].contiguous(),
                               bu.cuda()[e * inter:(e + 1) * inter].contiguous(), lora_scale=2.0, prenorm=True)
        y1 = wq.down_w4(hs[s:s + 1].contiguous(), sub(dn, e, d), out_f32=True)
        # both are fp32 sums of exact products: one bf16 rounding apart at most, 1e-4 of the largest for fp32
        dh = (hs[s].float() - h1[0].float()).abs()
        assert (dh <= h1[0].float().abs() * 2.0 ** -7 + 1e-5).all() and (dh == 0).float().mean() > 0.97, s
        assert ((ys[s] - y1[0]).abs() <= 1e-4 * y1.abs().max()).all(), s
    torch.cuda.synchronize()
    assert wq.device_status() == 0


@pytest.mark.parametrize("E,k", [(8, 4), (33, 5)])
def test_grouped_experts_rank_as_the_slots_do(wq, E, k):
    """Enough slots that they are grouped: ties, signed zeros, extreme logits, and NaNs of
    one token, of all of a token's logits and unselected ones.  The choices are those
    of the slots' launches, and a NaN weight makes its own token NaN only."""
    d, inter, group, m = 2048, 2048, 64, 24
    n = lambda rows, cols, bits, s: wq.pack(torch.randn((rows, cols), device="cuda",
                                                        generator=torch.Generator("cuda").manual_seed(s)) * 0.02, group, bits)
    layer = wq.MoELayer(wq.MLPLayer(n(E * inter, d, 2, 1), n(E * inter, d, 2, 2), n(E * d, inter, 4, 3)), E, k)
    x = synth.activations((m, d), 8).cuda()
    lg = np.random.default_rng(E).integers(-3, 2, (m, E)).astype(np.float32)  # many ties
    lg[:, ::3] *= -0.0
    lg[0, E // 2], lg[0, -1], lg[0, 0] = 3e38, 1e-40, -3e38
    nan = np.uint32(0x7FC00000).view(np.float32)
    lg[5, 2], lg[9, :], lg[11, 1] = nan, nan, -nan
    t = torch.from_numpy(lg).cuda()
    y, idx, wt, _, _ = wq.moe_forward(x, t, layer, with_slots=True)
    for i in range(m):
        _, i1, w1, _, _ = wq.moe_forward(x[i:i + 1], t[i:i + 1].clone(), layer, with_slots=True)
        assert torch.equal(idx[i], i1[0]) and torch.equal(wt[i].isnan(), w1[0].isnan()), i
        e = idx[i].tolist()
        assert len(set(e)) == k and min(e) >= 0 and max(e) < E, i
    bad = torch.zeros(m, dtype=torch.bool, device="cuda")
    bad[[5, 9]] = True
    assert torch.equal(y.isnan().all(1), bad) and torch.equal(y.isnan().any(1), bad)
    assert wq.device_status() == 0
