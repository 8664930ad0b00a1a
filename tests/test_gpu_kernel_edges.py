"""The kernels' branches at the sizes where they can go wrong: every tile width of the dequant-GEMM with one tile per CTA, several
tiles per CTA and a cluster per tile, first and last rows of a tile, heads over two tiles; the merged K/V projection at its
smallest and largest contexts; the packing kernel's group lengths."""
from dataclasses import replace

import pytest
import torch

import test_gpu_layer as layer
import test_gpu_quantizers as quantizers
import test_gpu_int8_activations as int8_activations
from paper_2603_22943_b200 import binding as tb
from paper_2603_22943_b200 import synth
import taq_testlib as tl
from oracle import taq_oracle as orc

pytestmark = pytest.mark.gpu


def layout(rows, n_out, k_in, bits, group, kind, heads=1, int8_activations=False):
    """Tile width of a launch, "p" on pairs of CTAs, "x2" or "x4" where so many CTAs share a tile, "+" where a CTA walks several tiles (148 SMs)."""
    wd = tb.weight_desc(n_out, k_in, bits, group)
    plan = tb.taq_linear_plan(wd, rows, kind, heads=heads, int8_activations=int8_activations)
    if not int8_activations and kind != tb.TAQ_OUT_F32 and tb.taq_linear_pair_plan(wd, rows, kind, heads)["bn"]:
        return f"{plan['bn']}p"
    ctas = (rows + 127) // 128 * (n_out // plan["bn"]) * plan["split"] if plan["bn"] else 0
    return f"{plan['bn']}" + (f"x{plan['split']}" if plan["split"] > 1 else "") + ("+" if ctas > 148 else "")


# (the layouts of the fp16, the fp32 and the per-head int8 output: a change of the rule that chooses them says here which of them is no
# longer run.  Scale groups of 64 do not go to pairs, nor do some shapes with 8-bit weights; see also test_requests_of_few_rows.)
@pytest.mark.parametrize("rows,n_out,k_in,bits,group,heads,half,single,per_head", [
    (1, 640, 640, 4, 128, 8, "64", "64", "80"),              # one row
    (129, 640, 640, 8, 0, 10, "64", "64", "64"),             # a second row tile of one row
    (2047, 640, 640, 4, 128, 10, "80", "80", "128p"),
    (2047, 640, 640, 4, 64, 10, "80", "80", "128"),
    (5616, 640, 640, 4, 128, 10, "128p", "64+", "128p"),
    (5616, 640, 640, 4, 64, 10, "64+", "64+", "128+"),
    (5505, 640, 640, 8, 0, 8, "128p", "64+", "160p"),        # a last row tile of one row
    (5505, 640, 640, 4, 64, 8, "64+", "64+", "80+"),
    (4225, 640, 640, 4, 128, 8, "160p", "160", "160p"),
    (4225, 640, 640, 4, 64, 8, "160", "160", "160"),
    (64, 1280, 1280, 4, 128, 20, "64x2", "64x2", "64x2"),    # shares of whole groups
    (300, 1280, 1280, 8, 0, 20, "64x2", "64x2", "64x2"),     # ... and of k-blocks
    (129, 1280, 1280, 4, 0, 8, "64x2", "64x2", "80x2"),      # heads over two tiles
    (129, 1280, 1280, 8, 0, 8, "64x2", "64x2", "160p"),
    (1100, 1280, 1280, 4, 128, 8, "80", "80", "160x2"),
    (1100, 1280, 1280, 8, 0, 8, "80", "80", "160p"),
    (1, 3840, 2048, 8, 0, 24, "64x2", "64x2", "160x2"),
    (1, 1600, 1600, 8, 0, 10, "64x2", "64x2", "160x4"),
    (97, 320, 192, 4, 128, 8, "64", "64", "80"),             # an odd number of k-blocks, a short last group
    (200, 320, 64, 8, 0, 8, "80", "80", "80"),               # one k-block
    (64, 1280, 1280, 8, 0, 8, "64x2", "64x2", "160p"),
    (3000, 1280, 320, 4, 128, 20, "128p", "128+", "128p"),
    (3000, 1280, 320, 4, 64, 20, "128+", "128+", "128+"),
    (4300, 1280, 1280, 4, 128, 8, "160p", "160+", "160p"),
    (4300, 1280, 1280, 4, 64, 8, "160+", "160+", "160+"),
    (20000, 64, 64, 8, 0, 1, "64+", "64+", "64+"),
    (20000, 80, 64, 8, 0, 2, "80+", "80+", "80+"),
    (1100, 2048, 64, 8, 0, 32, "128", "128", "128"),
    (7000, 2048, 64, 8, 0, 32, "128+", "128+", "128+"),
    (1100, 2400, 64, 8, 0, 60, "160", "160", "160"),
    (1, 640, 768, 4, 128, 8, "64x2", "64x2", "80x2"),
])
def test_linear_tiles(rows, n_out, k_in, bits, group, heads, half, single, per_head):
    assert layout(rows, n_out, k_in, bits, group, tb.TAQ_OUT_F16) == half
    assert layout(rows, n_out, k_in, bits, group, tb.TAQ_OUT_F32) == single
    assert layout(rows, n_out, k_in, bits, group, tb.TAQ_OUT_INT8_HEAD_ROWS, heads) == per_head
    layer.test_quantized_linear(rows, n_out, k_in, bits, group, heads)


# (tile widths of the launches on pairs of CTAs, 0 where they do not run there)
@pytest.mark.parametrize("rows,n_out,k_in,bits,group,heads,dense,per_head", [
    (5633, 640, 640, 4, 128, 8, 128, 160),             # the last tile: one row of the first CTA, none of the second
    (5505, 640, 640, 8, 0, 10, 128, 128),              # ... one row of the second CTA; accumulators of two, two and one pairs of k-blocks
    (9999, 640, 192, 4, 128, 16, 128, 160),            # an odd number of k-blocks, a short last group, heads of 40
    (20000, 640, 64, 8, 0, 16, 128, 160),              # one k-block
    (9473, 320, 320, 4, 128, 8, 0, 160),
    (12289, 640, 512, 4, 256, 4, 160, 160),            # groups of two pairs of k-blocks, heads of 160
    (3000, 1280, 320, 4, 128, 20, 128, 128),
    (2049, 1280, 1280, 4, 0, 8, 160, 160),             # one group of 4-bit codes
    (1, 1280, 1280, 8, 0, 8, 0, 160),
])
def test_linear_tiles_on_pairs(rows, n_out, k_in, bits, group, heads, dense, per_head):
    wd = tb.weight_desc(n_out, k_in, bits, group)
    assert tb.taq_linear_pair_plan(wd, rows, tb.TAQ_OUT_F16)["bn"] == dense
    assert tb.taq_linear_pair_plan(wd, rows, tb.TAQ_OUT_INT8_HEAD_ROWS, heads)["bn"] == per_head
    layer.test_quantized_linear(rows, n_out, k_in, bits, group, heads)


def test_pairs_write_their_rows_only():
    """Requests side by side, each with weights of its own: the last tile of one ends inside the rows of the next."""
    assert tb.taq_linear_pair_plan(tb.weight_desc(640, 640, 4, 128), 520, tb.TAQ_OUT_F16, n_requests=8)["bn"] != 0
    shape, desc, ckpts, route, reqs_data, packed, y, kv_blocks = layer._serving_case(n_ckpt=3, n_req=8, n_query=520, C_=640, Dc=768)
    for r, c in enumerate(route):
        layer._check_request(shape, desc, ckpts[int(c)], reqs_data[r], packed[int(c)], kv_blocks[r], y[r: r + 1])
    rows, heads = 5633, 8
    n = rows * 640
    wd, blob = tb.weight_desc(640, 640, 4, 128), packed[0]["Wq"]
    x = torch.randn(rows, 640, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).half()
    codes, group_scales = tb.taq_unpack_weights(wd, blob)
    want = x.double() @ (codes.double() * group_scales.view(640, -1).repeat_interleave(128, 1).double()).T
    want_scales = want.view(rows, heads, -1).abs().amax(-1) / 127

    def guarded(count, dtype):
        buf = torch.full((count + 4096,), -7, dtype=dtype, device="cuda")
        return buf, buf[2048: 2048 + count]

    for kind, dtype in ((tb.TAQ_OUT_F16, torch.float16), (tb.TAQ_OUT_INT8_HEAD_ROWS, torch.int8)):
        per_head = kind == tb.TAQ_OUT_INT8_HEAD_ROWS
        (buf, out), (scale_buf, scales) = guarded(n, dtype), guarded(rows * heads, torch.float32)
        tb.taq_quantized_linear(wd, x, blob, kind, heads=heads, y=out, scales=scales if per_head else None)
        tb.taq_poll_device_status()
        for b in (buf, scale_buf):
            assert bool((b[:2048] == -7).all()) and bool((b[-2048:] == -7).all())
        if per_head:
            assert bool(((scales.view(rows, heads).double() - want_scales).abs() <= 2e-5 * want_scales).all())
            layer._code_agreement(out.view(rows, heads, -1).cpu().numpy(), (want.view(rows, heads, -1) / want_scales[..., None]).round().cpu().numpy(), "codes")
        else:                                        # half a unit in the last place of an fp16 value, and fp32 sums of 640 products
            assert bool(((out.view(rows, 640).double() - want).abs() <= 2.0 ** -11 * want.abs() + 2e-5 * want.abs().max()).all())


# (none of these goes to pairs.  fp16 rows on 160-wide tiles, the first two one per CTA, the others several; per-head rows on 128, 128, 80, 128 and
# 160 columns, several per CTA)
@pytest.mark.parametrize("channels,heads,n_req,w_bits", [(1280, 20, 18, 4), (1280, 20, 18, 8), (640, 8, 64, 8), (640, 10, 64, 4), (1280, 16, 33, 8)])
def test_requests_of_few_rows(channels, heads, n_req, w_bits):
    """Batched layers whose requests fill a quarter of a row tile: tiles of several requests in one CTA's walk.  Sums of to_q are of whole numbers, so
    that the query codes are those of the single projection, whatever its layout, and the oracle starts from them."""
    wd = tb.weight_desc(channels, channels, w_bits, 128 if w_bits == 4 else 0)
    assert tb.taq_linear_pair_plan(wd, 34, tb.TAQ_OUT_F16, n_requests=n_req)["bn"] == 0
    assert tb.taq_linear_pair_plan(wd, 34, tb.TAQ_OUT_INT8_HEAD_ROWS, heads, n_requests=n_req)["bn"] == 0
    shape, desc, ckpts, route, reqs_data, packed, y, kv_blocks = layer._serving_case(n_ckpt=3, n_req=n_req, n_query=34, C_=channels, Dc=768, heads=heads, w_bits=w_bits, whole=True)
    cfg = tl.oracle_cfg(shape)
    for r, c in enumerate(route):
        ck, rd = ckpts[int(c)], reqs_data[r]
        g = tl.gpu_decisions(shape, {**ck.weights, **rd}, {"desc": desc, "packed": packed[int(c)], "kv": kv_blocks[r]})
        O = orc.taq_attention(g["Q_tilde"], g["K_tilde"], g["V_tilde"], rd["mask"], cfg)
        tl.assert_layer_close(y[r: r + 1], orc.taq_out(O, ck.weights["Wout"], ck.weights["bout"], cfg), f"request {r}")


@pytest.mark.parametrize("rows,k_in,n_out,bits,group,dense", [
    (1, 320, 320, 4, 128, "64"), (257, 1280, 1280, 4, 128, "64"), (4225, 640, 640, 4, 128, "160"), (300, 656, 640, 8, 0, "64"),
    (1, 1280, 1280, 4, 128, "64x2"), (5505, 64, 320, 4, 128, "64+"), (3000, 320, 1280, 4, 128, "128+"),
])
def test_integer_linear_tiles(rows, k_in, n_out, bits, group, dense):
    assert layout(rows, n_out, k_in, bits, group, tb.TAQ_OUT_F32, int8_activations=True) == dense
    int8_activations.test_integer_gemm_equals_the_integer_definition(rows, k_in, n_out, bits, group)


@pytest.mark.parametrize("channels,heads,ctx_dim,n_ctx,batch,w_bits", [
    (320, 8, 768, 9, 1, 4), (320, 8, 768, 80, 3, 8), (640, 8, 768, 77, 2, 4), (640, 10, 2048, 20, 1, 4),
    (1280, 20, 2048, 77, 1, 8), (1280, 8, 768, 64, 2, 8), (640, 10, 2048, 77, 9, 4),
    (1280, 8, 768, 9, 1, 4), (1280, 8, 768, 80, 4, 4), (1280, 8, 768, 77, 5, 4),      # heads on two tiles; more of them than one wave
])
def test_kv_projection(channels, heads, ctx_dim, n_ctx, batch, w_bits):
    shape = replace(synth.config1(), batch=batch, channels=channels, heads=heads, ctx_dim=ctx_dim, n_ctx=n_ctx, w_bits=w_bits, w_group=128 if w_bits == 4 else 0,
                    trigger=(1, n_ctx - 1), n_query=130, name=f"edge_{channels}_{heads}_{ctx_dim}_{n_ctx}")
    layer.test_kv_project(shape)
    data = synth.make_layer(shape)
    y, parts = tl.gpu_layer(shape, data, return_parts=True)          # reads the operand images that the projection left
    tl.check_layer(shape, data, y, parts)


@pytest.mark.parametrize("n_out,k_in,bits,group", [
    (40, 512, 4, 256), (24, 1024, 4, 512), (16, 2560, 8, 0), (9, 136, 8, 0), (33, 352, 4, 32), (7, 1000, 4, 128), (5, 2560, 4, 0),
    (1200, 4160, 4, 32), (19000, 512, 4, 256), (9600, 520, 8, 0),        # more groups than 4736 blocks take at once, for 8, 32 and 128 threads per group
])
def test_pack_group_lengths(n_out, k_in, bits, group):
    quantizers.test_pack_weights_codes_bit_exact(n_out, k_in, bits, group)


@pytest.mark.parametrize("n_query", [1, 31, 33, 127, 129, 160, 257])
def test_one_kernel_layer_writes_its_rows_only(n_query):
    """C = 320: the rows of Y leave in quarters of a tile; rows of two sequences side by side, nothing beyond the last."""
    shape = synth.shrink(synth.config2(), n_query)
    data = synth.make_layer(shape)
    _, parts = tl.gpu_layer(shape, data, return_parts=True)
    n = shape.rows * shape.channels
    buf = torch.full((n + 2048,), -7.0, dtype=torch.float16, device="cuda")
    P = parts["packed"]
    tb.taq_layer_forward(parts["desc"], tl.dev(data["X"]), P["Wq"], P["Wout"], parts["kv"], parts["mask"], buf[1024: 1024 + n])
    tb.taq_poll_device_status()
    assert bool((buf[:1024] == -7.0).all()) and bool((buf[1024 + n:] == -7.0).all())
    y = buf[1024: 1024 + n].reshape(shape.batch, n_query, shape.channels).cpu().numpy()
    tl.check_layer(shape, data, y, parts)


def test_kv_projections_of_one_shape_and_two_trigger_capacities():
    """The capacity moves everything behind the trigger rows in a K~/V~ block; nothing of one call's layout is kept for the other."""
    shape = synth.shrink(synth.config2(), 8)
    data = synth.make_layer(shape)
    P = tl.pack_layer_weights(shape, data)
    blocks = {}
    for capacity in (2, 5, 2):
        desc = tl.gpu_desc(shape, max_trigger=capacity)
        kv = torch.zeros(tb.taq_kv_bytes(desc), dtype=torch.uint8, device="cuda")
        tb.taq_kv_project(desc, tl.dev(data["ctx"]), P["Wk"], P["Wv"], tl.dev(data["mask"]), kv)
        blocks[capacity] = tl.parse_kv_block(desc, kv)
        L = tb.taq_kv_layout_of(desc)
        blocks[capacity]["images"] = kv.view(shape.batch, -1)[:, L.off_operands:].cpu().numpy()
    tb.taq_poll_device_status()
    for name in ("K_codes", "V_codes", "K_scales", "V_scales", "slot", "images"):
        assert (blocks[2][name] == blocks[5][name]).all(), name
    for name in ("K_trigger", "V_trigger"):
        assert (blocks[2][name] == blocks[5][name][:, :2]).all(), name


# (280 channels: rows of Q~ start 8 bytes apart from 16-byte boundaries, too)
@pytest.mark.parametrize("channels,heads", [(640, 10), (160, 4), (280, 7)])
@pytest.mark.parametrize("q_bits", [8, 0])
def test_attention_in_pieces_of_any_alignment(channels, heads, q_bits):
    """Heads of 64 and 40 channels are read and written in pieces as wide as the address allows: right, and the same bits 16 bytes further."""
    shape = replace(synth.config1(), batch=2, n_query=130, channels=channels, heads=heads, name=f"pieces_{channels}_{heads}")
    layer.test_cross_attention_isolated(shape, 130, q_bits)
    shape = replace(shape, q_bits=q_bits)
    data = synth.make_layer(shape)
    desc = tl.gpu_desc(shape)
    P = tl.pack_layer_weights(shape, data)
    mask = tl.dev(data["mask"])
    kv = tb.taq_kv_project(desc, tl.dev(data["ctx"]), P["Wk"], P["Wv"], mask)
    n = shape.rows * channels
    gen = torch.Generator("cuda").manual_seed(1)
    q = torch.randint(-127, 128, (n,), device="cuda", generator=gen).to(torch.int8) if q_bits else torch.randn(n, device="cuda", generator=gen).half()
    scales = torch.rand(shape.rows * heads, device="cuda", generator=gen) / 30 if q_bits else None
    outs = []
    for shift in (0, 16):                                            # bytes
        qq = torch.zeros(n + 64, dtype=q.dtype, device="cuda")[shift // q.element_size():][:n].copy_(q)
        o = torch.full((n + 64,), -7.0, dtype=torch.float16, device="cuda")
        tb.taq_cross_attention(desc, qq, scales, kv, mask, o[shift // 2: shift // 2 + n])
        tb.taq_poll_device_status()
        assert bool((o[: shift // 2] == -7.0).all()) and bool((o[shift // 2 + n:] == -7.0).all())
        outs.append(o[shift // 2: shift // 2 + n].clone())
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("channels,heads", [(640, 10), (160, 4), (320, 8), (640, 8), (1280, 8)])
@pytest.mark.parametrize("n_ctx", [1, 40, 64, 65, 80])
def test_attention_of_zero_queries(channels, heads, n_ctx):
    """A row of zero codes has scale 0: every token weighs the same, and padding keys nothing, as with any other scale."""
    shape = replace(synth.config1(), n_query=130, channels=channels, heads=heads, n_ctx=n_ctx, trigger=(0,), name=f"zero_{channels}_{heads}_{n_ctx}")
    data = synth.make_layer(shape)
    desc = tl.gpu_desc(shape)
    P = tl.pack_layer_weights(shape, data)
    mask = tl.dev(data["mask"])
    kv = tb.taq_kv_project(desc, tl.dev(data["ctx"]), P["Wk"], P["Wv"], mask)
    q = torch.zeros(shape.rows, channels, dtype=torch.int8, device="cuda")
    q[::2] = torch.randint(-127, 128, q[::2].shape, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).to(torch.int8)
    scales = torch.full((shape.rows, heads), 0.02, device="cuda")
    want = tb.taq_cross_attention(desc, q, scales, kv, mask)
    scales[1::2] = 0.0
    got = tb.taq_cross_attention(desc, q, scales, kv, mask)
    tb.taq_poll_device_status()
    assert bool(torch.isfinite(got).all()) and torch.equal(got, want)
    p = tl.parse_kv_block(desc, kv)
    v = p["V_codes"][0].astype("f8") * p["V_scales"][0][..., None]                   # [H, T, d] of the ordinary tokens
    v[:, 0] = p["V_trigger"][0][0]
    prob = torch.full((n_ctx,), float(round(255.0 / n_ctx)), dtype=torch.float64)    # the nearest code, and fp16 for the trigger column
    prob[0] = torch.tensor(255.0 / n_ctx).half().double()
    mean = (v * prob.numpy()[None, :, None] / 255.0).sum(1).reshape(-1)
    # V~ and O are fp16 values: half a unit in the last place each, of a sum of n_ctx products
    assert abs(got.view(-1, channels)[1].double().cpu().numpy() - mean).max() <= 2.0 ** -11 * (abs(v).max() + abs(mean).max())


@pytest.mark.parametrize("channels,heads", [(640, 10), (160, 4), (640, 8), (1280, 8)])
@pytest.mark.parametrize("n_ctx", [1, 9, 40, 64, 77])
def test_attention_of_any_query_scale(channels, heads, n_ctx):
    """Padding keys weigh nothing beside the smallest and the largest scales, too, and rows of a tile do not depend on their neighbours' scales."""
    shape = replace(synth.config1(), n_query=130, channels=channels, heads=heads, n_ctx=n_ctx, trigger=(0,), name=f"scale_{channels}_{heads}_{n_ctx}")
    data = synth.make_layer(shape)
    desc = tl.gpu_desc(shape)
    P = tl.pack_layer_weights(shape, data)
    mask = tl.dev(data["mask"])
    kv = tb.taq_kv_project(desc, tl.dev(data["ctx"]), P["Wk"], P["Wv"], mask)
    q = torch.randint(-127, 128, (shape.rows, channels), device="cuda", generator=torch.Generator("cuda").manual_seed(1)).to(torch.int8)
    d = channels // heads

    def attention(scale, codes=q):
        scales = torch.full((shape.rows, heads), 0.02, device="cuda")
        scales[1::2] = scale
        o = tb.taq_cross_attention(desc, codes, scales, kv, mask).view(-1, channels)
        tb.taq_poll_device_status()
        return o

    plain, flat = attention(0.02), attention(0.0)
    assert torch.equal(flat[::2], plain[::2])
    # logits of at most 127 * 127 * 160 units, each under 1: beside these scales all are 0
    for scale in (1e-45, 1e-38, 1e-30, 1e-24):
        assert torch.equal(attention(scale), flat), scale
    # the sign of scale and codes together does not matter (the maximum taken off the logits does, hence ties)
    tl.assert_same_up_to_code_ties(attention(-0.02, torch.where(torch.arange(shape.rows, device="cuda")[:, None] % 2 == 1, -q, q)), plain, "negative scales")
    # A scale at which the largest logit takes all of it, of single codes of 1: logits of about 1e9, whose last place (64) is nothing that the sums
    # of powers of two could not hold.
    p = tl.parse_kv_block(desc, kv)
    k, v = (p[n + "_codes"][0].astype("f8") * p[n + "_scales"][0][..., None] for n in "KV")      # [H, T, d]
    k[:, 0], v[:, 0] = p["K_trigger"][0][0], p["V_trigger"][0][0]
    k, v = torch.from_numpy(k), torch.from_numpy(v).half().double()                               # (V~ is an fp16 operand)
    single = q.view(-1, heads, d).clone()
    single[1::2] = torch.nn.functional.one_hot(torch.arange(shape.rows, device="cuda") % d, d)[1::2, None]
    logits = torch.einsum("rhd,htd->rht", single[1::2].cpu().double(), k)
    top = logits.topk(min(2, n_ctx), dim=-1).values
    clear = (top[..., 0] - top[..., -1] > 1e-5 * top[..., 0].abs() + 1e-5) | (n_ctx == 1)         # (1e9 / 8 of that: far more than 64 + 24)
    got = attention(1e9, single.view(-1, channels))
    assert torch.equal(got[::2], plain[::2])
    got = got[1::2].view(-1, heads, d).cpu().double()
    want = v[torch.arange(heads), logits.argmax(-1)]                                              # [rows, H, d]
    # the one probability is 255 of 255; O = V~ * 255 * (1 / 255) in fp32, rounded to fp16
    assert bool(clear.any()) and bool(((got - want).abs() <= 2.0 ** -11 * want.abs() + 1e-7)[clear].all())


@pytest.mark.parametrize("channels,n_ctx", [(320, 9), (320, 77), (640, 9), (640, 77)])
def test_layer_of_tiny_query_projections(channels, n_ctx):
    """A to_q of tiny weights leaves tiny scales, beside which every logit is 0: the same output as of a to_q of zeros."""
    shape = replace(synth.config2(), n_query=130, channels=channels, n_ctx=n_ctx, name=f"tiny_q_{channels}_{n_ctx}")
    data = synth.make_layer(shape)
    none = dict(data, Wq=0.0 * data["Wq"])
    want = tl.gpu_layer(shape, none)
    tl.assert_layer_close(want, tl.oracle_layer(shape, none)["Y"], "zero queries")
    for size in (1e-35, 1e-30, 1e-25):
        assert (tl.gpu_layer(shape, dict(data, Wq=(size * data["Wq"]).astype("f4"))) == want).all(), size


@pytest.mark.parametrize("ctx_dim,batch", [(1024, 1), (2048, 1), (2048, 4), (4096, 1)])
def test_kv_sums_of_wide_contexts_stay_short(ctx_dim, batch):
    """8-bit weights have one scale per row, so a share of the K loop is one sum in the tensor core, which loses bits with its length.  Heads of 160
    channels: root mean square error of K's scales 3.4e-7 from sums of 512 elements, 7.3e-7 of 1024, 1.8e-6 of 2048, 3.8e-6 of 4096."""
    channels, heads, n_ctx = 1280, 8, 77
    desc = tb.layer_desc(batch, 64, channels, heads, n_ctx, ctx_dim, 8, 0)
    wd = tb.weight_desc(channels, ctx_dim, 8, 0)
    gen = torch.Generator("cuda").manual_seed(1)
    wk = tb.taq_pack_weights(wd, torch.randn(channels, ctx_dim, device="cuda", generator=gen) / ctx_dim ** 0.5)
    ctx = torch.randn(batch, n_ctx, ctx_dim, device="cuda", generator=gen).half()
    kv = tb.taq_kv_project(desc, ctx, wk, wk, torch.zeros(batch, n_ctx, dtype=torch.uint8, device="cuda"))
    tb.taq_poll_device_status()
    codes, scales = tb.taq_unpack_weights(wd, wk)
    want = (ctx.double() @ (codes.double() * scales.view(-1, 1).double()).T).view(batch, n_ctx, heads, -1).transpose(1, 2).abs().amax(-1) / 127
    got = torch.from_numpy(tl.parse_kv_block(desc, kv)["K_scales"]).cuda().double()
    rms = ((got - want) / want).pow(2).mean().sqrt().item()
    assert rms <= {1024: 5e-7, 2048: 1.1e-6, 4096: 1.1e-6}[ctx_dim], rms       # (between the lengths that are meant and twice those)
