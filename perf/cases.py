"""What is timed: the calls that a program serving personalised diffusion checkpoints makes of this library.

One UNet denoising step runs ``taq_layer_forward`` on every cross-attention layer, a server runs
``taq_layer_forward_batched`` on a batch of requests that carry their own checkpoints, each prompt costs one
``taq_kv_project`` per layer, each checkpoint one ``taq_pack_weights`` per matrix, and ``taq_cross_attention`` serves
callers that project elsewhere.  Shapes are those of the benchmark's five configurations (SD-1.5 and SDXL cross-attention
layers) and of other image sizes, batches and bit-widths of the same layers.  As in the benchmark, hidden states are
N(0, 1) with one channel in a hundred scaled by 20, text contexts N(0, 1) with trigger rows scaled by 3, and weights
N(0, 1 / fan-in).
"""
import math

import torch

from paper_2603_22943_b200 import binding as tb

#: (channels, heads, width of the text context) of the SD-1.5 and SDXL cross-attention layers
SD15 = ((320, 8, 768), (640, 8, 768), (1280, 8, 768))
SDXL = ((640, 10, 2048), (1280, 20, 2048))


def _layer(kind, **kw):
    case = dict(kind=kind, net="layer", batch=2, n_query=4096, channels=320, heads=8, n_ctx=77, ctx_dim=768, w_bits=4, w_group=128, q_bits=8, kv_bits=8,
                p_bits=8, a_bits=16, triggers=2)
    case.update(kw)
    return case


def _unet(kind, **kw):
    case = dict(kind=kind, net="sd15", batch=2, height=64, width=64, n_ctx=77, w_bits=4, w_group=128, q_bits=8, kv_bits=8, p_bits=8, a_bits=16, triggers=2)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest layer of a UNet, one image, 8-bit weights: launches and latency are all there is
        dict(_layer("denoise", batch=1, n_query=64, channels=1280, w_bits=8, w_group=0, triggers=1), name="layer_8x8_w8"),
        # the highest-resolution SD-1.5 layer for one image with classifier-free guidance: the headline configuration
        dict(_layer("denoise"), name="layer_64x64_w4"),
        # the two SDXL layers, heads of 64 channels
        dict(_layer("denoise", channels=640, heads=10, ctx_dim=2048, triggers=3), name="layer_sdxl_64x64"),
        dict(_layer("denoise", n_query=1024, channels=1280, heads=20, ctx_dim=2048, triggers=3), name="layer_sdxl_32x32"),
        # a portrait image (latent 104 x 72, so 52 x 36 tokens here), three prompts at once, the 8/4-bit rows of the paper's tables
        dict(_layer("denoise", batch=3, n_query=1872, channels=640, kv_bits=4, p_bits=4), name="layer_portrait_4bit"),
        # the integer reading of the bit-widths: int8 activations into every projection, 8-bit weights
        dict(_layer("denoise", n_query=1024, channels=640, w_bits=8, w_group=0, a_bits=8), name="layer_32x32_w8a8"),
        # all sixteen cross-attention layers of one SD-1.5 denoising step, 512 x 512 with guidance: what an image costs fifty times
        dict(_unet("denoise"), name="unet_step"),
        # serving, the largest call: 64 requests of as many checkpoints on the highest-resolution layer
        dict(_layer("serve", batch=64, triggers=3), name="serve_64_layer"),
        # serving, ordinary: 8 requests of as many checkpoints through all sixteen layers
        dict(_unet("serve", batch=8, triggers=3), name="serve_8_step"),
        # a new prompt (with the empty one): keys and values of all sixteen layers
        dict(_unet("project"), name="project_unet"),
        # the attention core alone, a batch of low-resolution tiles whose projections were done elsewhere
        dict(_layer("attention", batch=64, n_query=256, channels=1280), name="attention_16x16_b64"),
        # loading a checkpoint: the four matrices of a 1280-channel layer
        dict(kind="pack", channels=1280, ctx_dim=768, w_bits=4, w_group=128, name="pack_layer"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("denoise", "denoise", "denoise", "denoise", "serve", "serve", "project", "project", "attention", "pack"))
    w_bits = rng.choice((4, 4, 8))
    w_group = rng.choice((128, 128, 128, 0)) if w_bits == 4 else 0
    if kind == "pack":
        return dict(kind=kind, channels=8 * _log_int(rng, 40, 320), ctx_dim=8 * _log_int(rng, 40, 320), w_bits=w_bits, w_group=w_group)
    bits = dict(w_bits=w_bits, w_group=w_group, q_bits=rng.choice((8, 8, 8, 0)), kv_bits=rng.choice((8, 8, 4)), p_bits=rng.choice((8, 8, 4)), triggers=rng.randint(1, 3))
    if kind in ("denoise", "serve", "project") and rng.random() < 0.25:            # all layers of a UNet at some image size
        height, width = 8 * rng.randint(4, 12), 8 * rng.randint(4, 12)
        most = max(1, (8 if kind != "denoise" else 4) * 4096 // (height * width))
        return _unet(kind, height=height, width=width, batch=_log_int(rng, 1, min(8, most)), **bits)
    channels, heads, ctx_dim = rng.choice(SD15 + SD15 + SDXL)
    if kind == "denoise":
        batch = _log_int(rng, 1, 8)
        n_query = _log_int(rng, 16, max(16, 2 * 4096 * 1280 // (batch * channels)))
        bits["a_bits"] = rng.choice((16, 16, 8))
    elif kind == "serve":
        batch = _log_int(rng, 1, 64)
        n_query = _log_int(rng, 16, max(16, min(4096, 64 * 4096 * 320 * 320 // (batch * channels * channels))))
    elif kind == "project":
        batch, n_query = _log_int(rng, 1, 64), 64
        bits["a_bits"] = rng.choice((16, 16, 8))
    else:
        batch = _log_int(rng, 1, 64)
        n_query = _log_int(rng, 16, max(16, min(4096, 64 * 256 * 1280 // (batch * channels))))
    n_ctx = 77 if rng.random() < 0.75 else rng.randint(20, 77)
    return _layer(kind, batch=batch, n_query=min(n_query, 16384), channels=channels, heads=heads, n_ctx=n_ctx, ctx_dim=ctx_dim, **bits)


def _shapes(case):
    """(query tokens, channels, heads, context width) of the layers of one pass."""
    if case["net"] == "layer":
        return [(case["n_query"], case["channels"], case["heads"], case["ctx_dim"])]
    n = case["height"] * case["width"]
    return [(n, 320, 8, 768)] * 5 + [(n // 4, 640, 8, 768)] * 5 + [(n // 16, 1280, 8, 768)] * 5 + [(n // 64, 1280, 8, 768)]


def _desc(case, shape, batch):
    n, c, h, dc = shape
    return tb.layer_desc(batch, n, c, h, case["n_ctx"], dc, case["w_bits"], case["w_group"], q_bits=case["q_bits"], kv_bits=case["kv_bits"], p_bits=case["p_bits"],
                         max_trigger=case["triggers"])


class _Inputs:
    """Random inputs on the GPU from one seed."""

    def __init__(self, case, seed):
        self.case = case
        self.gen = torch.Generator("cuda").manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.gen, device="cuda")

    def hidden(self, batch, n, c):
        scale = torch.ones(c, device="cuda")
        scale[torch.randperm(c, generator=self.gen, device="cuda")[:max(1, round(c / 100))]] = 20.0
        return (self.normal(batch, n, c) * scale).half()

    def mask(self, rows):
        """One contiguous span of 1 to `triggers` tokens per row, never at position 0."""
        t, most = self.case["n_ctx"], self.case["triggers"]
        span = torch.randint(1, most + 1, (rows, 1), generator=self.gen, device="cuda")
        start = 1 + torch.randint(0, t - most, (rows, 1), generator=self.gen, device="cuda")
        at = torch.arange(t, device="cuda")
        return ((at >= start) & (at < start + span)).to(torch.uint8)

    def context(self, mask, dc):
        return (self.normal(*mask.shape, dc) * (1.0 + 2.0 * mask[..., None])).half()

    def packed(self, n_out, k_in, bias=False):
        wd = tb.weight_desc(n_out, k_in, self.case["w_bits"], self.case["w_group"])
        return tb.taq_pack_weights(wd, self.normal(n_out, k_in) / math.sqrt(k_in), 0.1 * self.normal(n_out) if bias else None)


def _kv_views(desc, kv, n):
    """The parts of n K~/V~ blocks: int8 codes, scales, fp16 operand images, logit factors."""
    L, blocks = tb.taq_kv_layout_of(desc), kv.view(n, -1)
    images = blocks[:, L.off_operands:].view(n, desc.heads, L.operand_head_bytes)
    return [blocks[:, :L.off_k_scales].view(torch.int8), blocks[:, L.off_k_scales:L.off_k_trigger].view(torch.float32),
            images[..., :-1024].view(torch.float16), images[..., -1024:-1024 + 320].view(torch.float32)]


def prepare(case, seed):
    inp = _Inputs(case, seed)
    kind = case["kind"]
    if kind == "pack":
        c, dc = case["channels"], case["ctx_dim"]
        todo = []
        for k_in, bias in ((c, False), (dc, False), (dc, False), (c, True)):
            wd = tb.weight_desc(c, k_in, case["w_bits"], case["w_group"])
            w = inp.normal(c, k_in) / math.sqrt(k_in)
            b = 0.1 * inp.normal(c) if bias else None
            todo.append((wd, w, b, torch.zeros(tb.taq_packed_weight_bytes(wd), dtype=torch.uint8, device="cuda")))
        return kind, todo, [t[3] for t in todo]
    batch, a8 = case["batch"], case["a_bits"] == 8
    mask = inp.mask(batch)
    todo, outs, workspace_bytes, keep = [], [], 128, []
    for shape in _shapes(case):
        n, c, h, dc = shape
        if kind == "serve":
            # every request: its own checkpoint (four packed matrices), prompt and trigger span
            desc = _desc(case, shape, 1)
            ctx = inp.context(mask, dc)
            kv = torch.zeros((batch, tb.taq_kv_bytes(desc)), dtype=torch.uint8, device="cuda")
            admit = [(inp.packed(c, dc), inp.packed(c, dc), kv[r], mask[r]) for r in range(batch)]
            tb.taq_kv_project_batched(desc, tb.make_request_table(admit, "cuda"), batch, ctx)
            use = [(inp.packed(c, c), inp.packed(c, c, bias=True), kv[r], mask[r]) for r in range(batch)]
            y = torch.empty((batch, n, c), dtype=torch.float16, device="cuda")
            todo.append((desc, tb.make_request_table(use, "cuda"), inp.hidden(batch, n, c), y))
            keep.append((use, admit))
            outs.append(y)
            workspace_bytes = max(workspace_bytes, tb.taq_workspace_bytes(desc, batch))
            continue
        desc = _desc(case, shape, batch)
        ctx, wk, wv = inp.context(mask, dc), inp.packed(c, dc), inp.packed(c, dc)
        kv = torch.zeros(tb.taq_kv_bytes(desc), dtype=torch.uint8, device="cuda")
        if kind == "project":
            todo.append((desc, ctx, wk, wv, kv))
            outs += _kv_views(desc, kv, batch)
            if a8:
                workspace_bytes = max(workspace_bytes, tb.lib().taq_kv_project_a8_workspace_bytes(desc))
            continue
        (tb.taq_kv_project_a8 if a8 else tb.taq_kv_project)(desc, ctx, wk, wv, mask, kv)
        x, wq = inp.hidden(batch, n, c), inp.packed(c, c)
        y = torch.empty((batch, n, c), dtype=torch.float16, device="cuda")
        outs.append(y)
        if kind == "attention":
            wd = tb.weight_desc(c, c, case["w_bits"], case["w_group"])
            if case["q_bits"] == 8:
                q, q_scales = tb.taq_quantized_linear(wd, x, wq, tb.TAQ_OUT_INT8_HEAD_ROWS, heads=h)
            else:
                q, q_scales = tb.taq_quantized_linear(wd, x, wq), None
            todo.append((desc, q, q_scales, kv, y))
        else:
            todo.append((desc, x, wq, inp.packed(c, c, bias=True), kv, y))
            workspace_bytes = max(workspace_bytes, tb.taq_workspace_bytes_a8(desc) if a8 else tb.taq_workspace_bytes(desc))
    if a8:
        kind += "_a8"
    return kind, todo, outs, mask, torch.empty(workspace_bytes, dtype=torch.uint8, device="cuda"), keep


def run(state):
    kind, todo, outs = state[:3]
    if kind == "pack":
        for wd, w, bias, blob in todo:
            tb.taq_pack_weights(wd, w, bias, blob)
        return outs
    mask, workspace = state[3:5]
    if kind == "denoise":
        for desc, x, wq, wout, kv, y in todo:
            tb.taq_layer_forward(desc, x, wq, wout, kv, mask, y, workspace)
    elif kind == "denoise_a8":
        for desc, x, wq, wout, kv, y in todo:
            tb.taq_layer_forward_a8(desc, x, wq, wout, kv, mask, y, workspace)
    elif kind == "serve":
        for desc, table, x, y in todo:
            tb.taq_layer_forward_batched(desc, table, x.shape[0], x, y, workspace)
    elif kind == "project":
        for desc, ctx, wk, wv, kv in todo:
            tb.taq_kv_project(desc, ctx, wk, wv, mask, kv)
    elif kind == "project_a8":
        for desc, ctx, wk, wv, kv in todo:
            tb.taq_kv_project_a8(desc, ctx, wk, wv, mask, kv, workspace)
    else:
        for desc, q, q_scales, kv, y in todo:
            tb.taq_cross_attention(desc, q, q_scales, kv, mask, y)
    return outs


def work(case):
    per_weight = lambda n_out, k_in: n_out * k_in * case["w_bits"] / 8 + 4 * n_out * (1 if not case["w_group"] else math.ceil(k_in / case["w_group"]))
    if case["kind"] == "pack":
        c, dc = case["channels"], case["ctx_dim"]
        return {"bytes": sum(4 * c * k + per_weight(c, k) for k in (c, c, dc, dc)) + 8 * c, "flops": 0}
    kind, b, t, nbytes, flops = case["kind"], case["batch"], case["n_ctx"], 0, 0
    for n, c, h, dc in _shapes(case):
        kv = b * (2 * t * c + 2 * 4 * t * h)                       # K~ and V~: one byte per code, one scale per (token, head)
        if kind == "project":
            nbytes += b * t * (2 * dc + 1) + 2 * per_weight(c, dc) + kv
            flops += 2 * 2 * b * t * c * dc
        elif kind == "attention":
            nbytes += b * n * (c + 4 * h if case["q_bits"] == 8 else 2 * c) + b * n * 2 * c + kv
            flops += 4 * b * n * t * c
        else:
            nbytes += b * n * 4 * c + (b if kind == "serve" else 1) * (2 * per_weight(c, c) + 4 * c) + kv
            flops += b * n * (4 * c * c + 4 * t * c)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Packed blobs are the same bytes.  The rest is fp16 (or int8 codes) behind fp32 sums and round-to-nearest quantizers:
    sums in another order put a code in a hundred thousand on the other side of a tie.  With 8-bit codes that leaves the
    outputs within 1e-3 in the 2-norm, the contract of the repository's tests; a step of a 4-bit code is 18 times as wide."""
    if case["kind"] == "pack":
        return "exact"
    if case["kv_bits"] == 4 or case["p_bits"] == 4:
        return {"rel": 3e-3, "max": 0.6, "differ": 2e-3}
    return {"rel": 1e-3, "max": 0.15, "differ": 2e-3}
