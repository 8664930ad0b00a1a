"""Layer passes enqueued one behind the other, as a denoising loop does: every kernel may start while its predecessor is still
running, so each one's reads of what the predecessor writes, and its writes over what the predecessor reads, are put to the test
only here.  The passes of a sequence have inputs of their own and take turns on workspaces of their own and on one that all
share; each pass must give, bit for bit, what it gives alone on an idle GPU."""
import pytest
import torch

from paper_2603_22943_b200 import binding as tb

pytestmark = pytest.mark.gpu

ROUNDS = 8


def _sections(desc, a_bits):
    """(name, offset, bytes per row) of a pass's workspace; every section starts on a multiple of 128 bytes."""
    rows, c, h = desc.batch * desc.n_query, desc.channels, desc.heads
    out, off = [], 0
    for name, per_row in ([("activation codes", c), ("activation scales", 4)] if a_bits == 8 else []) + [("Q~", c), ("Q~ scales", 4 * h), ("O", 2 * c)]:
        out.append((name, off, per_row))
        off += (rows * per_row + 127) // 128 * 128
    return out


def _where(desc, a_bits, got, want):
    """Which sections of two workspaces differ, in which rows and heads."""
    text, rows, h = [], desc.batch * desc.n_query, desc.heads
    for name, off, per_row in _sections(desc, a_bits):
        d = (got[off: off + rows * per_row] != want[off: off + rows * per_row]).view(rows, per_row)
        if bool(d.any()):
            r = d.any(1).nonzero().flatten().tolist()
            heads = d.view(rows, h, per_row // h).any(2).any(0).nonzero().flatten().tolist() if per_row % h == 0 else "-"
            text.append(f"{name}: {len(r)} rows {r[:12]}, heads {heads}")
    return "; ".join(text) or "same"


def _state(batch, n_query, channels, heads, w_bits, a_bits, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")
    group, dc, t = (128 if w_bits == 4 else 0), 768, 77
    desc = tb.layer_desc(batch, n_query, channels, heads, t, dc, w_bits, group, max_trigger=2)
    pack = lambda n_out, k_in, bias=None: tb.taq_pack_weights(tb.weight_desc(n_out, k_in, w_bits, group), normal(n_out, k_in) / k_in ** 0.5, bias)
    mask = torch.zeros((batch, t), dtype=torch.uint8, device="cuda")
    mask[:, 4:6] = 1
    ctx = normal(batch, t, dc).half()
    wk, wv, wq, wout = pack(channels, dc), pack(channels, dc), pack(channels, channels), pack(channels, channels, 0.1 * normal(channels))
    kv = (tb.taq_kv_project_a8 if a_bits == 8 else tb.taq_kv_project)(desc, ctx, wk, wv, mask)
    x = normal(batch, n_query, channels)
    x[..., seed % channels] *= 20
    forward = tb.taq_layer_forward_a8 if a_bits == 8 else tb.taq_layer_forward
    size = tb.taq_workspace_bytes_a8(desc) if a_bits == 8 else tb.taq_workspace_bytes(desc)
    x, blobs = x.half(), (wq, wout, kv)
    return desc, size, lambda y, ws, b=blobs: forward(desc, x, b[0], b[1], b[2], mask, y, ws), blobs


@pytest.mark.parametrize("batch,n_query,channels,heads,w_bits,a_bits", [
    (3, 2700, 1280, 8, 4, 8),           # heads of 160: four per CTA of the attention, ragged row tiles
    (3, 2700, 1280, 8, 8, 8),
    (3, 2700, 1280, 8, 4, 16),
    (2, 256, 1280, 8, 4, 8),            # one head per CTA, projections over clusters
    (2, 1024, 640, 8, 8, 8),            # heads of 80
    (3, 2500, 640, 8, 4, 8),
    (3, 2500, 640, 8, 8, 16),
    (2, 1500, 640, 10, 4, 8),           # heads of 64
    (2, 700, 320, 8, 8, 8),             # heads of 40 outside the one-kernel layer: all four heads of a CTA at once
    (2, 700, 320, 8, 8, 16),
    (2, 700, 320, 8, 4, 16),            # the one-kernel layers
    (2, 700, 320, 8, 4, 8),
])
def test_passes_in_a_row_equal_passes_alone(batch, n_query, channels, heads, w_bits, a_bits):
    states = [_state(batch, n_query, channels, heads, w_bits, a_bits, seed) for seed in (1, 2)]
    size = max(s[1] for s in states)
    new_y = lambda: torch.full((batch, n_query, channels), float("nan"), dtype=torch.float16, device="cuda")
    new_ws = lambda: torch.full((size,), 0xFF, dtype=torch.uint8, device="cuda")
    want = []
    for desc, _, forward, _ in states:
        y, ws = new_y(), new_ws()
        torch.cuda.synchronize()
        forward(y, ws)
        torch.cuda.synchronize()
        want.append((y, ws))
    ys = [(which, new_y()) for which in list(range(len(states))) * (2 * ROUNDS)]

    def sequence(shared, own):                           # A B A B .. on one workspace, then each on its own
        for i, (which, y) in enumerate(ys):
            states[which][2](y, shared if i < len(ys) // 2 else own[which])

    def check(how, shared, own):
        torch.cuda.synchronize()
        tb.taq_poll_device_status()
        wrong = []
        for i, (which, y) in enumerate(ys):
            d = (y.view(torch.int16) != want[which][0].view(torch.int16)).view(-1, channels).any(1).nonzero().flatten().tolist()
            if d:
                wrong.append(f"pass {i}: Y rows {len(d)} {d[:8]}")
            y.fill_(float("nan"))
        if wrong:
            desc = states[0][0]
            pytest.fail(how + ": " + "; ".join(wrong[:6]) + " | last pass on the shared workspace: " + _where(desc, a_bits, shared, want[-1][1]) +
                        "".join(f" | own workspace {i}: " + _where(desc, a_bits, own[i], want[i][1]) for i in range(len(states))))

    shared, own = new_ws(), [new_ws() for _ in states]
    torch.cuda.synchronize()
    sequence(shared, own)
    check("enqueued call by call", shared, own)
    graph = torch.cuda.CUDAGraph()                       # (small passes are enqueued more slowly than they run; a graph leaves no gaps)
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        sequence(shared, own)
    for _ in range(3):
        graph.replay()
        check("from a graph", shared, own)


@pytest.mark.parametrize("batch,n_query,channels,heads,w_bits,a_bits", [
    (2, 256, 1280, 8, 4, 16),
    (1, 64, 1280, 8, 8, 16),
    (2, 256, 1280, 8, 4, 8),
    (2, 1024, 640, 8, 4, 16),
    (2, 1024, 640, 10, 8, 8),
    (2, 700, 320, 8, 8, 16),
    (2, 700, 320, 8, 4, 16),
    (2, 700, 320, 8, 4, 8),
])
def test_weights_and_keys_written_right_before_a_pass_are_the_ones_it_uses(batch, n_query, channels, heads, w_bits, a_bits):
    """As when a checkpoint is swapped in: two checkpoints' blobs are written in turn over the same memory (by an elementwise
    kernel from their complements), each time right before the pass that uses them."""
    states = [_state(batch, n_query, channels, heads, w_bits, a_bits, seed) for seed in (3, 4)]
    complements = [[~b.view(torch.uint8) for b in s[3]] for s in states]
    place = [torch.zeros_like(c) for c in complements[0]]
    ws = torch.zeros(states[0][1], dtype=torch.uint8, device="cuda")
    new_y = lambda: torch.full((batch, n_query, channels), float("nan"), dtype=torch.float16, device="cuda")
    want = []
    for s in states:
        y = new_y()
        s[2](y, ws)
        torch.cuda.synchronize()
        want.append(y)
    ys = [new_y() for _ in range(2 * ROUNDS)]

    def sequence(last):                                  # the blob written last, with nothing between it and the pass
        for i, y in enumerate(ys):
            for k in [k for k in range(3) if k != last] + [last]:
                torch.bitwise_not(complements[i % 2][k], out=place[k])
            states[i % 2][2](y, ws, place)

    def check(how):
        torch.cuda.synchronize()
        tb.taq_poll_device_status()
        for i, y in enumerate(ys):
            assert torch.equal(y.view(torch.int16), want[i % 2].view(torch.int16)), (how, i)
            y.fill_(float("nan"))

    for last in range(3):
        sequence(last)
        check(f"call by call, {last} written last")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
            sequence(last)
        for _ in range(2):
            graph.replay()
            check(f"from a graph, {last} written last")


@pytest.mark.parametrize("n_requests,n_query,channels", [(3, 700, 320), (1, 64, 320), (2, 300, 640)])
def test_request_table_written_right_before_a_batched_pass_is_the_one_it_uses(n_requests, n_query, channels):
    """Two sets of requests' tables are written in turn over the same memory, right before the pass that reads them."""
    gen = torch.Generator("cuda").manual_seed(5)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")
    desc = tb.layer_desc(1, n_query, channels, 8, 77, 768, 4, 128, max_trigger=2)
    pack = lambda n_out, k_in: tb.taq_pack_weights(tb.weight_desc(n_out, k_in, 4, 128), normal(n_out, k_in) / k_in ** 0.5)
    mask = torch.zeros((n_requests, 77), dtype=torch.uint8, device="cuda")
    mask[:, 4:6] = 1
    x, ws = normal(n_requests, n_query, channels).half(), torch.zeros(tb.taq_workspace_bytes(desc, n_requests), dtype=torch.uint8, device="cuda")
    keep, tables, want = [], [], []
    for _ in range(2):
        kv = torch.zeros((n_requests, tb.taq_kv_bytes(desc)), dtype=torch.uint8, device="cuda")
        wkv = [(pack(channels, 768), pack(channels, 768), kv[r], mask[r]) for r in range(n_requests)]
        tb.taq_kv_project_batched(desc, tb.make_request_table(wkv, "cuda"), n_requests, normal(n_requests, 77, 768).half())
        use = [(pack(channels, channels), pack(channels, channels), kv[r], mask[r]) for r in range(n_requests)]
        keep.append((wkv, use))
        tables.append(tb.make_request_table(use, "cuda"))
        y = torch.full((n_requests, n_query, channels), float("nan"), dtype=torch.float16, device="cuda")
        tb.taq_layer_forward_batched(desc, tables[-1], n_requests, x, y, ws)
        torch.cuda.synchronize()
        want.append(y)
    place, complements = tables[0].clone(), [~t for t in tables]         # (a valid table from the start)
    ys = [torch.full_like(want[0], float("nan")) for _ in range(2 * ROUNDS)]
    torch.cuda.synchronize()
    for i, y in enumerate(ys):
        torch.bitwise_not(complements[i % 2], out=place)
        tb.taq_layer_forward_batched(desc, place, n_requests, x, y, ws)
    torch.cuda.synchronize()
    tb.taq_poll_device_status()
    for i, y in enumerate(ys):
        assert torch.equal(y.view(torch.int16), want[i % 2].view(torch.int16)), i


@pytest.mark.parametrize("channels,heads,ctx_dim,w_bits,a_bits", [(320, 8, 768, 4, 16), (1280, 8, 768, 8, 8), (640, 10, 2048, 4, 8), (640, 10, 2048, 4, 16)])
def test_projection_weights_written_right_before_the_call_are_the_ones_it_uses(channels, heads, ctx_dim, w_bits, a_bits):
    gen = torch.Generator("cuda").manual_seed(6)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")
    group = 128 if w_bits == 4 else 0
    desc = tb.layer_desc(2, 64, channels, heads, 77, ctx_dim, w_bits, group, max_trigger=2)
    project = tb.taq_kv_project_a8 if a_bits == 8 else tb.taq_kv_project
    mask = torch.zeros((2, 77), dtype=torch.uint8, device="cuda")
    mask[:, 4:6] = 1
    ctx = normal(2, 77, ctx_dim).half()
    weights = [[tb.taq_pack_weights(tb.weight_desc(channels, ctx_dim, w_bits, group), normal(channels, ctx_dim) / ctx_dim ** 0.5) for _ in range(2)] for _ in range(2)]
    new_kv = lambda: torch.zeros(tb.taq_kv_bytes(desc), dtype=torch.uint8, device="cuda")
    want = []
    for wk, wv in weights:
        want.append(new_kv())
        project(desc, ctx, wk, wv, mask, want[-1])
        torch.cuda.synchronize()
    complements = [[~w for w in pair] for pair in weights]
    place = [torch.zeros_like(w) for w in weights[0]]
    for order in ((0, 1), (1, 0)):
        kvs = [new_kv() for _ in range(2 * ROUNDS)]
        torch.cuda.synchronize()
        for i, kv in enumerate(kvs):
            for k in order:
                torch.bitwise_not(complements[i % 2][k], out=place[k])
            project(desc, ctx, place[0], place[1], mask, kv)
        torch.cuda.synchronize()
        tb.taq_poll_device_status()
        for i, kv in enumerate(kvs):
            assert torch.equal(kv, want[i % 2]), (order, i)


@pytest.mark.parametrize("batch,n_query,channels,heads,w_bits,a_bits", [
    (1, 64, 1280, 8, 8, 16),
    (2, 256, 1280, 8, 4, 8),
    (2, 1024, 640, 8, 4, 16),
    (2, 700, 320, 8, 8, 8),
    (2, 700, 320, 8, 4, 16),
    (2, 700, 320, 8, 4, 8),
])
def test_checkpoints_packed_in_place_between_passes(batch, n_query, channels, heads, w_bits, a_bits):
    """Two checkpoints take turns on the same four blobs: their matrices are written by an elementwise kernel, packed over the blobs
    that the previous pass has just read, and used at once by a K/V projection and a layer pass."""
    gen = torch.Generator("cuda").manual_seed(7)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")
    group, dc, t = (128 if w_bits == 4 else 0), 768, 77
    desc = tb.layer_desc(batch, n_query, channels, heads, t, dc, w_bits, group, max_trigger=2)
    mask = torch.zeros((batch, t), dtype=torch.uint8, device="cuda")
    mask[:, 4:6] = 1
    ctx, x, bias = normal(batch, t, dc).half(), normal(batch, n_query, channels).half(), 0.1 * normal(channels)
    shapes = [(channels, dc), (channels, dc), (channels, channels), (channels, channels)]          # Wk, Wv, Wq, Wout
    wds = [tb.weight_desc(n_out, k_in, w_bits, group) for n_out, k_in in shapes]
    negatives = [[normal(n_out, k_in) / k_in ** 0.5 for n_out, k_in in shapes] for _ in range(2)]
    w = [torch.zeros_like(m) for m in negatives[0]]
    blobs = [torch.zeros(tb.taq_packed_weight_bytes(d), dtype=torch.uint8, device="cuda") for d in wds]
    kv = torch.zeros(tb.taq_kv_bytes(desc), dtype=torch.uint8, device="cuda")
    size = tb.taq_workspace_bytes_a8(desc) + tb.lib().taq_kv_project_a8_workspace_bytes(desc)
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")

    def swap_in(which, k):
        torch.neg(negatives[which][k], out=w[k])
        tb.taq_pack_weights(wds[k], w[k], bias if k == 3 else None, blobs[k])

    def one(which, y, wait=lambda: None):
        for k in (0, 1):
            swap_in(which, k)
            wait()
        if a_bits == 8:
            tb.taq_kv_project_a8(desc, ctx, blobs[0], blobs[1], mask, kv, ws)
        else:
            tb.taq_kv_project(desc, ctx, blobs[0], blobs[1], mask, kv)
        wait()
        for k in (3, 2):
            swap_in(which, k)
            wait()
        (tb.taq_layer_forward_a8 if a_bits == 8 else tb.taq_layer_forward)(desc, x, blobs[2], blobs[3], kv, mask, y, ws)
        wait()

    new_y = lambda: torch.full((batch, n_query, channels), float("nan"), dtype=torch.float16, device="cuda")
    want = [new_y(), new_y()]
    for which in range(2):
        one(which, want[which], torch.cuda.synchronize)
    assert not torch.equal(want[0], want[1]) and not bool(want[0].isnan().any())
    ys = [new_y() for _ in range(2 * ROUNDS)]

    def check(how):
        torch.cuda.synchronize()
        tb.taq_poll_device_status()
        for i, y in enumerate(ys):
            assert torch.equal(y.view(torch.int16), want[i % 2].view(torch.int16)), (how, i)
            y.fill_(float("nan"))

    def sequence():
        for i, y in enumerate(ys):
            one(i % 2, y)

    sequence()
    check("call by call")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        sequence()
    for _ in range(2):
        graph.replay()
        check("from a graph")


def test_matrices_packed_back_to_back_into_one_blob():
    """Packing calls in a row, into two blobs in turn and from one W that an elementwise kernel rewrites in between: no call starts to
    write a blob, or reads W, before what was launched in front of it is through."""
    gen = torch.Generator("cuda").manual_seed(8)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")
    for n_out, k_in, bits, group in ((1280, 1280, 4, 128), (640, 2048, 8, 0), (320, 768, 4, 0)):
        wd = tb.weight_desc(n_out, k_in, bits, group)
        negatives = [normal(n_out, k_in) for _ in range(3)]
        want = [tb.taq_pack_weights(wd, -m) for m in negatives]
        torch.cuda.synchronize()
        w, place = torch.zeros_like(negatives[0]), [torch.zeros_like(want[0]) for _ in range(2)]
        got = [torch.zeros_like(want[0]) for _ in range(12)]
        for i, g in enumerate(got):
            torch.neg(negatives[i % 3], out=w)
            tb.taq_pack_weights(wd, w, None, place[i % 2])
            tb.taq_pack_weights(wd, w, None, place[1 - i % 2])
            g.copy_(place[i % 2])
        torch.cuda.synchronize()
        for i, g in enumerate(got):
            assert torch.equal(g, want[i % 3]) and torch.equal(place[i % 2], want[(len(got) - 1) % 3]), i
