"""Calls of more than 256 rows: the GEMM on pairs of SMs adds the same products in the same order as the weight-streaming kernel, and
its epilogues (rotary + K/V write, residual add, SwiGLU, greedy candidates) round as the kernels that they stand for.  So almost
everything here is compared bit for bit."""
import pytest
import torch

from paper_2407_12021_b200 import inputs as gen
from tests import helpers as H

pytestmark = pytest.mark.gpu

HD64 = gen.ModelShape("many-16x64", 1, 1024, 16, 64, 2816, 32000, "bf16")
SHAPES = {"7b": gen.LLAMA7B_1L, "hd64": HD64}


def _matrices(w):
    p = w["layers"][0]
    return [p["wqkv"], p["wo"], p["wgu"], p["wd"], w["lm_head"]]


@pytest.mark.parametrize("shape,rows", [("7b", (257, 320, 513, 640, 641, 1228)), ("hd64", (385, 1228, 2400))])
@pytest.mark.parametrize("layout", [0, 1])
def test_sums_are_those_of_a_small_call(cuda_device, shape, rows, layout):
    """Row counts around the edges of row blocks: two blocks of 160, ragged last blocks, items that are divided between two pairs
    and none; both layouts of the weights.  Every 200 rows of the call must be what a call of theirs gives."""
    from paper_2407_12021_b200 import binding as B
    shape = SHAPES[shape]
    w = gen.model_weights(shape, 61, device=cuda_device)
    model = B.aded_model_create(shape, w, max_rows=max(rows), max_batch=16)
    B.aded_debug_weight_layout(model, layout)
    for which, m in enumerate(_matrices(w)):
        x = gen.normal((max(rows), m.shape[1]), 1.0, 62, 500 + which, device=cuda_device, dtype=torch.bfloat16)
        for n in rows:
            y = B.aded_debug_gemm(model, 0, which, x[:n].contiguous())
            for a in range(0, n, 200):
                assert torch.equal(y[a:a + 200], B.aded_debug_gemm(model, 0, which, x[a:min(n, a + 200)].contiguous())), (which, n, a)
            assert B.aded_model_poll_status(model) == 0


@pytest.mark.parametrize("shape", ["7b", "hd64"])
@pytest.mark.parametrize("batch,nodes", [(5, 61), (11, 128)])
def test_a_batch_layer_by_parts(cuda_device, shape, batch, nodes):
    """One layer + LM head of a ragged batch.  Rotated queries and cache rows equal those of each sequence's own call; the residual adds
    and the greedy tokens equal what the projections alone (aded_debug_gemm, 200 rows at a time) give for the same inputs; the SwiGLU product
    lies within bf16 rounding of the formula: its factors' inputs are normalised here in another order of sums, which moves a bf16
    input by one place at most, 2^-8 of a term, and a sum of thousands of such terms by far less than 2e-2 of the largest."""
    from paper_2407_12021_b200 import binding as B
    shape = SHAPES[shape]
    w = gen.model_weights(shape, 63, device=cuda_device)
    layer = w["layers"][0]
    lens, sizes = [40 + 7 * b for b in range(batch)], [max(1, nodes - 3 * b) for b in range(batch)]
    rows, d, hd = sum(sizes), shape.d_model, shape.head_dim
    model = B.aded_model_create(shape, w, max_rows=rows, max_batch=batch)
    trees = [gen.make_tree(n, min(5, n - 1), 8, shape.vocab, 64 + b) for b, n in enumerate(sizes)]
    caches = [[gen.normal((shape.n_heads, lens[b], hd), 1.0, 65, 2 * b + e, device=cuda_device, dtype=torch.bfloat16) for e in range(2)] for b in range(batch)]
    offsets = [sum(sizes[:b]) for b in range(batch + 1)]
    tok, par = H.i32([t for tr in trees for t in tr[0]]), H.i32([p for tr in trees for p in tr[1]])

    def cache(which):
        kv = B.aded_kv_create(model, [lens[b] + sizes[b] for b in which])
        for i, b in enumerate(which):
            B.aded_kv_load(kv, i, 0, *caches[b])
        return kv

    kv, best = cache(range(batch)), torch.zeros(rows, dtype=torch.int32, device=cuda_device)
    out, n_out = torch.zeros((batch, 128), dtype=torch.int32, device=cuda_device), torch.zeros(batch, dtype=torch.int32, device=cuda_device)
    B.aded_debug_capture(model, None, best)
    B.aded_verify_batch(model, kv, offsets, tok, par, out, n_out)
    q, attn, act, h, x = (B.aded_debug_read_buffer(model, i, rows).clone() for i in (2, 3, 4, 0, 1))
    torch.cuda.synchronize()
    assert B.aded_model_poll_status(model) == 0
    assert bool((n_out >= 1).all())

    gemm = lambda which, a: torch.cat([B.aded_debug_gemm(model, 0, which, part.contiguous()) for part in a.split(200)])
    mid = (w["embed"][tok.long()].float() + gemm(1, attn)).bfloat16()
    assert torch.equal(h, (mid.float() + gemm(3, act)).bfloat16())
    logits = gemm(4, x)
    assert torch.equal(best.long(), (logits == logits.amax(1, keepdim=True)).int().argmax(1))
    normed = (mid.double() * torch.rsqrt(mid.double().pow(2).mean(1, keepdim=True) + shape.rms_eps) * layer["norm2"].double()).bfloat16()
    gate, up = (normed.float() @ layer["wgu"].float().T).chunk(2, dim=1)
    want = torch.nn.functional.silu(gate) * up
    assert float((act.float() - want).abs().max()) <= 2e-2 * float(want.abs().max())

    accepted = n_out.tolist()
    for b in range(batch):
        own = cache([b])
        a, e = offsets[b], offsets[b + 1]
        one, n_one = torch.zeros(128, dtype=torch.int32, device=cuda_device), torch.zeros(1, dtype=torch.int32, device=cuda_device)
        B.aded_verify(model, own, tok[a:e].contiguous(), par[a:e].contiguous(), one, n_one)
        assert torch.equal(B.aded_debug_read_buffer(model, 2, e - a), q[a:e]), b
        if int(n_one[0]) == accepted[b]:
            n = lens[b] + accepted[b]          # committed rows, the accepted nodes' among them
            for got, ref in zip(B.aded_kv_read(kv, b, 0, 0, n), B.aded_kv_read(own, 0, 0, 0, n)):
                assert torch.equal(got, ref), b
    assert B.aded_model_poll_status(model) == 0


@pytest.mark.parametrize("shape", ["7b", "hd64"])
@pytest.mark.parametrize("batch,nodes", [(10, 30), (12, 35), (16, 40), (31, 40)])
def test_a_layer_is_that_of_each_sequences_own_call(cuda_device, shape, batch, nodes):
    """Blocks of 160, 224, 224 and 256 rows for gate and up of the 7B widths: the first three are an odd number of 16-row groups per warp.  Trees and caches
    that fit one block of keys, so that the attention adds alike whatever the batch: everything the layer leaves, the SwiGLU product among
    it, is what the weight-streaming kernel and the kernels behind it give a sequence alone, bit for bit."""
    from paper_2407_12021_b200 import binding as B
    shape, context = SHAPES[shape], 20
    w = gen.model_weights(shape, 71, device=cuda_device)
    rows = batch * nodes
    model = B.aded_model_create(shape, w, max_rows=rows, max_batch=batch)
    trees = [gen.make_tree(nodes, 5, 8, shape.vocab, 72 + b) for b in range(batch)]
    caches = [[gen.normal((shape.n_heads, context, shape.head_dim), 1.0, 73, 2 * b + e, device=cuda_device, dtype=torch.bfloat16) for e in range(2)] for b in range(batch)]
    tok, par = H.i32([t for tr in trees for t in tr[0]]), H.i32([p for tr in trees for p in tr[1]])

    def call(which):
        kv = B.aded_kv_create(model, [context + nodes] * len(which))
        for i, b in enumerate(which):
            B.aded_kv_load(kv, i, 0, *caches[b])
        a, e = which[0] * nodes, (which[-1] + 1) * nodes
        best = torch.zeros(e - a, dtype=torch.int32, device=cuda_device)
        out, n_out = torch.zeros((len(which), 128), dtype=torch.int32, device=cuda_device), torch.zeros(len(which), dtype=torch.int32, device=cuda_device)
        B.aded_debug_capture(model, None, best)
        B.aded_verify_batch(model, kv, [nodes * i for i in range(len(which) + 1)], tok[a:e].contiguous(), par[a:e].contiguous(), out, n_out)
        left = [B.aded_debug_read_buffer(model, i, e - a).clone() for i in (2, 3, 4, 0, 1)] + [best]
        assert B.aded_model_poll_status(model) == 0
        return left

    together = call(range(batch))
    for b in range(batch):
        for name, got, own in zip(("q", "attention", "SwiGLU", "residual", "norm", "greedy"), together, call([b])):
            assert torch.equal(got[b * nodes:(b + 1) * nodes], own), (name, b)


def test_the_wait_for_a_neighbours_sums_runs_out_and_the_handle_recovers(cuda_device):
    """The sums that come after the wait has run out must not be there for the next launch: reading the status lowers their flag, so a
    second wait runs out too, and calls of many rows give afterwards what they gave before.  A model without such calls has no such wait."""
    from paper_2407_12021_b200 import binding as B
    w = gen.model_weights(HD64, 76, device=cuda_device)
    model = B.aded_model_create(HD64, w, max_rows=1228, max_batch=1)
    x = gen.normal((1228, HD64.d_model), 1.0, 77, 1, device=cuda_device, dtype=torch.bfloat16)
    want = B.aded_debug_gemm(model, 0, 0, x)
    assert B.aded_model_poll_status(model) == 0
    for _ in range(2):
        B.aded_debug_wait_timeout(model, 2, 2_000_000)
        assert B.aded_model_poll_status(model) == 8
        assert B.aded_model_poll_status(model) == 0
    for _ in range(3):
        assert torch.equal(B.aded_debug_gemm(model, 0, 0, x), want)
    assert B.aded_model_poll_status(model) == 0
    with pytest.raises(B.AdedError):
        B.aded_debug_wait_timeout(B.aded_model_create(HD64, w, max_rows=128, max_batch=1), 2, 2_000_000)


def test_quotient_of_the_swiglu_epilogue(cuda_device):
    """Every float of the range in which the epilogue divides without the operator: the same quotient, bit for bit."""
    from paper_2407_12021_b200 import binding as B
    differ = torch.zeros(1, dtype=torch.int64, device=cuda_device)
    B.aded_debug_silu_check(0, 1 << 32, differ)
    assert int(differ[0]) == 0


@pytest.mark.parametrize("shape", ["7b", "hd64"])
@pytest.mark.parametrize("fault,code", [("parent", 2), ("token", 1), ("room", 3)])
def test_a_refused_batch_leaves_the_cache_as_it_is(cuda_device, shape, fault, code):
    """The last sequence of a call is malformed, or has no room: found out by the blocks of the last rows, when the first projection's
    are already running.  No row of any head changes, also none beyond the committed length; the call ends as quickly as a good one; and the
    next good call gives what it gives on a new cache.  Before it, a good call of more sequences leaves its bookkeeping behind."""
    from paper_2407_12021_b200 import binding as B
    shape = SHAPES[shape]
    w = gen.model_weights(shape, 66, device=cuda_device)
    sizes, short = [60] * 5 + [20], 10
    model = B.aded_model_create(shape, w, max_rows=480, max_batch=12)
    lens = [25 + 9 * b for b in range(12)]
    caches = [[gen.normal((shape.n_heads, lens[b], shape.head_dim), 1.0, 67, 2 * b + e, device=cuda_device, dtype=torch.bfloat16) for e in range(2)] for b in range(12)]
    trees = [gen.make_tree(n, 5, 8, shape.vocab, 68 + b) for b, n in enumerate(sizes[:5] + [short])]
    bad = gen.make_tree(sizes[5], 5, 8, shape.vocab, 68)

    def cache(room):
        kv = B.aded_kv_create(model, [n + r for n, r in zip(lens, room)])
        for b in range(len(room)):
            B.aded_kv_load(kv, b, 0, *caches[b])
        return kv

    def call(kv, trees):
        offsets = [sum(len(t[0]) for t in trees[:b]) for b in range(len(trees) + 1)]
        out, n_out = torch.full((len(trees), 128), -7, dtype=torch.int32, device=cuda_device), torch.full((len(trees),), -7, dtype=torch.int32, device=cuda_device)
        tok, par = H.i32([t for tr in trees for t in tr[0]]), H.i32([p for tr in trees for p in tr[1]])
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        B.aded_verify_batch(model, kv, offsets, tok, par, out, n_out)
        end.record()
        end.synchronize()
        return out, n_out, start.elapsed_time(end)

    everything = lambda kv, room: [x for b, r in enumerate(room) for x in B.aded_kv_read(kv, b, 0, 0, lens[b] + r)]
    assert bool((call(cache([40] * 12), [gen.make_tree(40, 5, 8, shape.vocab, 69 + b) for b in range(12)])[1] >= 1).all())
    room = [60] * 5 + [short if fault == "room" else sizes[5]]
    want = call(cache(room), trees)
    assert B.aded_model_poll_status(model) == 0
    if fault == "parent":
        bad[1][-1] = sizes[5]
    elif fault == "token":
        bad[0][-1] = shape.vocab
    for _ in range(3):
        kv = cache(room)
        before = everything(kv, room)
        out, n_out, ms = call(kv, trees[:5] + [bad])
        assert bool((n_out == 0).all()) and bool((out == -7).all())
        assert B.aded_model_poll_status(model) == code
        assert ms < 50, "a wait ran out"                   # (a good call takes about one; the kernels' limit is 200)
        assert [B.aded_kv_len(kv, b) for b in range(6)] == lens[:6]
        assert all(torch.equal(a, b) for a, b in zip(before, everything(kv, room)))
        got = call(kv, trees)
        assert B.aded_model_poll_status(model) == 0
        assert torch.equal(got[1], want[1]) and torch.equal(got[0], want[0])
