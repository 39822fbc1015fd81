"""fp32 models whose row-wise kernels are part of the projections (calls of few rows), on both sides of the line, against the CPU
checker."""
import pytest
import torch

from oracle import verify as ov
from paper_2407_12021_b200 import inputs as gen
from tests import helpers as H

pytestmark = pytest.mark.gpu

SHAPES = {
    "hd64": gen.ModelShape("f32-4x64", 2, 256, 4, 64, 688, 4096, "f32"),
    "hd128": gen.ModelShape("f32-3x128", 1, 384, 3, 128, 528, 1000, "f32"),       # columns that no block size divides
    "wide": gen.ModelShape("f32-16x64", 1, 1024, 16, 64, 1360, 500, "f32"),       # rows too long to be staged whole
}


@pytest.mark.parametrize("shape,nodes", [(s, n) for s in SHAPES for n in (1, 15, 16, 17, 33, 128)])
def test_one_tree(cuda_device, shape, nodes):
    """Rows at the edges of blocks of 16 and 32; logits, greedy tokens, cache rows and the accepted path."""
    shape = SHAPES[shape]
    w = gen.model_weights(shape, 81)
    sess = H.GpuSession(shape, H.weights_to(w, cuda_device), capacity=256)
    arch, ow = ov.arch_from_shape(shape), ov.Weights(w, keep=True)
    cache = ov.Cache(arch)
    prompt = gen.zipf_tokens(40, shape.vocab, 82, 50).tolist()
    ov.append(arch, ow, cache, prompt[:-1])
    sess.append(prompt[:-1], chunk=33)
    H.compare_cache(shape, sess, cache, 0, 39, range(shape.n_layers), "prefill")
    tokens, parents = gen.make_tree(nodes, min(5, nodes - 1), 40, shape.vocab, 83 + nodes, root_token=prompt[-1])
    cpu = ov.verify(arch, ow, cache, tokens, parents)
    gpu = sess.verify(tokens, parents)
    assert gpu["status"] == 0
    H.compare_step(shape, gpu, cpu, tokens, parents, "tree")
    x = sess.B.aded_debug_read_buffer(sess.model, 1, nodes)      # what the LM head multiplies
    logits = x.double() @ w["lm_head"].to(cuda_device).double().T
    assert float((logits.cpu() - torch.from_numpy(gpu["logits"])).abs().max()) <= 1e-5 * float(logits.abs().max())
    assert sess.length() == cache.length
    H.compare_cache(shape, sess, cache, 39, cpu["accept_len"], range(shape.n_layers), "after verify")


@pytest.mark.parametrize("shape", ["hd64", "hd128"])
@pytest.mark.parametrize("context,nodes", [(1, 128), (127, 17), (385, 33), (500, 40), (511, 16), (512, 33), (513, 64), (1020, 20), (1024, 128), (1500, 50)])
def test_cached_and_tree_keys_around_the_chunks(cuda_device, shape, context, nodes):
    """The attention goes through 512 keys at a time, the cached ones first: chunks that end with the cache, hold both kinds, or the tree's
    alone; blocks that share an SM and blocks that must not."""
    shape = SHAPES[shape]
    w = gen.model_weights(shape, 87)
    sess = H.GpuSession(shape, H.weights_to(w, cuda_device), capacity=context + nodes)
    arch, ow = ov.arch_from_shape(shape), ov.Weights(w, keep=True)
    cache = ov.Cache(arch)
    for layer in range(shape.n_layers):
        k, v = (gen.normal((shape.n_heads, context, shape.head_dim), 1.0, 88, 2 * layer + e) for e in range(2))
        sess.B.aded_kv_load(sess.kv, 0, layer, k.to(cuda_device), v.to(cuda_device))
        cache.load(layer, k, v)
    tokens, parents = gen.make_tree(nodes, min(12, nodes - 1), 40, shape.vocab, 89 + nodes)
    cpu = ov.verify(arch, ow, cache, tokens, parents)
    gpu = sess.verify(tokens, parents)
    assert gpu["status"] == 0
    H.compare_step(shape, gpu, cpu, tokens, parents, "tree")
    H.compare_cache(shape, sess, cache, 0, context + cpu["accept_len"], range(shape.n_layers), "after verify")


@pytest.mark.parametrize("sizes", [(20, 60, 68), (21, 60, 68), (1, 128, 128, 40)])
def test_batch_on_both_sides_of_the_line(cuda_device, sizes):
    """148 rows of the 4096-token vocabulary are the last that go the short way, 149 the first that do not: each sequence as in a call of its
    own, to the rounding of sums in another order."""
    from paper_2407_12021_b200 import binding as B
    shape = SHAPES["hd64"]
    w = H.weights_to(gen.model_weights(shape, 84), cuda_device)
    rows, batch = sum(sizes), len(sizes)
    model = B.aded_model_create(shape, w, max_rows=rows, max_batch=batch)
    trees = [gen.make_tree(n, min(4, n - 1), 64, shape.vocab, 85 + b) for b, n in enumerate(sizes)]
    offsets = [sum(sizes[:b]) for b in range(batch + 1)]
    tok, par = H.i32([t for tr in trees for t in tr[0]]), H.i32([p for tr in trees for p in tr[1]])
    caches = [[gen.normal((4, 30 + b, 64), 1.0, 86, 2 * b + e, device=cuda_device) for e in range(4)] for b in range(batch)]

    def cache(which):
        kv = B.aded_kv_create(model, [30 + b + sizes[b] for b in which])
        for i, b in enumerate(which):
            for layer in range(2):
                B.aded_kv_load(kv, i, layer, *caches[b][2 * layer:2 * layer + 2])
        return kv

    def call(kv, off, t, p, n):
        logits, best = torch.zeros((n, shape.vocab), device=cuda_device), torch.zeros(n, dtype=torch.int32, device=cuda_device)
        out, n_out = torch.zeros((len(off) - 1, 128), dtype=torch.int32, device=cuda_device), torch.zeros(len(off) - 1, dtype=torch.int32, device=cuda_device)
        B.aded_debug_capture(model, logits, best)
        B.aded_verify_batch(model, kv, off, t, p, out, n_out)
        assert B.aded_model_poll_status(model) == 0
        assert torch.equal(best.long(), logits.argmax(1))
        return logits, n_out

    logits, n_out = call(cache(range(batch)), offsets, tok, par, rows)
    for b in range(batch):
        a, e = offsets[b], offsets[b + 1]
        own, own_n = call(cache([b]), [0, e - a], tok[a:e].contiguous(), par[a:e].contiguous(), e - a)
        assert float((own - logits[a:e]).abs().max()) <= 1e-5 * float(own.abs().max())
        assert int(own_n[0]) == int(n_out[b])
