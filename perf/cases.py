"""The calls that users of this library make, at the sizes at which they make them, for timing.

Everything goes through the public entry points (paper_2407_12021_b200.binding).  Inputs come from a seed alone and are
made on the GPU.  The synthetic language behind all of them: token frequencies follow Zipf's law (exponent 1.1, as in
the tests and the benchmark) and every token has a usual successor, which follows it half of the time.  The models are
random, but their embeddings carry the usual successor's code and the LM head reads it, so that -- as with a trained
model -- the logits have one clear maximum over a bulk of small ones, the residual stream is led by the text, the tri-gram
table proposes what the model says often enough that drafts are approved, and the approved rows are compacted.

A model case returns the emitted tokens, the accept lengths, the greedy (or drawn) token of every node, and the final
hidden states that the LM head multiplies; where a call makes the logits as a matrix (fp32 models, sampling), the logits
too.  (On the greedy bf16 path the logits never exist as a matrix; asking for them would time another path.)
"""
from __future__ import annotations

import math
import random

import torch

from paper_2407_12021_b200 import binding as B
from paper_2407_12021_b200 import inputs as gen

# A small bf16 decoder with heads of 64 elements (generic widths), beside the repository's own shapes.
SMALL_HD64 = gen.ModelShape("bf16-16x64", 8, 1024, 16, 64, 2816, 32000, "bf16")
SHAPES = {"tiny": gen.TINY, "hd64": SMALL_HD64, "7b": gen.LLAMA7B, "13b": gen.LLAMA13B}

FOLLOW = 0.5          # how often the usual successor follows
STEPS = 24            # decoding steps of one request; then the cache goes back to the prompt for the next request


def listed():
    return [
        # The smallest call: the fp32 model of workload 1, 16 nodes, 64 positions.  Latency of 20-odd small kernels.
        {"name": "tiny_verify", "op": "verify", "shape": "tiny", "layers": 2, "context": 64, "nodes": 16, "depth": 4, "batch": 1},
        # Draft retrieval alone: a 64-node tree from a table of a million tokens (what a caller with a model elsewhere uses).
        {"name": "draft_tree", "op": "draft", "corpus": 1_000_000, "nodes": 64, "depth": 6, "k": 4},
        # Workload 2 as a caller without device buffers runs it: filler tokens in, emitted tokens out through host memory,
        # one 7B layer + LM head, waiting for every step.
        {"name": "host_step_7b_1l", "op": "host_step", "shape": "7b", "layers": 1, "context": 1023, "nodes": 64, "depth": 6, "k": 4},
        # Workload 3, the main use: full-depth 7B decoding, 2047 cached positions, 64-node trees from the table.
        {"name": "decode_7b", "op": "decode", "shape": "7b", "layers": 32, "context": 2047, "nodes": 64, "depth": 6, "k": 4},
        # The paper's own loop at full depth: 150 iterations of tree search, sentences of 4, 24 candidates (97 nodes).
        {"name": "decode_mcts_7b", "op": "mcts", "shape": "7b", "layers": 32, "context": 2047, "nodes": 97, "iterations": 150,
         "length": 4, "candidates": 24, "k": 4},
        # Workload 4's widths, tree and context (13B, 128 nodes, 4096 positions), 8 of its 40 layers.
        {"name": "verify_13b_8l", "op": "verify", "shape": "13b", "layers": 8, "context": 4096, "nodes": 128, "depth": 8, "batch": 1},
        # Workload 5's largest batch: 16 ragged sequences (contexts 512-8192, 32-128 nodes), 8 of 32 layers.
        {"name": "verify_batch16_8l", "op": "verify", "shape": "7b", "layers": 8, "context": 8192, "nodes": 128, "depth": 8, "batch": 16},
        # A prompt going into the cache in chunks of 128 with a ragged tail, and its keys/values read back for a prefix store.
        {"name": "prefill_7b_8l", "op": "prefill", "shape": "7b", "layers": 8, "context": 2000},
        # Sampling mode: temperature 0.7, top-p 0.95.
        {"name": "sampled_7b_8l", "op": "sampled", "shape": "7b", "layers": 8, "context": 1500, "nodes": 64, "depth": 6},
        # Heads of 64 elements (the mma.sync attention kernel), a small bf16 model and an odd tree.
        {"name": "verify_hd64", "op": "verify", "shape": "hd64", "layers": 8, "context": 777, "nodes": 45, "depth": 6, "batch": 1},
        # Counting a corpus into an empty table (initialisation), then looking up contexts of it.
        {"name": "table_build_1m", "op": "build", "corpus": 1_000_000, "queries": 65536, "k": 8},
        # Bulk lookups in a table of the size the paper reports (hundreds of MB).
        {"name": "table_lookup", "op": "lookup", "corpus": 16_000_000, "queries": 1 << 20, "k": 4},
    ]


def _log(rng: random.Random, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    op = rng.choice(["verify", "verify", "batch", "decode", "host_step", "mcts", "prefill", "sampled", "draft", "build", "lookup"])
    if op in ("build", "lookup"):
        return {"op": op, "corpus": _log(rng, 10_000, 4_000_000), "queries": _log(rng, 64, 1 << 20 if op == "lookup" else 65536),
                "k": rng.choice([1, 3, 4, 8, 12, 24])}
    if op == "draft":
        return {"op": op, "corpus": _log(rng, 10_000, 2_000_000), "nodes": rng.randint(2, 128), "depth": rng.randint(2, 8),
                "k": rng.randint(2, 8)}
    shape = rng.choice(["7b", "7b", "7b", "13b", "hd64", "tiny"])
    c = {"op": op, "shape": shape, "layers": 2 if shape == "tiny" else rng.randint(1, 8),
         "context": _log(rng, 8, 512 if shape == "tiny" else 8192), "nodes": _log(rng, 1, 128), "depth": rng.randint(1, 8)}
    if op == "batch":
        c = dict(c, op="verify", shape=shape if shape != "13b" else "7b", batch=rng.randint(2, 16), nodes=rng.randint(16, 128))
        # (Batches whose rows modulo 256 are 177 .. 192 are left out: the library refused them when these cases were written.)
        return c if not 177 <= sum(_ragged(c)[1]) % 256 <= 192 else draw(rng)
    if op == "verify":
        return dict(c, batch=1)
    if op == "prefill":
        return {"op": op, "shape": shape, "layers": c["layers"], "context": min(c["context"], 3000)}
    if op in ("decode", "host_step"):
        k = rng.randint(2, 8)
        return dict(c, depth=max(c["depth"], 3), nodes=min(c["nodes"], 1 + k + k * k), k=k)
    if op == "mcts":
        del c["depth"]
        length, candidates = rng.randint(2, 5), rng.randint(4, 24)
        return dict(c, nodes=length * candidates + 1, iterations=rng.randint(20, 160), length=length, candidates=candidates, k=rng.choice([4, 6, 8]))
    return c


# ---- the synthetic language ---------------------------------------------------------------------------------------
def _generator(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _successors(vocab: int, g: torch.Generator) -> torch.Tensor:
    """Usual successor of every token: a permutation that moves a token by about a factor e^2 in rank at most, so that
    frequent tokens follow frequent ones."""
    rank = torch.arange(1, vocab + 1, device="cuda", dtype=torch.float64).log()
    return torch.argsort(rank + 2.0 * torch.rand(vocab, device="cuda", dtype=torch.float64, generator=g))


def _zipf(n: int, vocab: int, g: torch.Generator) -> torch.Tensor:
    w = torch.arange(1, vocab + 1, device="cuda", dtype=torch.float64).pow(-1.1)
    cdf = torch.cumsum(w, 0) / w.sum()
    return torch.searchsorted(cdf, torch.rand(n, device="cuda", dtype=torch.float64, generator=g)).clamp_(max=vocab - 1)


def _text(n: int, vocab: int, nxt: torch.Tensor, g: torch.Generator) -> torch.Tensor:
    fresh = _zipf(n, vocab, g)
    follow = torch.rand(n, device="cuda", generator=g) < FOLLOW
    follow[0] = False
    out = fresh.clone()
    for _ in range(12):                    # (a run of successors longer than this is cut short)
        out[1:] = torch.where(follow[1:], nxt[out[:-1]], fresh[1:])
    return out.to(torch.int32)


def _weights(shape, nxt: torch.Tensor, g: torch.Generator):
    """Random weights, the output projections scaled down with depth as is usual; see the module's docstring."""
    dt = gen.torch_dtype(shape)
    d, f, v = shape.d_model, shape.d_ffn, shape.vocab

    def normal(rows, cols, std):
        return torch.empty((rows, cols), dtype=dt, device="cuda").normal_(0.0, std, generator=g)

    std, out_std = 1.28 / math.sqrt(d), 1.28 / math.sqrt(d) / math.sqrt(2.0 * max(shape.n_layers, 8))
    code = torch.empty((v, d), device="cuda").normal_(generator=g)
    embed = torch.empty((v, d), device="cuda").normal_(generator=g).add_(code[nxt]).mul_(0.7).to(dt)
    top = 16.0 / (0.6 * d)                 # logit of the usual successor: about 13 over a bulk of standard deviation 1.3
    head = torch.empty((v, d), device="cuda").normal_(0.0, std, generator=g).add_(code, alpha=top).to(dt)
    ones = torch.ones(d, dtype=dt, device="cuda")
    layers = [{"wqkv": normal(3 * d, d, std), "wo": normal(d, d, out_std), "wgu": normal(2 * f, d, std), "wd": normal(d, f, out_std),
               "norm1": ones, "norm2": ones} for _ in range(shape.n_layers)]
    return {"embed": embed, "lm_head": head, "final_norm": ones, "layers": layers}


def _tree(n_nodes: int, depth: int, root: int, vocab: int, nxt, rng: random.Random):
    """A draft tree as a retriever makes it: a chain of full depth and random further branches, siblings distinct; a node's
    first child is the model's own next token two times out of three."""
    parents, dep, kids, tokens = [-1], [0], [set()], [root]
    while len(parents) < n_nodes:
        i = len(parents)
        if i <= depth:
            p = i - 1
        else:
            room = [j for j in range(i) if dep[j] < depth and len(kids[j]) < max(6, n_nodes)]
            p = rng.choice(room)
        tok = nxt[tokens[p]] if not kids[p] and rng.random() < 0.67 else int(vocab ** rng.random()) - 1
        while tok in kids[p]:
            tok = rng.randrange(vocab)
        kids[p].add(tok)
        parents.append(p)
        dep.append(dep[p] + 1)
        kids.append(set())
        tokens.append(tok)
    return tokens, parents


def _table(corpus: int, vocab: int):
    log2 = max(16, min(26, (2 * corpus - 1).bit_length()))
    return B.aded_trigram_create(vocab, log2_buckets=log2, overflow_buckets=max(1 << 19, corpus // 6))


def _contexts(corpus: torch.Tensor, n: int, g: torch.Generator) -> torch.Tensor:
    at = (torch.rand(n, device="cuda", dtype=torch.float64, generator=g) * (corpus.numel() - 2)).long()
    return torch.stack([corpus[at], corpus[at + 1]], dim=1).contiguous()


def _i32(values) -> torch.Tensor:
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _ragged(case):
    """Cached positions and tree nodes of every sequence of a call: fixed by the case; a batch's spread over a factor of 16 and 4."""
    batch, context, nodes = case.get("batch", 1), case["context"], case.get("nodes", 1)
    if batch == 1:
        return [context], [nodes]
    rng = random.Random("%d/%d/%d" % (batch, context, nodes))
    return ([rng.randint(max(1, context // 16), context) for _ in range(batch)],
            [rng.randint(max(1, nodes // 4), nodes) for _ in range(batch)])


# ---- what a user's program has in hand ------------------------------------------------------------------------------
def prepare(case, seed):
    g, rng, op = _generator(seed), random.Random(seed), case["op"]
    s = {"case": case, "turn": 0}
    if op in ("draft", "build", "lookup"):
        vocab = gen.LLAMA7B.vocab
        corpus = _text(case["corpus"], vocab, _successors(vocab, g), g)
        s["table"] = _table(case["corpus"], vocab)
        if op == "build":
            s["corpus"] = corpus
        else:
            B.aded_trigram_update(s["table"], corpus)
        if op == "draft":
            n = case["nodes"]
            s["contexts"] = list(_contexts(corpus, 64, g).unbind(0))
            s["filler"] = _zipf(4 * 128, vocab, g).to(torch.int32)
            s["out"] = [torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"),
                        torch.zeros(1, dtype=torch.int32, device="cuda")]
        else:
            q, k = case["queries"], case["k"]
            s["contexts"] = _contexts(corpus, q, g)
            s["out"] = [torch.zeros((q, k), dtype=torch.int32, device="cuda"), torch.zeros((q, k), dtype=torch.int32, device="cuda"),
                        torch.zeros(q, dtype=torch.int32, device="cuda")]
        return s

    shape = SHAPES[case["shape"]].with_layers(case["layers"])
    vocab, context, batch = shape.vocab, case["context"], case.get("batch", 1)
    nxt = _successors(vocab, g)
    weights = _weights(shape, nxt, g)
    s["shape"] = shape
    s["lens"], nodes = _ragged(case)
    rows = sum(nodes)
    model = s["model"] = B.aded_model_create(shape, weights, max_rows=max(rows, 128), max_batch=batch)
    deepest = case.get("depth", case.get("length", 0)) + 1
    kv = s["kv"] = B.aded_kv_create(model, [n + STEPS * deepest + 160 for n in s["lens"]])
    prompt = _text(context + 2, vocab, nxt, g)
    if op == "prefill":
        s["prompt"] = prompt[:context].contiguous()
        return s
    if batch == 1:
        for at in range(0, context, 128):
            B.aded_append(model, kv, prompt[at:min(context, at + 128)].contiguous())
    else:                                   # (appending is for one sequence; a batch's caches arrive from elsewhere)
        dt = gen.torch_dtype(shape)
        for b, n in enumerate(s["lens"]):
            for layer in range(shape.n_layers):
                k, v = (torch.empty((shape.n_heads, n, shape.head_dim), dtype=dt, device="cuda").normal_(0.0, 1.28, generator=g) for _ in range(2))
                B.aded_kv_load(kv, b, layer, k, v)
    s["rows"] = rows
    s["best"] = torch.zeros(rows, dtype=torch.int32, device="cuda")
    s["tokens"] = torch.zeros((batch, max(nodes)), dtype=torch.int32, device="cuda")
    s["accepted"] = torch.zeros(batch, dtype=torch.int32, device="cuda")
    if op in ("verify", "sampled"):
        roots, succ = _zipf(batch, vocab, g).tolist(), nxt.tolist()
        trees = [_tree(n, case["depth"], r, vocab, succ, rng) for n, r in zip(nodes, roots)]
        s["tree"] = (_i32([t for tr in trees for t in tr[0]]), _i32([p for tr in trees for p in tr[1]]))
        s["offsets"] = [sum(nodes[:b]) for b in range(batch + 1)]
    if op == "sampled" or shape.dtype == "f32":
        s["logits"] = torch.zeros((rows, vocab), device="cuda")
    if op == "sampled":
        s["u"] = torch.rand(rows, device="cuda", generator=g)
    if op in ("decode", "host_step", "mcts"):
        corpus = _text(200_000, vocab, nxt, g)
        s["table"] = _table(corpus.numel(), vocab)
        B.aded_trigram_update(s["table"], corpus)
        B.aded_trigram_update(s["table"], prompt)
        s["start"] = prompt[-2:].contiguous()
        s["context"] = s["start"].clone()
        s["filler"] = [f.contiguous() for f in _zipf(STEPS * 4 * 128, vocab, g).to(torch.int32).view(STEPS, -1)]
    if op == "mcts":
        s["u"] = list(torch.rand((STEPS, case["iterations"] * case["length"]), device="cuda", generator=g).unbind(0))
    if op == "host_step":
        s["filler"] = [f.cpu().pin_memory() for f in s["filler"]]
        s["tokens"], s["accepted"] = torch.zeros(rows, dtype=torch.int32).pin_memory(), torch.zeros(1, dtype=torch.int32).pin_memory()
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------
def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "draft":
        ctx = s["contexts"][s["turn"] % len(s["contexts"])]
        s["turn"] += 1
        B.aded_draft_tree(s["table"], ctx, case["nodes"], case["depth"], case["k"], s["filler"], *s["out"])
        return s["out"]
    if op in ("build", "lookup"):
        if op == "build":
            B.aded_trigram_clear(s["table"])
            B.aded_trigram_update(s["table"], s["corpus"])
        B.aded_trigram_topk(s["table"], s["contexts"], case["k"], *s["out"])
        return s["out"]

    model, kv = s["model"], s["kv"]
    if op == "prefill":
        n = case["context"]
        B.aded_kv_set_len(kv, 0, 0)         # a new request on this cache
        for at in range(0, n, 128):
            B.aded_append(model, kv, s["prompt"][at:min(n, at + 128)])
        return [t for layer in range(case["layers"]) for t in B.aded_kv_read(kv, 0, layer, 0, n)]

    at = s["turn"] % STEPS
    if s["turn"] and at == 0:               # the request is done: the next one with the same prompt
        for b, n in enumerate(s["lens"]):
            B.aded_kv_set_len(kv, b, n)
        if "context" in s:
            s["context"].copy_(s["start"])
    s["turn"] += 1
    B.aded_debug_capture(model, s.get("logits"), s["best"])
    if op == "decode":
        B.aded_decode_step(model, kv, s["table"], s["context"], case["nodes"], case["depth"], case["k"], s["filler"][at], s["tokens"].view(-1), s["accepted"])
    elif op == "host_step":
        B.aded_decode_step_host(model, kv, s["table"], s["context"], case["nodes"], case["depth"], case["k"], s["filler"][at], s["tokens"], s["accepted"])
    elif op == "mcts":
        B.aded_decode_step_mcts(model, kv, s["table"], s["context"], case["nodes"], case["iterations"], case["length"], case["candidates"], case["k"],
                                s["u"][at], s["filler"][at], s["tokens"].view(-1), s["accepted"])
    elif op == "sampled":
        B.aded_verify_sampled(model, kv, *s["tree"], 0.7, 0.95, s["u"], s["tokens"].view(-1), s["accepted"])
    elif case["batch"] == 1:
        B.aded_verify(model, kv, *s["tree"], s["tokens"].view(-1), s["accepted"])
    else:
        B.aded_verify_batch(model, kv, s["offsets"], *s["tree"], s["tokens"], s["accepted"])
    hidden = B.aded_debug_read_buffer(model, 1, s["rows"])
    out = [s["tokens"], s["accepted"], s["best"], hidden]
    return out + [s["logits"]] if "logits" in s else out


# ---- what a pass cannot do without, and how close two correct passes are ---------------------------------------------------
def work(case):
    op = case["op"]
    if op == "draft":                       # contexts of the inner nodes: a bucket each; the tree
        return {"bytes": 64.0 * (1 + case["nodes"] // case["k"]) + 8.0 * case["nodes"], "flops": 0.0}
    if op in ("build", "lookup"):           # contexts and lists; a context's bucket; when building: the text, and a table entry per window
        q, k = case["queries"], case["k"]
        return {"bytes": q * (8.0 + 8.0 * k + 4.0 + 64.0) + (case["corpus"] * (4.0 + 8.0) if op == "build" else 0.0), "flops": 0.0}
    shape = SHAPES[case["shape"]].with_layers(case["layers"])
    el = 4.0 if shape.dtype == "f32" else 2.0
    d, n_layers, context = shape.d_model, shape.n_layers, case["context"]
    if op == "prefill":                     # every call of 128 tokens reads the weights and the keys/values so far; the cache is read back once
        calls = (context + 127) // 128
        past = sum(range(0, context, 128))
        attended = context * (context + 1) / 2
        return {"bytes": calls * n_layers * shape.params_per_layer * el + (past + 3 * context) * shape.kv_bytes_per_position(),
                "flops": 2.0 * context * n_layers * shape.params_per_layer + 4.0 * attended * d * n_layers}
    lens, nodes = _ragged(case)
    rows, cached = sum(nodes), sum(lens)
    flops = 2.0 * rows * (n_layers * shape.params_per_layer + shape.vocab * d) + 4.0 * sum(a * b for a, b in zip(lens, nodes)) * d * n_layers
    bytes_ = shape.weight_bytes_per_step + (cached + rows) * shape.kv_bytes_per_position() + rows * d * el
    if op == "sampled" or shape.dtype == "f32":
        bytes_ += rows * shape.vocab * 4.0
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Counts, lists and trees are whole numbers and exact.  The tokens of a model case are exact too: the margin between the
    best two logits is far above any rounding.  Hidden states, logits and cache rows of bf16 models: the bf16 attention kernels
    of the library, which add the same products in another order, differ by 5e-4 after one layer, 8e-3 after 8 and 1.7e-2
    after 32 (largest difference 1e-2, 5e-2, 1e-1); about four times that, as far as 3e-2."""
    if case["op"] in ("draft", "build", "lookup"):
        return "exact"
    if SHAPES[case["shape"]].dtype == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": min(3e-2, 4e-3 * case["layers"]), "max": min(0.4, 0.05 * case["layers"])}
