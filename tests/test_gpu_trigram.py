"""GPU parity of the tri-gram store against the CPU checker: counts and top-k lists bit-exact."""
import numpy as np
import pytest
import torch

from oracle.trigram import TrigramStore
from paper_2407_12021_b200 import inputs as gen

pytestmark = pytest.mark.gpu


def _topk_gpu(B, t, ctx, k):
    q = len(ctx)
    c = torch.tensor(ctx, dtype=torch.int32, device="cuda").reshape(q, 2)
    tok = torch.empty((q, k), dtype=torch.int32, device="cuda")
    cnt = torch.empty((q, k), dtype=torch.int32, device="cuda")
    tot = torch.empty((q,), dtype=torch.int32, device="cuda")
    B.aded_trigram_topk(t, c, k, tok, cnt, tot)
    torch.cuda.synchronize()
    return tok.tolist(), cnt.tolist(), tot.tolist()


def _check_against(B, t, st: TrigramStore, contexts, ks=(1, 4, 32)):
    for k in ks:
        tok, cnt, tot = _topk_gpu(B, t, contexts, k)
        for i, (a, b) in enumerate(contexts):
            wt, wc = st.topk(a, b, k)
            assert tok[i] == wt and cnt[i] == wc, (a, b, k, tok[i], wt, cnt[i], wc)
            assert tot[i] == st.total(a, b)


def test_c1_table_from_10k_zipf_corpus(cuda_device):
    """Workload 1's table: 10k-token Zipf(1.1) corpus over a 4096-token vocabulary, k = 4."""
    from paper_2407_12021_b200 import binding as B
    toks = gen.zipf_tokens(10000, 4096, 31, 1)
    st = TrigramStore()
    st.update(toks.tolist())
    t = B.aded_trigram_create(4096, log2_buckets=14, overflow_buckets=4096)
    B.aded_trigram_update(t, toks.cuda())
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(t) == 0
    entries, buckets = B.aded_trigram_stats(t)
    assert entries == len(st.entries())
    assert buckets >= len(st.table)
    # every stored tri-gram, bit-exact
    for (a, b, c), n in list(st.entries().items())[::7]:
        assert B.aded_trigram_get(t, a, b, c) == n
    assert B.aded_trigram_get(t, 4095, 4095, 4095) == 0
    ctxs = list(st.table.keys())
    ctxs.sort(key=lambda ab: -len(st.table[ab]))
    contexts = ctxs[:300] + ctxs[-200:] + [(4095, 4094), (7, 4000)]
    _check_against(B, t, st, contexts)


def test_incremental_updates_match_stepwise(cuda_device):
    """The per-step pattern: every step passes [two previous tokens] ++ [new tokens]."""
    from paper_2407_12021_b200 import binding as B
    stream = gen.zipf_tokens(3000, 50, 32, 1).tolist()     # tiny vocabulary: long chains, many duplicates
    st = TrigramStore()
    t = B.aded_trigram_create(50, log2_buckets=12, overflow_buckets=2048)
    pos = 2
    lens = gen.randint(2000, 9, 32, 2)
    i = 0
    while pos < len(stream):
        n = 1 + lens[i]; i += 1
        span = stream[pos - 2:pos + n]
        st.update(span)
        B.aded_trigram_update_host(t, torch.tensor(span, dtype=torch.int32))
        pos += n
    assert B.aded_trigram_poll_status(t) == 0
    whole = TrigramStore()
    whole.update(stream)
    assert whole.entries() == st.entries()
    assert B.aded_trigram_stats(t)[0] == len(st.entries())
    _check_against(B, t, st, list(st.table.keys())[:400])


def test_duplicates_in_one_call_saturation_and_short_spans(cuda_device):
    from paper_2407_12021_b200 import binding as B
    t = B.aded_trigram_create(10, log2_buckets=4, overflow_buckets=64, cap=5)
    st = TrigramStore(cap=5)
    span = [3] * 40 + [1, 2] * 30
    st.update(span)
    B.aded_trigram_update(t, torch.tensor(span, dtype=torch.int32, device="cuda"))
    for n in (0, 1, 2):
        B.aded_trigram_update(t, torch.tensor(span[:n], dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert B.aded_trigram_get(t, 3, 3, 3) == 5 == st.count(3, 3, 3)
    assert B.aded_trigram_get(t, 1, 2, 1) == 5
    assert B.aded_trigram_get(t, 3, 3, 1) == 1
    _check_against(B, t, st, [(3, 3), (1, 2), (2, 1), (3, 1), (9, 9)], ks=(1, 3))


def test_min_count_filter_and_errors(cuda_device):
    from paper_2407_12021_b200 import binding as B
    t = B.aded_trigram_create(100, log2_buckets=6, overflow_buckets=8, min_count=2)
    st = TrigramStore()
    span = [1, 1, 9, 1, 1, 3, 1, 1, 7, 1, 1, 7]
    st.update(span)
    B.aded_trigram_update(t, torch.tensor(span, dtype=torch.int32, device="cuda"))
    tok, cnt, tot = _topk_gpu(B, t, [(1, 1)], 4)
    assert (tok[0], cnt[0]) == st.topk(1, 1, 4, min_count=2) and tot[0] == st.total(1, 1)
    # an out-of-vocabulary token is reported, not counted
    B.aded_trigram_update(t, torch.tensor([1, 2, 100], dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(t) == 1
    assert B.aded_trigram_poll_status(t) == 0
    # table full: 64 home buckets cannot hold 90 distinct contexts
    full = B.aded_trigram_create(100, log2_buckets=4, overflow_buckets=0)
    B.aded_trigram_update(full, torch.arange(0, 92, dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(full) == 4


def test_large_table_bulk_update_and_queries(cuda_device):
    """10^6 Zipf tokens over a 32000-token vocabulary; sampled contexts against the checker."""
    from paper_2407_12021_b200 import binding as B
    toks = gen.zipf_tokens(1_000_000, 32000, 33, 1)
    st = TrigramStore()
    st.update(toks.tolist())
    t = B.aded_trigram_create(32000, log2_buckets=21, overflow_buckets=1 << 18)
    B.aded_trigram_update(t, toks.cuda())
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(t) == 0
    assert B.aded_trigram_stats(t)[0] == len(st.entries())
    ctxs = list(st.table.keys())
    ctxs.sort(key=lambda ab: -len(st.table[ab]))
    sample = ctxs[:64] + ctxs[1000::997][:400]
    _check_against(B, t, st, sample, ks=(4,))


def _entries_gpu(B, t, min_count=0):
    keys, counts = B.aded_trigram_export(t, min_count)
    torch.cuda.synchronize()
    k, c = keys.cpu().tolist(), counts.cpu().tolist()
    out = {tuple(kk): cc for kk, cc in zip(k, c)}
    assert len(out) == len(k), "an entry was exported twice"
    return out


def test_export_prune_save_load(cuda_device, tmp_path):
    """Table persistence and the elimination threshold: exported entries, the pruned table and a table
    read back from a file equal the checker's, bit for bit; the pruned table keeps working."""
    from paper_2407_12021_b200 import binding as B
    vocab = 60
    toks = gen.zipf_tokens(6000, vocab, 41, 1)
    st = TrigramStore(cap=50)
    st.update(toks.tolist())
    t = B.aded_trigram_create(vocab, log2_buckets=12, overflow_buckets=4096, cap=50)
    B.aded_trigram_update(t, toks.cuda())
    assert _entries_gpu(B, t) == st.entries()
    assert _entries_gpu(B, t, 12) == {k: n for k, n in st.entries().items() if n >= 12}
    path = str(tmp_path / "table.bin")
    B.aded_trigram_save(t, path)
    # a copy read from the file
    t2 = B.aded_trigram_create(vocab, log2_buckets=13, overflow_buckets=8192, cap=50)   # another geometry than the source
    B.aded_trigram_load(t2, path)
    assert _entries_gpu(B, t2) == st.entries()
    # loading again adds the counts (saturating)
    B.aded_trigram_load(t2, path)
    twice = TrigramStore(cap=50)
    twice.merge(st.entries())
    twice.merge(st.entries())
    assert _entries_gpu(B, t2) == twice.entries()
    # a file for another vocabulary is refused
    from paper_2407_12021_b200.binding import AdedError
    t3 = B.aded_trigram_create(vocab + 1, log2_buckets=10, overflow_buckets=64)
    with pytest.raises(AdedError):
        B.aded_trigram_load(t3, path)
    with pytest.raises(AdedError):
        B.aded_trigram_load(t2, str(tmp_path / "missing.bin"))
    # elimination threshold 12 (the paper's setting): the table is rebuilt from what stays
    _, buckets_before = B.aded_trigram_stats(t)
    B.aded_trigram_prune(t, 12)
    st.prune(12)
    assert _entries_gpu(B, t) == st.entries()
    entries_after, buckets_after = B.aded_trigram_stats(t)
    assert entries_after == len(st.entries()) and buckets_after < buckets_before
    ctxs = list(st.table.keys())[:200] + [(vocab - 1, vocab - 1)]
    _check_against(B, t, st, ctxs, ks=(1, 4))
    # and keeps counting: no duplicate entries appear where pruned ones used to be
    more = gen.zipf_tokens(3000, vocab, 42, 1)
    B.aded_trigram_update(t, more.cuda())
    st.update(more.tolist())
    assert _entries_gpu(B, t) == st.entries()
    B.aded_trigram_clear(t)
    assert _entries_gpu(B, t) == {} and B.aded_trigram_stats(t) == (0, 0)
    assert B.aded_trigram_poll_status(t) == 0 and B.aded_trigram_poll_status(t2) == 0


def test_import_of_duplicate_entries_with_large_counts_saturates(cuda_device):
    """Imported counts may be large and one tri-gram may appear several times in an import: the stored count
    is min(sum, cap) as in the checker's merge, never a wrapped 32-bit sum.  The default cap is 2^31 - 1;
    a cap above it is refused."""
    from paper_2407_12021_b200 import binding as B
    big = 2 ** 31 - 2
    keys, counts, entries = [], [], []
    for i in range(64):                       # 64 tri-grams, each four times in one import, counts near 2^31
        for rep in range(4):
            keys.append([i % 7, i % 5, i])
            counts.append(big - rep)
            entries.append(((i % 7, i % 5, i), big - rep))
    for cap in (0, 1000, 2 ** 31 - 1):
        t = B.aded_trigram_create(100, log2_buckets=8, overflow_buckets=64, cap=cap)
        st = TrigramStore(cap=cap if cap else 2 ** 31 - 1)
        st.update([1, 2, 3, 1, 2, 3])          # an entry that is there before the import
        B.aded_trigram_update(t, torch.tensor([1, 2, 3, 1, 2, 3], dtype=torch.int32, device=cuda_device))
        kt = torch.tensor(keys + [[1, 2, 3]], dtype=torch.int32, device=cuda_device)
        ct = torch.tensor([c - 2 ** 32 if c >= 2 ** 31 else c for c in counts + [big]], dtype=torch.int32, device=cuda_device)
        B.aded_trigram_import(t, kt, ct)
        for key, n in entries + [((1, 2, 3), big)]:
            st.merge({key: n})
        torch.cuda.synchronize()
        assert B.aded_trigram_poll_status(t) == 0
        for i in range(64):
            assert B.aded_trigram_get(t, i % 7, i % 5, i) == st.count(i % 7, i % 5, i) == st.cap
        assert B.aded_trigram_get(t, 1, 2, 3) == st.count(1, 2, 3) == st.cap
        assert B.aded_trigram_get(t, 2, 3, 1) == st.count(2, 3, 1) == 1
    with pytest.raises(B.AdedError) as err:
        B.aded_trigram_create(100, log2_buckets=8, overflow_buckets=64, cap=2 ** 31)
    assert err.value.status == 1


def _star(n, vocab=20000):
    """A span in which the context (1, 2) has n continuations, first seen in the order of their ids, and a third of them twice."""
    ids = [3 + i for i in range(n)] + [3 + i for i in range(0, n, 3)]
    return [t for i in ids for t in (1, 2, i)]


@pytest.mark.parametrize("n", [5, 6, 7, 12, 13, 24, 25, 47, 48, 49, 1536, 1537, 2054, 2055, 6150, 6151])
def test_contexts_at_the_ends_of_extents(cuda_device, n):
    """Continuations beyond six lie in extents of 6, 12, 24, ... entries: one context just below, at and above their ends (and
    above the length from which a whole block scans it), asked for many times in one call beside others."""
    from paper_2407_12021_b200 import binding as B
    span = _star(n)
    st = TrigramStore()
    st.update(span)
    t = B.aded_trigram_create(20000, log2_buckets=16, overflow_buckets=4096)
    B.aded_trigram_update(t, torch.tensor(span, dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(t) == 0
    assert B.aded_trigram_stats(t) == (len(st.entries()), len(st.table) + sum((len(v) - 1) // 6 for v in st.table.values() if len(v) > 6))
    assert _entries_gpu(B, t) == st.entries()
    for c in (3, 2 + n, 3 + n, 3 + n // 2):
        assert B.aded_trigram_get(t, 1, 2, c) == st.count(1, 2, c)
    contexts = ([(1, 2), (2, 3), (19999, 1), (3, 1)] * 40)[:157]
    _check_against(B, t, st, contexts, ks=(1, 8, 9, 32))
    _check_against(B, t, st, contexts[:1], ks=(3,))


@pytest.mark.parametrize("n", [7, 12, 13, 18, 19, 43])
def test_configured_overflow_is_the_limit(cuda_device, n):
    """Entries beyond six count in units of six against overflow_buckets: exactly enough is enough, one fewer is a full table,
    which keeps what it holds, goes on counting it and refuses new entries again after the status was read."""
    from paper_2407_12021_b200 import binding as B
    need = (n - 6 + 5) // 6
    rows = [[1, 2, 3 + i] for i in range(n)]

    def update(t, row):
        B.aded_trigram_update(t, torch.tensor(row, dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        return B.aded_trigram_poll_status(t)

    t = B.aded_trigram_create(100, log2_buckets=8, overflow_buckets=need)
    assert [update(t, r) for r in rows] == [0] * n
    t = B.aded_trigram_create(100, log2_buckets=8, overflow_buckets=need - 1)
    fits = 6 * need
    assert [update(t, r) for r in rows] == [0] * fits + [4] * (n - fits)
    assert [update(t, r) for r in rows] == [0] * fits + [4] * (n - fits)
    assert _entries_gpu(B, t) == {tuple(r): 2 for r in rows[:fits]}
    assert B.aded_trigram_stats(t)[0] == fits
    # the same at once: whatever is kept is counted right
    t = B.aded_trigram_create(100, log2_buckets=8, overflow_buckets=need - 1)
    assert update(t, [x for r in rows for x in r]) == 4
    kept = _entries_gpu(B, t)
    assert all(kept[k] == 1 for k in kept) and B.aded_trigram_stats(t)[0] == len(kept)
    B.aded_trigram_clear(t)
    assert update(t, rows[0]) == 0 and _entries_gpu(B, t) == {tuple(rows[0]): 1}


@pytest.mark.parametrize("limit", [0, 1, 2, 5, 9, 10, 64, 300])
def test_many_entries_at_once_fill_the_table_to_its_limit(cuda_device, limit):
    """Contexts that grow by hundreds of entries in one call when there are fewer units than they ask for: every unit is given out and
    filled, the rest is refused and reported, what is kept is counted right, nothing else is touched -- the staging of the
    host entry points lies behind the pool -- and a table at its limit goes on counting what it holds."""
    from paper_2407_12021_b200 import binding as B
    vocab, contexts, each = 5000, 6, 400
    t = B.aded_trigram_create(vocab, log2_buckets=12, overflow_buckets=limit)
    rows = [[a, 100 + a, 200 + i * 7 % 3001] for i in range(each) for a in range(contexts)]
    for _ in range(3):
        B.aded_trigram_clear(t)
        for part in (rows[:6 * contexts], rows * 2):        # (six of every context are in its home bucket)
            B.aded_trigram_import(t, torch.tensor(part, dtype=torch.int32, device="cuda"), torch.ones(len(part), dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        kept = _entries_gpu(B, t)
        assert B.aded_trigram_poll_status(t) == 4
        assert set(kept) <= {tuple(r) for r in rows} and all(1 <= n <= 3 for n in kept.values())
        beyond = [sum(k[0] == a for k in kept) - 6 for a in range(contexts)]
        assert all(n >= 0 for n in beyond) and sum((n + 5) // 6 for n in beyond) == limit
        entries, buckets = B.aded_trigram_stats(t)
        assert (entries, buckets) == (len(kept), contexts + limit)
        held = list(kept)[:40]
        assert all(B.aded_trigram_get(t, *r) == kept[r] for r in held)
        # what the table holds is counted on; the staging buffers of the host calls are what they say
        for r in held:
            B.aded_trigram_update_host(t, torch.tensor(r, dtype=torch.int32))
        assert B.aded_trigram_poll_status(t) == 0
        assert all(B.aded_trigram_get(t, *r) == kept[r] + 1 for r in held)
        after = _entries_gpu(B, t)
        assert after == {r: n + (r in held) for r, n in kept.items()}
        st = TrigramStore()
        st.merge(after)
        ctx = [(a, 100 + a) for a in range(contexts)] + [(1, 2)]
        tok, cnt = torch.empty((7, 8), dtype=torch.int32), torch.empty((7, 8), dtype=torch.int32)
        B.aded_trigram_topk_host(t, torch.tensor(ctx, dtype=torch.int32), 8, tok, cnt)
        assert [(tok[i].tolist(), cnt[i].tolist()) for i in range(7)] == [st.topk(a, b, 8) for a, b in ctx]


def test_repeated_and_absent_contexts_in_one_call(cuda_device):
    """Blocks answer a context once for all queries that ask for it: more queries than one block takes, every context many
    times, several long ones per block, absent and out-of-range contexts between them."""
    from paper_2407_12021_b200 import binding as B
    spans = [1, 2, 3] * 5
    for a in range(7):                          # seven contexts of 2500 continuations
        spans += [t for i in range(2500) for t in (a, 10 + a, 100 + (i * 7 + a) % 4000)]
    st = TrigramStore()
    st.update(spans)
    t = B.aded_trigram_create(5000, log2_buckets=16, overflow_buckets=1 << 14)
    B.aded_trigram_update(t, torch.tensor(spans, dtype=torch.int32, device="cuda"))
    base = [(a, 10 + a) for a in range(7)] + [(1, 2), (2, 3), (4999, 4999), (-1, 3), (5000, 1), (10, 100)]
    for q in (len(base), 1000, 40000):
        contexts = (base * (q // len(base) + 1))[:q]
        for k in (2, 12):
            tok, cnt, tot = _topk_gpu(B, t, contexts, k)
            want = {c: (st.topk(*c, k), st.total(*c)) for c in base}
            for i, c in enumerate(contexts):
                assert ((tok[i], cnt[i]), tot[i]) == want[c], (q, k, i, c)


def test_more_lookups_than_the_blocks_hold_in_ordinary_shared_memory(cuda_device):
    """One continuation each for so many contexts that a block's share needs more than 48 KB of shared memory."""
    from paper_2407_12021_b200 import binding as B
    toks = gen.zipf_tokens(20000, 300, 81, 1)
    st = TrigramStore()
    st.update(toks.tolist())
    t = B.aded_trigram_create(300, log2_buckets=16, overflow_buckets=1 << 13)
    B.aded_trigram_update(t, toks.cuda())
    keys = list(st.table.keys())[:3000] + [(299, 299), (-1, 3)]
    want = [st.topk(a, b, 1) + (st.total(a, b),) for a, b in keys]
    q = 1_500_000
    at = torch.arange(q, device="cuda") % len(keys)
    ctx = torch.tensor(keys, dtype=torch.int32, device="cuda")[at].contiguous()
    tok, cnt = torch.empty((q, 1), dtype=torch.int32, device="cuda"), torch.empty((q, 1), dtype=torch.int32, device="cuda")
    tot = torch.empty(q, dtype=torch.int32, device="cuda")
    B.aded_trigram_topk(t, ctx, 1, tok, cnt, tot)
    for got, i in ((tok.view(-1), 0), (cnt.view(-1), 1), (tot, 2)):
        assert torch.equal(got, torch.tensor([w[i][0] if i < 2 else w[i] for w in want], dtype=torch.int32, device="cuda")[at])


@pytest.mark.parametrize("windows", [(1 << 17) - 1, 1 << 17, (1 << 17) + 1, (1 << 17) + 2047])
def test_long_spans_on_both_sides_of_the_bulk_update(cuda_device, windows):
    """Spans of 2^17 windows on are added up per block first: the counts at the line, with a ragged last block, with a cap that many
    blocks reach together, and with a token outside the vocabulary (reported; windows with it, and those that come up after the
    report, are not counted)."""
    from paper_2407_12021_b200 import binding as B
    toks = gen.zipf_tokens(windows + 2, 300, 51, 1)
    for cap in (0, 7):
        st = TrigramStore(cap=cap) if cap else TrigramStore()
        t = B.aded_trigram_create(300, log2_buckets=17, overflow_buckets=1 << 16, cap=cap)
        for _ in range(2):
            st.update(toks.tolist())
            B.aded_trigram_update(t, toks.cuda())
        torch.cuda.synchronize()
        assert B.aded_trigram_poll_status(t) == 0
        assert _entries_gpu(B, t) == st.entries()
    bad = toks.clone()
    bad[windows // 2] = 300
    t = B.aded_trigram_create(300, log2_buckets=17, overflow_buckets=1 << 16)
    B.aded_trigram_update(t, bad.cuda())
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(t) == 1
    st = TrigramStore()
    st.update(bad.tolist())
    most = st.entries()
    assert all(max(k) < 300 and n <= most[k] for k, n in _entries_gpu(B, t).items())
    B.aded_trigram_clear(t)                                # once it has been read, the table counts again
    B.aded_trigram_update(t, toks.cuda())
    st = TrigramStore()
    st.update(toks.tolist())
    assert _entries_gpu(B, t) == st.entries() and B.aded_trigram_poll_status(t) == 0


@pytest.mark.parametrize("q", [(1 << 16) - 1, 1 << 16, (1 << 16) + 1, 150001])
def test_lookups_on_both_sides_of_the_grouped_path(cuda_device, q):
    """From 2^16 queries on a context is scanned once per call, with the output arrays as scratch: contexts all in the home bucket,
    beyond it, long ones, absent ones; each asked for by one and by many queries; with and without the sums."""
    from paper_2407_12021_b200 import binding as B
    spans = gen.zipf_tokens(30000, 400, 61, 1).tolist()
    for a in range(18):                         # more long contexts than a block scans together
        spans += [t for i in range(2100) for t in (a, 400 + a, 450 + (i * 7 + a) % 3000)]
    st = TrigramStore()
    st.update(spans)
    t = B.aded_trigram_create(5000, log2_buckets=17, overflow_buckets=1 << 15)
    B.aded_trigram_update(t, torch.tensor(spans, dtype=torch.int32, device="cuda"))
    keys = list(st.table.keys())
    rare = keys[::3][:4000]
    pool = [(a, 400 + a) for a in range(18)] + keys[:50] + [(4999, 4999), (-1, 3), (5000, 1), (7, -2)]
    contexts = (rare + pool * (q // len(pool) + 1))[:q]
    for k in (1, 2, 3, 8, 9):
        tok, cnt, tot = _topk_gpu(B, t, contexts, k)
        want = {c: (st.topk(*c, k), st.total(*c)) for c in set(contexts)}
        bad = [(i, c) for i, c in enumerate(contexts) if ((tok[i], cnt[i]), tot[i]) != want[c]]
        assert not bad, (q, k, bad[:3])
    c = torch.tensor(contexts, dtype=torch.int32, device="cuda")
    out_t, out_c = torch.empty((q, 4), dtype=torch.int32, device="cuda"), torch.empty((q, 4), dtype=torch.int32, device="cuda")
    B.aded_trigram_topk(t, c, 4, out_t, out_c, None)
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(t) == 0
    got = list(zip(out_t.tolist(), out_c.tolist()))
    assert all(got[i] == st.topk(*contexts[i], 4) for i in range(0, q, 97))


def test_table_without_room_for_pool_and_index(cuda_device, tmp_path):
    """Where the device has no room for the pool and its index (272-400 bytes per overflow bucket) a table is made of chains of buckets
    (64 bytes): every operation gives what it gives on an ordinary table."""
    from paper_2407_12021_b200 import binding as B
    vocab = 5000
    text = gen.zipf_tokens(200_000, vocab, 71, 1).tolist()
    text += [t for i in range(2500) for t in (3, 4, 100 + i)] + [t for i in range(0, 2500, 2) for t in (3, 4, 100 + i)]
    toks = torch.tensor(text, dtype=torch.int32, device="cuda")
    torch.cuda.empty_cache()
    full = B.aded_trigram_create(vocab, log2_buckets=18, overflow_buckets=1 << 17)
    B.aded_trigram_update(full, toks[:3])                  # (kernels are loaded before the room is taken)
    B.aded_trigram_clear(full)
    torch.cuda.synchronize()
    taken = torch.empty(torch.cuda.mem_get_info()[0] - (600 << 20), dtype=torch.uint8, device="cuda")
    before = torch.cuda.mem_get_info()[0]
    tight = B.aded_trigram_create(vocab, log2_buckets=18, overflow_buckets=3_000_000)      # 0.2 GB; 1 GB otherwise
    assert before - torch.cuda.mem_get_info()[0] < 300 << 20
    del taken
    torch.cuda.empty_cache()
    tables, answers = (full, tight), []
    keys = list(zip(text[0:4000:2], text[1:4000:2]))
    pool = [(3, 4), (1, 1), (vocab - 1, vocab - 1), (-1, 3)] + keys
    contexts = (pool * (70_000 // len(pool) + 1))[:70_000]
    filler = gen.zipf_tokens(512, vocab, 72, 1).cuda()
    u = torch.tensor(gen.uniform01(600, 73, 1).numpy().astype(np.float32), device="cuda")
    for t in tables:
        got = []
        B.aded_trigram_update(t, toks)                     # a long span, then short ones
        B.aded_trigram_update(t, toks[:5000])
        B.aded_trigram_update_host(t, toks[5000:5200].cpu())
        got.append(sorted(_entries_gpu(B, t).items()))
        got.append(B.aded_trigram_stats(t))
        got += [B.aded_trigram_get(t, 3, 4, c) for c in (100, 101, 2599, 2600)]
        got += [_topk_gpu(B, t, contexts[:q], k) for q, k in ((300, 1), (300, 9), (300, 32), (70_000, 1), (70_000, 4))]
        for ctx in ((3, 4), keys[5], (vocab - 1, vocab - 1)):
            tree = [torch.zeros(m, dtype=torch.int32, device="cuda") for m in (64, 64, 1)]
            B.aded_draft_tree(t, torch.tensor(ctx, dtype=torch.int32, device="cuda"), 64, 6, 8, filler, *tree)
            got += [x.tolist() for x in tree]
            got.append(B.aded_mcts_draft(t, torch.tensor(ctx, dtype=torch.int32, device="cuda"), 150, 4, 24, 8, u))
        B.aded_trigram_save(t, str(tmp_path / "table.bin"))
        B.aded_trigram_prune(t, 2)
        got.append(sorted(_entries_gpu(B, t).items()))
        B.aded_trigram_load(t, str(tmp_path / "table.bin"))
        got.append(sorted(_entries_gpu(B, t).items()))
        got.append(B.aded_trigram_stats(t))
        B.aded_trigram_clear(t)
        got += [B.aded_trigram_stats(t), B.aded_trigram_poll_status(t)]
        answers.append(got)
    assert len(answers[0]) == len(answers[1])
    assert all(a == b for a, b in zip(*answers)), [i for i, (a, b) in enumerate(zip(*answers)) if a != b]
    st = TrigramStore()
    for span in (text, text[:5000], text[5000:5200]):
        st.update(span)
    assert dict(answers[1][0]) == st.entries() and answers[1][-1] == 0


@pytest.mark.parametrize("entries", [518, 519, 600, 2600])
def test_export_with_more_long_contexts_than_a_block_shares(cuda_device, entries):
    """Contexts of more than 512 entries beyond their home bucket are exported by all warps of a block, up to 64 of them per block; here
    two blocks hold 200, just below, at and above the line and over several rounds."""
    from paper_2407_12021_b200 import binding as B
    a = torch.arange(200, device="cuda").repeat_interleave(entries)
    c = torch.arange(entries, device="cuda").repeat(200)
    rows = torch.stack([a, a + 1000, (c * 7 + a) % 4999], dim=1).to(torch.int32).contiguous()
    counts = (1 + c % 3).to(torch.int32)
    t = B.aded_trigram_create(5000, log2_buckets=9, overflow_buckets=200 * ((entries + 5) // 6))
    B.aded_trigram_import(t, rows, counts)
    torch.cuda.synchronize()
    assert B.aded_trigram_poll_status(t) == 0

    def packed(r):
        return ((r[:, 0].long() * 5000 + r[:, 1].long()) * 5000 + r[:, 2].long())

    for least in (0, 2, 4):
        keys, got = B.aded_trigram_export(t, least)
        want = packed(rows)[counts >= least] * 4 + counts[counts >= least]
        assert torch.equal((packed(keys) * 4 + got).sort().values, want.sort().values)


@pytest.mark.parametrize("k,offset", [(2, 0), (2, 1), (3, 0), (4, 0), (4, 1), (4, 2), (6, 0), (8, 0), (12, 0), (32, 0)])
def test_grouped_lookups_of_a_large_table(cuda_device, k, offset):
    """Tables of much text group from 4096 queries on.  Rows that are answered in the first kernel and rows whose counts its hash
    table takes, contexts of every size on both sides of what a thread, a warp and a block look up, repeated within and across the first
    kernel's blocks, absent and invalid ones, rows of one, two and four words per store: all as the same lookups in small calls."""
    from paper_2407_12021_b200 import binding as B
    vocab = 3000
    t = B.aded_trigram_create(vocab, log2_buckets=21, overflow_buckets=1 << 16)
    sizes = [1, 5, 6, 7, 8, 12, 13, 18, 19, 30, 31, 53, 54, 55, 60, 200, 2053, 2054, 2055, 2600]
    for i, n in enumerate(sizes):                          # context (2900 + i, i): n continuations, some of them twice
        span = [tok for c in range(n) for tok in (2900 + i, i, (c * 7 + i) % vocab)] + [tok for c in range(0, n, 3) for tok in (2900 + i, i, (c * 7 + i) % vocab)]
        B.aded_trigram_update(t, torch.tensor(span, dtype=torch.int32, device="cuda"))
    B.aded_trigram_update(t, gen.zipf_tokens(20000, 300, 71, 1).cuda())
    launched = B.aded_launch_count()
    B.aded_trigram_topk(t, torch.zeros((4096, 2), dtype=torch.int32, device="cuda"), k, *(torch.zeros((4096, k), dtype=torch.int32, device="cuda") for _ in range(2)))
    assert B.aded_launch_count() - launched == 1           # little text: one kernel
    B.aded_trigram_update(t, torch.full((600_000,), 299, dtype=torch.int32, device="cuda"))
    g = torch.Generator().manual_seed(72)
    for q in (4096, 5001):
        ctx = torch.stack([gen.zipf_tokens(q, 300, 73, 1), gen.zipf_tokens(q, 300, 74, 1)], dim=1)
        pick = torch.randint(0, 4 * len(sizes), (q,), generator=g)
        for i in range(len(sizes)):
            ctx[pick == i] = torch.tensor([2900 + i, i], dtype=ctx.dtype)
        ctx[::97] = torch.tensor([-1, 5], dtype=ctx.dtype)
        ctx[5::89] = torch.tensor([7, vocab], dtype=ctx.dtype)
        ctx = ctx.to(torch.int32).cuda().contiguous()

        def rows(n):
            flat = [torch.full((n * k + offset,), -5, dtype=torch.int32, device="cuda") for _ in range(2)]
            return [f[offset:].view(n, k) for f in flat] + [torch.full((n,), -5, dtype=torch.int32, device="cuda")]

        tok, cnt, total = rows(q)
        launched = B.aded_launch_count()
        B.aded_trigram_topk(t, ctx, k, tok, cnt, total)
        assert B.aded_launch_count() - launched == 3
        for a in range(0, q, 1000):
            part = ctx[a:a + 1000].contiguous()
            want = rows(part.shape[0])
            B.aded_trigram_topk(t, part, k, *want)
            for got, ref in zip((tok, cnt, total), want):
                assert torch.equal(got[a:a + 1000], ref), (q, a)
    assert B.aded_trigram_poll_status(t) == 0
