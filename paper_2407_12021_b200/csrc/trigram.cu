// Tri-gram store on the GPU (Eq. 1 counts, Algorithm 2 update, top-k continuation lookup).
//
// The table itself -- layout, insertion, lookup -- is in tg_store.cuh; here are the kernels over it and the entry points.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "aded_internal.cuh"
#include "tg_store.cuh"

namespace aded {

// Empty home buckets: one 16-byte part per thread and step (header, or two entries), so that a warp's stores are whole lines
// (a thread per bucket wrote 128 MB in 52 us; with the index, 192 MB: 77 us then, 43 now).  Index and counters are cleared by the same
// launch: for a small table every further operation on the stream costs as much as its clearing (22 us with two more, 17 now).
__global__ void k_tg_init(uint4* b, size_t parts, uint4* index, size_t index_parts, uint32_t* used) {
    const size_t first = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    if (first < 2) used[first] = 0;
    for (size_t i = first; i < parts; i += step)
        b[i] = (i & 3) == 0 ? make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0u, 0u) : make_uint4(0xFFFFFFFFu, 0u, 0xFFFFFFFFu, 0u);
    for (size_t i = first; i < index_parts; i += step) index[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Algorithm 2, one thread per window.  Duplicate windows inside one call are independent atomic
// adds, so the result is min(count + multiplicity, cap) whatever the thread order.
__device__ __forceinline__ void tg_add_window(const TgView& t, int a, int b, int c) {
    if (*t.status != 0) return;
    if (a < 0 || b < 0 || c < 0 || a >= t.vocab || b >= t.vocab || c >= t.vocab) {
        tg_report(t, (int)ADED_ERR_INVALID_ARG);
        return;
    }
    tg_add(t, a, b, c, 1u, true);
}
__global__ void k_tg_update(TgView t, const int32_t* __restrict__ tok, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x + 2;
    if (i < n) tg_add_window(t, tok[i - 2], tok[i - 1], tok[i]);
}

// The same for a long span: a block first adds up equal windows of its BULK_WINDOWS in a hash table in shared memory and then
// raises every distinct tri-gram once.  In text a few tri-grams are a large share of all windows (one in twenty of the
// synthetic text's), and a count takes one atomic add at a time.  Sums are the same whatever the order; no count can wrap, as the
// increments of a launch add up to fewer than 2^31.  `n` windows begin at tok[0].
// Measured, one thread per window against this (an empty table / one that holds the span already), us: 131,000 tokens 103 / 40
// against 91 / 41, 262,000 183 / 64 against 134 / 54, 10^6 417 / 255 against 309 / 145, 4 x 10^6 1369 / 1106 against 944 / 562:
// the line is at BULK_MIN; below, blocks of this size leave the device idle (20,000: 37 / 19 against 67 / 33).  What bounds it
// then is random access to the home buckets and the index (about 7 x 10^9 windows a second), and when filling the hand-overs of
// new entries.  Blocks of 512 threads and 1024 windows (when these took 287 / 139): 291 / 149 at 10^6.
constexpr int BULK_THREADS = 1024, BULK_WINDOWS = 2048, BULK_SLOTS = 4096, BULK_MIN = 1 << 17;
__global__ void __launch_bounds__(BULK_THREADS) k_tg_update_bulk(TgView t, const int32_t* __restrict__ tok, int n) {
    extern __shared__ int32_t bulk_smem[];
    int32_t* s_tok = bulk_smem;                               // [BULK_WINDOWS + 2]
    int32_t* s_first = s_tok + BULK_WINDOWS + 2;              // [BULK_SLOTS] window that stands for the slot's tri-gram, -1 empty
    int32_t* s_count = s_first + BULK_SLOTS;                  // [BULK_SLOTS]
    __shared__ int s_stop;
    if (threadIdx.x == 0) s_stop = *t.status != 0;
    __syncthreads();
    if (s_stop) return;
    const int w0 = blockIdx.x * BULK_WINDOWS, nw = min(BULK_WINDOWS, n - w0);
    for (int i = threadIdx.x; i < nw + 2; i += BULK_THREADS) s_tok[i] = tok[w0 + i];
    for (int i = threadIdx.x; i < BULK_SLOTS; i += BULK_THREADS) { s_first[i] = -1; s_count[i] = 0; }
    __syncthreads();
    for (int i = threadIdx.x; i < nw; i += BULK_THREADS) {
        const int a = s_tok[i], b = s_tok[i + 1], c = s_tok[i + 2];
        if (a < 0 || b < 0 || c < 0 || a >= t.vocab || b >= t.vocab || c >= t.vocab) {
            tg_report(t, (int)ADED_ERR_INVALID_ARG);
            continue;
        }
        int at = (int)(tg_hash(tg_key(a, b) * 31ull + (uint32_t)c) & (BULK_SLOTS - 1));
        for (;;) {                                            // (twice as many slots as windows: ends)
            const int have = atomicCAS(&s_first[at], -1, i);
            if (have == -1 || (s_tok[have] == a && s_tok[have + 1] == b && s_tok[have + 2] == c)) break;
            at = (at + 1) & (BULK_SLOTS - 1);
        }
        atomicAdd(&s_count[at], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < BULK_SLOTS; i += BULK_THREADS) {
        const int w = s_first[i];
        if (w >= 0) tg_add(t, s_tok[w], s_tok[w + 1], s_tok[w + 2], (uint32_t)s_count[i], true);
    }
}

// Every stored tri-gram with count >= min_count as (a, b, c) and its count, in no particular order;
// *n_out counts all of them, only the first `max_entries` are written.  A warp takes 32 home buckets at a time, a lane each,
// and then together the further entries of those that have any.  The places of N entries per lane are taken with one atomic, and
// their reads do not depend on one another, and contexts of more than EXPORT_LONG entries are left to all warps of the block: with one atomic
// per 32 entries and a warp per context the one with the most continuations -- 7254 of them in the text of 10^6 tokens -- was a chain
// of 227 round trips, and a full export of that table (two passes) 631 us instead of 187.
constexpr int EXPORT_THREADS = 256, EXPORT_BATCH = 8, EXPORT_MAX_LONG = 64;
constexpr uint32_t EXPORT_LONG = 512;
template <int N>
__device__ __forceinline__ void tg_export_some(unsigned long long key, const TgSlot (&s)[N], uint32_t min_count, int lane, int32_t* keys, uint32_t* counts,
                                               unsigned long long max_entries, unsigned long long* n_out) {
    unsigned m[N];
    int n = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        m[i] = __ballot_sync(0xffffffffu, s[i].tok >= 0 && s[i].cnt >= min_count && s[i].cnt != 0);
        n += __popc(m[i]);
    }
    if (n == 0) return;
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(n_out, (unsigned long long)n);
    at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const unsigned long long mine = at + __popc(m[i] & ((1u << lane) - 1u));
        if ((m[i] >> lane & 1u) && mine < max_entries) {
            keys[3 * mine + 0] = (int32_t)(key >> 32);
            keys[3 * mine + 1] = (int32_t)(key & 0xFFFFFFFFu);
            keys[3 * mine + 2] = s[i].tok;
            counts[mine] = s[i].cnt;
        }
        at += __popc(m[i]);
    }
}
// A context's entries beyond its home bucket, `parts` warps taking turns.
__device__ __forceinline__ void tg_export_extents(const TgView& t, const TgWalk& w, unsigned long long key, int part, int parts, uint32_t min_count, int lane,
                                                  int32_t* keys, uint32_t* counts, unsigned long long max_entries, unsigned long long* n_out) {
    for (uint32_t i0 = (uint32_t)part * 32 * EXPORT_BATCH; i0 < w.n; i0 += (uint32_t)parts * 32 * EXPORT_BATCH) {
        TgSlot s[EXPORT_BATCH];
#pragma unroll
        for (int j = 0; j < EXPORT_BATCH; ++j) {
            const uint32_t p = i0 + 32 * j + lane, m = p / TG_UNIT;
            const int x = tg_extent(m);
            const uint32_t base = __shfl_sync(0xffffffffu, w.extent, x & 31);
            s[j] = TgSlot{-1, 0u};
            if (p < w.n && base != 0) s[j] = t.pool[((size_t)(base - 1) + (m + 1 - (1u << x))) * TG_UNIT + p % TG_UNIT];
        }
        tg_export_some(key, s, min_count, lane, keys, counts, max_entries, n_out);
    }
}
__global__ void __launch_bounds__(EXPORT_THREADS) k_tg_export(TgView t, uint32_t min_count, int32_t* __restrict__ keys, uint32_t* __restrict__ counts,
                                                              unsigned long long max_entries, unsigned long long* n_out) {
    __shared__ uint32_t s_home[EXPORT_MAX_LONG];
    __shared__ int s_long;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    if (threadIdx.x == 0) s_long = 0;
    __syncthreads();
    for (uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < (t.n_home + 31) / 32; g += warps) {
        const uint32_t mine = g * 32 + lane;
        const uint4 head = mine < t.n_home ? *reinterpret_cast<const uint4*>(t.buckets + mine) : make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0u, 0u);
        const unsigned long long key = (unsigned long long)head.y << 32 | head.x;
        const bool used = key != TG_EMPTY;
        if (!__any_sync(0xffffffffu, used)) continue;
        TgSlot home[6];
#pragma unroll
        for (int e = 0; e < 6; ++e) home[e] = used ? t.buckets[mine].e[e] : TgSlot{-1, 0u};
        tg_export_some(key, home, min_count, lane, keys, counts, max_entries, n_out);
        for (unsigned more = __ballot_sync(0xffffffffu, used && head.z != 0); more; more &= more - 1) {
            const int src = __ffs((int)more) - 1;
            TgWalk w;
            w.part = make_uint4(0u, 0u, __shfl_sync(0xffffffffu, head.z, src), __shfl_sync(0xffffffffu, head.w, src));
            tg_open_extents(t, w, lane);
            const unsigned long long k = __shfl_sync(0xffffffffu, key, src);
            if (w.chain)
                tg_each_chained(t, w.chain, lane, [&](uint4 v) {
                    const TgSlot two[2] = {TgSlot{(int32_t)v.x, v.y}, TgSlot{(int32_t)v.z, v.w}};
                    tg_export_some(k, two, min_count, lane, keys, counts, max_entries, n_out);
                });
            if (w.n > EXPORT_LONG) {
                int place = 0;
                if (lane == 0) place = atomicAdd(&s_long, 1);
                place = __shfl_sync(0xffffffffu, place, 0);
                if (place < EXPORT_MAX_LONG) {
                    if (lane == 0) s_home[place] = g * 32 + src;
                    continue;
                }
            }
            tg_export_extents(t, w, k, 0, 1, min_count, lane, keys, counts, max_entries, n_out);
        }
    }
    __syncthreads();
    for (int i = 0; i < min(s_long, EXPORT_MAX_LONG); ++i) {
        const unsigned long long key = t.buckets[s_home[i]].key;
        tg_export_extents(t, tg_open(t, s_home[i], lane), key, warp, EXPORT_THREADS / 32, min_count, lane, keys, counts, max_entries, n_out);
    }
}

// Adds exported entries to a table (counts add up, saturating).
__global__ void k_tg_import(TgView t, const int32_t* __restrict__ keys, const uint32_t* __restrict__ counts, unsigned long long n) {
    const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    if (i >= n || *t.status != 0) return;
    const int a = keys[3 * i], b = keys[3 * i + 1], c = keys[3 * i + 2];
    uint32_t inc = counts[i];
    if (a < 0 || b < 0 || c < 0 || a >= t.vocab || b >= t.vocab || c >= t.vocab) {
        atomicCAS(t.status, 0, (int)ADED_ERR_INVALID_ARG);
        return;
    }
    if (inc == 0) return;
    if (inc > t.cap) inc = t.cap;
    tg_add(t, a, b, c, inc, false);
}

// Top-k lists of q contexts.  A block takes `per_block` queries.  Its threads first look up the home buckets, one query each,
// and hang queries of the same context on one entry of a hash table in shared memory: in text, frequent contexts are asked for
// again and again, and they are the ones with thousands of continuations.  Every distinct context is then scanned once per
// block, by one warp -- or, while at most TOPK_WIDE contexts of the block have more than TOPK_LONG entries, those by the whole
// block -- and the list is written to all queries that asked for it.
// Measured (2^20 queries drawn from a 16-million-token text, k = 4; 4.9e9 entries on the contexts of all queries, 0.2-0.5e9 on
// the distinct ones of each block): bound by the L2 reads of the entries.
constexpr int TOPK_THREADS = 512, TOPK_WARPS = TOPK_THREADS / 32, TOPK_MAX_QUERIES = 3072;
constexpr uint32_t TOPK_LONG = 2048;
constexpr int TOPK_WIDE = 4, TOPK_LEAD_QUERIES = 2432;

// Slots of the block's hash table: a power of two, at most four fifths full.
static __host__ __device__ int topk_slots(int per_block) {
    int n = 32;
    while (n < per_block + per_block / 4) n *= 2;
    return n;
}
static size_t topk_smem(int per_block) { return (size_t)topk_slots(per_block) * 8 + (size_t)per_block * 8; }

// One context by all warps of the block; warp 0 hands the list and the sum to `write`.
template <typename F>
__device__ __forceinline__ void topk_wide(const TgView& t, int home, int k, int warp, int lane, unsigned long long* s_best, uint32_t* s_total, F write) {
    unsigned long long best = 0;
    uint32_t total = 0;
    tg_scan(t, tg_open(t, (uint32_t)home, lane), warp, TOPK_WARPS, k, lane, best, total);
    s_best[warp * 32 + lane] = lane < k ? best : 0ull;
    total = __reduce_add_sync(0xffffffffu, total);
    if (lane == 0) s_total[warp] = total;
    __syncthreads();
    if (warp == 0) {
        for (int w = 1; w < TOPK_WARPS; w += 2) tg_offer2(s_best[w * 32 + lane], w + 1 < TOPK_WARPS ? s_best[(w + 1) * 32 + lane] : 0ull, k, lane, best);
        total = __reduce_add_sync(0xffffffffu, lane < TOPK_WARPS ? s_total[lane] : 0u);
        write(best, total);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(TOPK_THREADS, 3)
k_tg_topk(TgView t, const int32_t* __restrict__ ctx, int q, int k, int per_block, int32_t* __restrict__ out_tok,
          uint32_t* __restrict__ out_cnt, uint32_t* __restrict__ out_total) {
    extern __shared__ int32_t topk_smem_raw[];
    const int slots = topk_slots(per_block);
    int32_t* s_key = topk_smem_raw;                 // [slots] home bucket, -1 empty
    int32_t* s_head = s_key + slots;                // [slots] last query (index in the block) hung on it, -1 none
    int32_t* s_next = s_head + slots;               // [per_block]
    int32_t* s_order = s_next + per_block;          // [per_block] the slots in use, long contexts from the back
    __shared__ int s_n, s_long, s_cursor;
    __shared__ unsigned long long s_best[TOPK_WARPS * 32];
    __shared__ uint32_t s_total[TOPK_WARPS];
    const int q0 = blockIdx.x * per_block, nq = min(per_block, q - q0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < slots; i += TOPK_THREADS) { s_key[i] = -1; s_head[i] = -1; }
    if (threadIdx.x == 0) { s_n = 0; s_long = 0; s_cursor = 0; }
    __syncthreads();
    for (int i = threadIdx.x; i < nq; i += TOPK_THREADS) {
        const int a = ctx[2 * (size_t)(q0 + i)], b = ctx[2 * (size_t)(q0 + i) + 1];
        int64_t home = -1;
        if (a >= 0 && b >= 0 && a < t.vocab && b < t.vocab) home = tg_find_home(t, tg_key(a, b), false);
        if (home < 0) {
            for (int r = 0; r < k; ++r) { out_tok[(size_t)(q0 + i) * k + r] = -1; out_cnt[(size_t)(q0 + i) * k + r] = 0; }
            if (out_total) out_total[q0 + i] = 0;
            continue;
        }
        int at = (int)(((uint32_t)home * 0x9E3779B1u) >> 8) & (slots - 1);
        for (;;) {                                  // (more slots than queries: ends)
            const int have = atomicCAS(&s_key[at], -1, (int)home);
            if (have == -1) {
                if ((t.buckets[home].n_more & ~TG_CLOSED) > TOPK_LONG) s_order[per_block - 1 - atomicAdd(&s_long, 1)] = at;
                else s_order[atomicAdd(&s_n, 1)] = at;
            }
            if (have == -1 || have == (int)home) break;
            at = (at + 1) & (slots - 1);
        }
        s_next[i] = atomicExch(&s_head[at], i);
    }
    __syncthreads();
    auto write = [&](int slot, unsigned long long best, uint32_t total) {
        for (int i = s_head[slot]; i >= 0; i = s_next[i]) {
            const size_t row = (size_t)(q0 + i);
            if (lane < k) {
                out_tok[row * k + lane] = tg_packed_tok(best);
                out_cnt[row * k + lane] = tg_packed_cnt(best);
            }
            if (lane == 0 && out_total) out_total[row] = total;
        }
    };
    const int n_long = s_long, n_short = s_n;
    const bool wide = n_long <= TOPK_WIDE;
    for (int j = 0; wide && j < n_long; ++j) {
        const int slot = s_order[per_block - 1 - j];
        topk_wide(t, s_key[slot], k, warp, lane, s_best, s_total, [&](unsigned long long best, uint32_t total) { write(slot, best, total); });
    }
    // the rest, longest first as far as they are sorted
    const int first = wide ? n_long : 0, jobs = n_long - first + n_short;
    for (;;) {
        int j = 0;
        if (lane == 0) j = atomicAdd(&s_cursor, 1);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= jobs) break;
        const int slot = j < n_long - first ? s_order[per_block - 1 - first - j] : s_order[j - (n_long - first)];
        unsigned long long best = 0;
        uint32_t total = 0;
        tg_scan(t, tg_open(t, (uint32_t)s_key[slot], lane), 0, 1, k, lane, best, total);
        write(slot, best, __reduce_add_sync(0xffffffffu, total));
    }
}

// Many queries: every context of the call is scanned once, by three kernels whose only scratch is the output arrays themselves
// (lookups of one table may run on several streams, so the table holds none).
//   1. k_topk_mark: a thread per query finds the home bucket.  Contexts with entries beyond it are grouped: the query's index
//      goes into a hash table that lies in out_cnt (all bits set before), and the first query of a context found there leads the
//      others.  out_tok[first of the row] says what a row is: MARK_OWN (answer it; its home bucket, or -1, is in the next
//      word) or the leader's index, encoded below MARK_OWN.  Contexts that are all in their home bucket are answered there and then.
//   2. k_topk_lead: the leaders' rows, and those whose counts the hash table took; it is overwritten with results.
//   3. k_topk_copy: the followers' rows, from their leaders'.
// Needs two words per row (k >= 2).  The table takes the smallest power of two that is at least half the queries; a query that
// finds no slot within MARK_PROBES answers itself.
// What bounds it: dependent reads of a table far larger than L2 (home bucket, directory, entries), in each kernel; the stores of the
// short rows, one word at a time, took as long as the reads, and a warp for every context with seven continuations twice as long as
// now.  Measured, 2^20 queries on the table of a 16-million-token text, us: k = 2, 4, 8: 151, 188, 253 before; 92, 100, 124 now
// (mark 46, lead 48, copy 14 under ncu, 57 + 93 + 32 before).
// Taken from the number of queries on from where it is the faster one, which depends on how long contexts are and so on how
// much text the table holds (topk_text).  k = 4, the per-block kernel against this, us, everything in L2 / a cold one, for a text of
// independent Zipf tokens and for one in which every other token is followed by its usual successor (longer contexts, asked for more often):
//   text             queries   Zipf               usual successors
//   10^5              2^15     25/29 -> 23/30     25/29 -> 22/28
//   2 x 10^5          2^15     29/35 -> 25/33     31/35 -> 24/32
//   4 x 10^5          2^13     23/27 -> 27/34     29/34 -> 25/32
//                     2^14     28/33 -> 27/34     37/40 -> 25/30
//   10^6              2^12     25/29 -> 31/38     36/39 -> 28/36
//                     2^13     33/37 -> 32/39     43/47 -> 28/34
//   4 x 10^6          2^12     33/37 -> 41/48     65/68 -> 36/46
//                     2^13     54/57 -> 40/46     81/86 -> 36/44
//   1.6 x 10^7        2^12     91/94 -> 52/60     125/122 -> 42/52
// (k = 2 gains less, k = 8 and 24 more.)
constexpr int MARK_OWN = -2, MARK_PROBES = 16;
static int topk_bulk_min(uint64_t text) { return text > 1u << 19 ? 1 << 12 : text > 1u << 18 ? 1 << 13 : text > 1u << 16 ? 1 << 15 : 1 << 16; }
__device__ __forceinline__ int mark_leader(int q) { return MARK_OWN - 1 - q; }       // (its own inverse)

// One thread's list: the first k of `key` (in order; eight of them, none beyond) as a row.  `vec`: the words of a row that one store takes.
__device__ __forceinline__ void topk_store(const unsigned long long (&key)[8], int k, int vec, int32_t* tok, uint32_t* cnt) {
#pragma unroll
    for (int r = 0; r < 8; r += 4) {
        if (r >= k) break;
        const int4 a = make_int4(tg_packed_tok(key[r]), tg_packed_tok(key[r + 1]), tg_packed_tok(key[r + 2]), tg_packed_tok(key[r + 3]));
        const uint4 c = make_uint4(tg_packed_cnt(key[r]), tg_packed_cnt(key[r + 1]), tg_packed_cnt(key[r + 2]), tg_packed_cnt(key[r + 3]));
        if (vec == 4) {
            *reinterpret_cast<int4*>(tok + r) = a;
            *reinterpret_cast<uint4*>(cnt + r) = c;
        } else if (vec == 2) {
            *reinterpret_cast<int2*>(tok + r) = make_int2(a.x, a.y);
            *reinterpret_cast<uint2*>(cnt + r) = make_uint2(c.x, c.y);
            if (r + 2 < k) {
                *reinterpret_cast<int2*>(tok + r + 2) = make_int2(a.z, a.w);
                *reinterpret_cast<uint2*>(cnt + r + 2) = make_uint2(c.z, c.w);
            }
        } else {
            tok[r] = a.x; cnt[r] = c.x;
            if (r + 1 < k) { tok[r + 1] = a.y; cnt[r + 1] = c.y; }
            if (r + 2 < k) { tok[r + 2] = a.z; cnt[r + 2] = c.z; }
            if (r + 3 < k) { tok[r + 3] = a.w; cnt[r + 3] = c.w; }
        }
    }
    for (int r = 8; r < k; ++r) { tok[r] = -1; cnt[r] = 0; }
}

// The six entries of a home bucket, best first, by one thread; the sum of their counts.
__device__ __forceinline__ uint32_t topk_bucket(const TgView& t, int home, unsigned long long (&key)[8]) {
    uint32_t total = 0;
    const uint4* part = reinterpret_cast<const uint4*>(t.buckets + (home < 0 ? 0 : home));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        uint4 v = make_uint4(0xFFFFFFFFu, 0u, 0xFFFFFFFFu, 0u);
        if (home >= 0) v = part[i + 1];
        if ((int32_t)v.x >= 0) total += v.y;
        if ((int32_t)v.z >= 0) total += v.w;
        key[2 * i] = tg_pack(t, (int32_t)v.x, v.y);
        key[2 * i + 1] = tg_pack(t, (int32_t)v.z, v.w);
    }
    key[6] = key[7] = 0;
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int j = r + 1; j < 6; ++j)
            if (key[j] > key[r]) { const unsigned long long x = key[r]; key[r] = key[j]; key[j] = x; }
    return total;
}
// A context that is all in its home bucket (or not stored: home < 0).
__device__ __forceinline__ void topk_home(const TgView& t, int home, int k, int vec, int32_t* tok, uint32_t* cnt, uint32_t* total_out) {
    unsigned long long key[8];
    const uint32_t total = topk_bucket(t, home, key);
    topk_store(key, k, vec, tok, cnt);
    if (total_out) *total_out = total;
}

// A block first finds equal contexts among its own queries (a hash table in shared memory, as k_tg_topk), and only the first of each
// goes to the table: one in twelve of the synthetic text's queries asks for the same context.  A context that is all in its home
// bucket is answered at once, where its row's counts are not part of the hash table (row >= deferred).
constexpr int MARK_THREADS = 512, MARK_SLOTS = 2 * MARK_THREADS;
__global__ void __launch_bounds__(MARK_THREADS, 4)
k_topk_mark(TgView t, const int32_t* __restrict__ ctx, int q, int k, int vec, uint32_t mask, int deferred, int32_t* __restrict__ out_tok,
            uint32_t* out_cnt, uint32_t* __restrict__ out_total) {
    __shared__ int2 s_ctx[MARK_THREADS];
    __shared__ int s_slot[MARK_SLOTS], s_mark[MARK_THREADS];
    pdl_enter();
    const int me = threadIdx.x;
    const long long at_row = (long long)blockIdx.x * MARK_THREADS + me;
    const bool mine = at_row < q;
    const int row = mine ? (int)at_row : 0;
    int2 c = make_int2(-1, -1);
    if (mine) c = make_int2(ctx[2 * (size_t)row], ctx[2 * (size_t)row + 1]);
    s_ctx[me] = c;
    s_slot[me] = -1;
    s_slot[MARK_THREADS + me] = -1;
    __syncthreads();
    const uint32_t hash = tg_hash(tg_key(c.x, c.y));
    int first = me;                                            // first of the block's queries with this context
    if (mine) {
        for (uint32_t at = hash & (MARK_SLOTS - 1);; at = (at + 1) & (MARK_SLOTS - 1)) {      // (twice as many slots as queries: ends)
            const int have = atomicCAS(&s_slot[at], -1, me);
            if (have == -1) break;
            if (s_ctx[have].x == c.x && s_ctx[have].y == c.y) { first = have; break; }
        }
    }
    int mark = MARK_OWN, home = -1;
    if (mine && first == me) {
        bool further = false;                                  // entries beyond the home bucket: the context is grouped
        if (c.x >= 0 && c.y >= 0 && c.x < t.vocab && c.y < t.vocab) {
            const int limit = t.n_home < (uint32_t)TG_MAX_PROBE ? (int)t.n_home : TG_MAX_PROBE;
            for (int probe = 0; probe < limit; ++probe) {
                const uint32_t at = (hash + probe) & t.n_home_mask;
                uint4 head;                                    // (all of the bucket comes from memory at once: its entries may be wanted next)
                asm volatile("ld.global.L2::64B.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(head.x), "=r"(head.y), "=r"(head.z), "=r"(head.w) : "l"(t.buckets + at));
                if (head.y == (uint32_t)c.x && head.x == (uint32_t)c.y) {
                    home = (int)at;
                    further = head.w != 0;
                    break;
                }
                if ((head.x & head.y) == 0xFFFFFFFFu) break;   // TG_EMPTY
            }
        }
        if (further) {
            uint32_t probe_at = (uint32_t)home * 0x9E3779B1u;
            probe_at ^= probe_at >> 15;
            for (int probe = 0; probe < MARK_PROBES; ++probe, ++probe_at) {
                uint32_t* slot = out_cnt + (probe_at & mask);
                uint32_t have = *reinterpret_cast<volatile uint32_t*>(slot);
                if (have == 0xFFFFFFFFu) have = atomicCAS(slot, 0xFFFFFFFFu, (uint32_t)row);
                if (have == 0xFFFFFFFFu) break;
                if (ctx[2 * (size_t)have] == c.x && ctx[2 * (size_t)have + 1] == c.y) { mark = mark_leader((int)have); break; }
            }
        }
        s_mark[me] = mark;
        if (!further && row >= deferred) {
            topk_home(t, home, k, vec, out_tok + (size_t)row * k, out_cnt + (size_t)row * k, out_total ? out_total + row : nullptr);
            mark = 0;                                          // (answered)
        }
    }
    __syncthreads();
    if (!mine || mark == 0) return;
    if (first != me) mark = s_mark[first] == MARK_OWN ? mark_leader(row - me + first) : s_mark[first];
    if (vec > 1) {
        *reinterpret_cast<int2*>(out_tok + (size_t)row * k) = make_int2(mark, home);
    } else {
        out_tok[(size_t)row * k] = mark;
        out_tok[(size_t)row * k + 1] = home;
    }
}

// A context to look up: its row, its home bucket, and what the bucket's header says (first extent, entries beyond the bucket).
struct TopkJob { int row, home; uint32_t more, n; };

// Contexts of up to LEAD_SMALL further entries, a thread each (k <= 8): most contexts have few, and a warp for one spends its
// instructions on lists of four that 32 lanes hold together (eight lanes each, four contexts per warp: 1000 instructions per four
// contexts, 20 us of 80 on the table of a 16-million-token text).
constexpr uint32_t LEAD_SMALL = 48;                // (units 0 .. 7, extents 0 .. 3: the directory's first four words say where)
__device__ __forceinline__ void topk_thread(const TgView& t, const TopkJob& job, int k, int vec, int32_t* tok, uint32_t* cnt, uint32_t* total_out) {
    unsigned long long key[8];
    const uint4 dir = *reinterpret_cast<const uint4*>(t.pool + (size_t)(job.more - 1) * TG_UNIT);
    uint32_t total = topk_bucket(t, job.home, key);
    const uint32_t pairs = (job.n + 1) / 2;
    constexpr int BATCH = 3;                       // a unit's entries at a time
    unsigned long long floor_key = key[0];         // the k-th best so far
#pragma unroll
    for (int r = 1; r < 8; ++r)
        if (r < k) floor_key = key[r];
    for (uint32_t m = 0; m * BATCH < pairs; ++m) {
        const int s = tg_extent(m);
        const uint32_t base = s == 0 ? job.more + TG_DIR_UNITS : s == 1 ? dir.y : s == 2 ? dir.z : dir.w;
        if (base == 0 || base == TG_FAILED) continue;
        const size_t unit = (size_t)(base - 1) + (m + 1 - (1u << s));
        if (!ADED_IN_RANGE(unit < t.n_units, t.status)) continue;
        const uint4* from = reinterpret_cast<const uint4*>(t.pool + unit * TG_UNIT);
        uint4 v[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            v[i] = make_uint4(0xFFFFFFFFu, 0u, 0xFFFFFFFFu, 0u);
            if (m * BATCH + i < pairs) v[i] = from[i];
            if (2 * (m * BATCH + i) + 1 >= job.n) { v[i].z = 0xFFFFFFFFu; v[i].w = 0u; }
        }
#pragma unroll
        for (int e = 0; e < 2 * BATCH; ++e) {
            const int32_t token = (int32_t)(e & 1 ? v[e / 2].z : v[e / 2].x);
            const uint32_t count = e & 1 ? v[e / 2].w : v[e / 2].y;
            if (token >= 0) total += count;
            unsigned long long x = tg_pack(t, token, count);
            if (x <= floor_key) continue;
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if (x > key[r]) { const unsigned long long y = key[r]; key[r] = x; x = y; }
            floor_key = key[0];
#pragma unroll
            for (int r = 1; r < 8; ++r)
                if (r < k) floor_key = key[r];
        }
    }
    topk_store(key, k, vec, tok, cnt);
    if (total_out) *total_out = total;
}

__global__ void __launch_bounds__(TOPK_THREADS, 3)
k_topk_lead(TgView t, int q, int k, int vec, int per_block, int32_t* __restrict__ out_tok, uint32_t* __restrict__ out_cnt, uint32_t* __restrict__ out_total) {
    __shared__ TopkJob s_job[TOPK_LEAD_QUERIES];   // few entries from the front, more from the back
    __shared__ int s_rows, s_n, s_big, s_long, s_cursor;
    __shared__ int2 s_long_job[4 * TOPK_WIDE];
    __shared__ unsigned long long s_best[TOPK_WARPS * 32];
    __shared__ uint32_t s_total[TOPK_WARPS];
    __shared__ uint16_t s_row[TOPK_LEAD_QUERIES];  // the block's rows that have to be answered
    pdl_enter();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) { s_rows = 0; s_n = 0; s_big = 0; s_long = 0; s_cursor = 0; }
    __syncthreads();
    const bool by_thread = k <= 8 && t.chain == nullptr;
    // A block takes every gridDim.x-th row: the frequent contexts' leaders are among the rows that were marked first.
#pragma unroll 4
    for (int i = threadIdx.x; i < per_block; i += TOPK_THREADS) {
        const long long row = (long long)i * gridDim.x + blockIdx.x;
        if (row < q && out_tok[row * k] == MARK_OWN) s_row[atomicAdd(&s_rows, 1)] = (uint16_t)i;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < s_rows; i += TOPK_THREADS) {
        TopkJob job;
        job.row = (int)((long long)s_row[i] * gridDim.x + blockIdx.x);
        job.home = out_tok[(size_t)job.row * k + 1];
        uint4 head = make_uint4(0u, 0u, 0u, 0u);
        if (job.home >= 0) head = *reinterpret_cast<const uint4*>(t.buckets + job.home);
        job.more = head.z;
        job.n = head.w & ~TG_CLOSED;
        if (job.n == 0) {
            topk_home(t, job.home, k, vec, out_tok + (size_t)job.row * k, out_cnt + (size_t)job.row * k, out_total ? out_total + job.row : nullptr);
            continue;
        }
        if (by_thread && job.n <= LEAD_SMALL && job.more != TG_FAILED && job.more != 0) {
            // (directory and first unit are on their way to L2 while the others are sorted)
            const char* dir = reinterpret_cast<const char*>(t.pool + (size_t)(job.more - 1) * TG_UNIT);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(dir));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(dir + (TG_DIR_UNITS + 1) * TG_UNIT * sizeof(TgSlot) - 1));
            s_job[atomicAdd(&s_n, 1)] = job;
            continue;
        }
        int place = 4 * TOPK_WIDE;
        if (job.n > TOPK_LONG) place = atomicAdd(&s_long, 1);
        if (place < 4 * TOPK_WIDE) s_long_job[place] = make_int2(job.row, job.home);
        else s_job[TOPK_LEAD_QUERIES - 1 - atomicAdd(&s_big, 1)] = job;
    }
    __syncthreads();
    auto write = [&](int row, unsigned long long best, uint32_t total) {
        if (lane < k) {
            out_tok[(size_t)row * k + lane] = tg_packed_tok(best);
            out_cnt[(size_t)row * k + lane] = tg_packed_cnt(best);
        }
        if (lane == 0 && out_total) out_total[row] = total;
    };
    // the longest by the whole block (as many as there is room for); then, as warps come free, 32 small ones at a time and the others one by one
    const int n_long = min(s_long, 4 * TOPK_WIDE), n_small = s_n, small_steps = (n_small + 31) / 32, steps = small_steps + s_big;
    for (int j = 0; j < n_long; ++j)
        topk_wide(t, s_long_job[j].y, k, warp, lane, s_best, s_total, [&](unsigned long long best, uint32_t total) { write(s_long_job[j].x, best, total); });
    for (;;) {
        int j = 0;
        if (lane == 0) j = atomicAdd(&s_cursor, 1);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= steps) break;
        if (j < small_steps) {
            const int i = j * 32 + lane;
            if (i < n_small) {
                const TopkJob job = s_job[i];
                topk_thread(t, job, k, vec, out_tok + (size_t)job.row * k, out_cnt + (size_t)job.row * k, out_total ? out_total + job.row : nullptr);
            }
            __syncwarp();
        } else {
            const TopkJob job = s_job[TOPK_LEAD_QUERIES - 1 - (j - small_steps)];
            unsigned long long best = 0;
            uint32_t total = 0;
            tg_scan(t, tg_open(t, (uint32_t)job.home, lane), 0, 1, k, lane, best, total);
            write(job.row, best, __reduce_add_sync(0xffffffffu, total));
        }
    }
}

// V: the words of a row that one load takes (1, 2, 4: k is a multiple of it and the arrays are aligned to it).
template <typename V>
__global__ void __launch_bounds__(256) k_topk_copy(int q, int k, V* __restrict__ out_tok, V* __restrict__ out_cnt, uint32_t* __restrict__ out_total) {
    pdl_enter();
    const uint32_t row = blockIdx.x * 256 + threadIdx.x;
    if (row >= (uint32_t)q) return;
    const int words = k / (int)(sizeof(V) / sizeof(int32_t));
    const int mark = reinterpret_cast<const int32_t*>(out_tok)[(size_t)row * k];
    if (mark >= MARK_OWN) return;
    const uint32_t lead = (uint32_t)mark_leader(mark);
    const size_t from = (size_t)lead * words, to = (size_t)row * words;
    uint32_t total = 0;
    if (out_total) total = out_total[lead];
    for (int r = 0; r < words; ++r) {
        const V a = out_tok[from + r], b = out_cnt[from + r];
        out_tok[to + r] = a;
        out_cnt[to + r] = b;
    }
    if (out_total) out_total[row] = total;
}

// Draft tree of n_nodes nodes for the context (ctx[0], ctx[1]); one block of 32 warps.
// Level by level: every node of the current level gets its top-k list -- the block's warps are shared out evenly, so that
// the first levels' few nodes, whose contexts may have thousands of continuations, are scanned by several warps each --
// then one warp appends the lists in node order, rank order: the same tree as visiting the nodes in index order.
// Latency-bound: a level is the chain home bucket -> directory -> entries -> merge.  The filler pass (draft_fill) hangs caller-
// supplied tokens under nodes with room, round-robin, until the tree is full.
constexpr int DRAFT_MAX_FILLER = 4 * ADED_MAX_NODES;

// Filler pass over a tree held in shared memory (tok, par, dep; kid[p][0 .. nkid[p]) the child tokens of node p), by one warp:
// nodes are visited round-robin, a visited node with depth < max_depth and fewer than k children gets the next filler token
// none of its children holds.  Returns the new node count (every lane); *fail when the filler runs out, holds a token outside the
// vocabulary, or no node has room.  The nodes with room wait in two lists (`turn`, [2][ADED_MAX_NODES]: of this round, to which new
// nodes are added, and of the next).  Up to 32 of them are served at once, a token each; the first whose token does not fit ends
// the step, as those behind it would have got other tokens.  The last one of a round goes on with its child, which is next in turn and has
// no children, the child with its own, and so on: a chain, a lane per link.
// Latency of the steps.  draft_tree for a context without continuations (all nodes are filler), us: a thread that visited every node; a warp
// with a token per step; this.  128 nodes, depth 8, k = 8: 30, 35, 9; 97 nodes, depth 4, k = 4: 31, 28, 11; a chain of 128: 24, 35, 6.
__device__ __forceinline__ int draft_fill(int32_t* tok, int32_t* par, int32_t* dep, int32_t* nkid, int32_t* kid, int n, int n_nodes,
                                          int max_depth, int k, const int32_t* fill, int n_filler, int vocab, int lane, int16_t* turn, bool* fail) {
    const unsigned below = (1u << lane) - 1u;
    int16_t *now = turn, *then = turn + ADED_MAX_NODES;
    int n_now = 0, n_then = 0, at = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const bool room = i < n && dep[i] < max_depth && nkid[i] < k;
        const unsigned m = __ballot_sync(0xffffffffu, room);
        if (room) now[n_now + __popc(m & below)] = (int16_t)i;
        n_now += __popc(m);
    }
    __syncwarp();
    int pos = 0;
    while (n < n_nodes) {
        if (at == n_now) {
            int16_t* const x = now;
            now = then;
            then = x;
            n_now = n_then;
            n_then = at = 0;
        }
        const bool chain = n_now - at == 1;
        const int served = min(min(32, chain ? max_depth - dep[now[at]] : n_now - at), min(n_nodes - n, n_filler - pos));
        if (served <= 0) { *fail = true; break; }                 // no node has room, or no token is left
        int p = 0, f = 0, nk = 0, depth = 0;
        bool clash = false;
        if (lane < served) {
            const bool link = chain && lane > 0;                  // (the parent is the lane before)
            p = link ? n + lane - 1 : now[at + lane];
            f = fill[pos + lane];
            nk = link ? 0 : nkid[p];
            depth = link ? dep[now[at]] + 1 + lane : dep[p] + 1;
            for (int j = 0; j < nk; ++j) clash |= kid[p * ADED_DRAFT_MAX_K + j] == f;
        }
        const unsigned clashes = __ballot_sync(0xffffffffu, clash), stops = clashes | __ballot_sync(0xffffffffu, lane < served && (f < 0 || f >= vocab));
        const int fit = stops ? __ffs((int)stops) - 1 : served;
        const bool mine = lane < fit, last = !chain || lane == fit - 1, deeper = mine && last && depth < max_depth, again = mine && nk + 1 < k;
        const unsigned deeper_m = __ballot_sync(0xffffffffu, deeper), again_m = __ballot_sync(0xffffffffu, again);
        if (mine) {
            const int c = n + lane;
            kid[p * ADED_DRAFT_MAX_K + nk] = f;
            nkid[p] = nk + 1;
            tok[c] = f;
            par[c] = p;
            dep[c] = depth;
            if (last) nkid[c] = 0;
            if (deeper) now[n_now + __popc(deeper_m & below)] = (int16_t)c;
            if (again) then[n_then + __popc(again_m & below)] = (int16_t)p;
        }
        n_now += __popc(deeper_m);
        n_then += __popc(again_m);
        n += fit;
        at += chain ? min(fit, 1) : fit;
        pos += fit;
        if (stops) {
            if (!(clashes >> fit & 1u)) { *fail = true; break; }   // (a token outside the vocabulary)
            ++pos;                                                // a child holds it: this node gets the next one
        }
        __syncwarp();
    }
    return n;
}

// The k best of the lists of `parts` warps, [parts][ADED_DRAFT_MAX_K] in shared memory, of which the first k of each are used.
__device__ __forceinline__ void draft_merge(const unsigned long long* lists, int parts, int k, int lane, unsigned long long& best) {
    constexpr int AT_ONCE = 32 / ADED_DRAFT_MAX_K;                // eight warps' lists at a time, two per lane
    for (int i = 0; i < parts; i += 2 * AT_ONCE) {
        const int from = i + lane / ADED_DRAFT_MAX_K, r = lane % ADED_DRAFT_MAX_K;
        const unsigned long long* list = lists + from * ADED_DRAFT_MAX_K + r;
        tg_offer2(from < parts && r < k ? list[0] : 0ull, from + AT_ONCE < parts && r < k ? list[AT_ONCE * ADED_DRAFT_MAX_K] : 0ull, k, lane, best);
    }
}

__global__ void __launch_bounds__(1024)
k_draft_tree(TgView t, const int32_t* __restrict__ ctx, int n_nodes, int max_depth, int k,
             const int32_t* __restrict__ filler, int n_filler, int32_t* __restrict__ out_tok,
             int32_t* __restrict__ out_par, int32_t* __restrict__ out_real) {
    __shared__ int32_t s_tok[ADED_MAX_NODES], s_par[ADED_MAX_NODES], s_dep[ADED_MAX_NODES], s_nkid[ADED_MAX_NODES];
    __shared__ int32_t s_cand[ADED_MAX_NODES * ADED_DRAFT_MAX_K];   // top-k lists, later the child tokens of every node
    __shared__ int32_t s_fill[DRAFT_MAX_FILLER];
    __shared__ unsigned long long s_part[32 * ADED_DRAFT_MAX_K];    // the lists of the warps that share a node
    __shared__ int16_t s_turn[2 * ADED_MAX_NODES];
    __shared__ int s_n, s_lo, s_hi, s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_enter();
    const int prev_token = ctx[0];
    if (threadIdx.x == 0) {
        s_tok[0] = ctx[1];
        s_par[0] = -1;
        s_dep[0] = 0;
        s_n = 1;
        s_lo = 0;
        s_hi = 1;
        s_fail = 0;
    }
    for (int i = threadIdx.x; i < n_filler; i += blockDim.x) s_fill[i] = filler[i];
    for (int i = threadIdx.x; i < ADED_MAX_NODES; i += blockDim.x) s_nkid[i] = 0;
    __syncthreads();
    for (int d = 0; d < max_depth; ++d) {
        const int lo = s_lo, hi = s_hi;
        if (lo >= hi || s_n >= n_nodes) break;
        int parts = 1;                                  // warps per node
        while (parts * 2 * (hi - lo) <= 32) parts *= 2;
        for (int node = lo + warp / parts; node < hi; node += 32 / parts) {
            const int u = node == 0 ? prev_token : s_tok[s_par[node]], w = s_tok[node];
            unsigned long long best = 0;
            uint32_t total = 0;
            tg_scan(t, tg_open(t, u, w, lane), warp % parts, parts, k, lane, best, total);
            if (lane < k) {
                if (parts == 1) s_cand[node * ADED_DRAFT_MAX_K + lane] = tg_packed_tok(best);
                else s_part[warp * ADED_DRAFT_MAX_K + lane] = best;
            }
        }
        __syncthreads();
        if (parts > 1 && warp < hi - lo) {
            unsigned long long best = 0;
            draft_merge(s_part + warp * parts * ADED_DRAFT_MAX_K, parts, k, lane, best);
            if (lane < k) s_cand[(lo + warp) * ADED_DRAFT_MAX_K + lane] = tg_packed_tok(best);
        }
        __syncthreads();
        if (warp == 0) {
            int n = s_n;
            for (int node0 = lo; node0 < hi && n < n_nodes; node0 += 32) {
                const int node = node0 + lane;
                int32_t tok[ADED_DRAFT_MAX_K];
                int mine = 0;                               // this node's children (valid entries come first)
#pragma unroll
                for (int j = 0; j < ADED_DRAFT_MAX_K; ++j) tok[j] = node < hi && j < k ? s_cand[node * ADED_DRAFT_MAX_K + j] : -1;
#pragma unroll
                for (int j = 0; j < ADED_DRAFT_MAX_K; ++j) mine += tok[j] >= 0;
                int upto = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int other = __shfl_up_sync(0xffffffffu, upto, o);
                    if (lane >= o) upto += other;
                }
                const int at = n + upto - mine;
                const int kept = max(0, min(mine, n_nodes - at));
#pragma unroll
                for (int j = 0; j < ADED_DRAFT_MAX_K; ++j)
                    if (j < kept) {
                        s_tok[at + j] = tok[j];
                        s_par[at + j] = node;
                        s_dep[at + j] = d + 1;
                    }
                if (kept > 0) s_nkid[node] = kept;          // s_cand[node][0 .. kept) are this node's child tokens
                n = min(n_nodes, n + __shfl_sync(0xffffffffu, upto, 31));
            }
            if (lane == 0) { s_lo = hi; s_hi = n; s_n = n; }
        }
        __syncthreads();
    }
    if (warp == 0) {
        int n = s_n;
        bool fail = false;
        if (lane == 0 && out_real) *out_real = n;
        if (filler && n < n_nodes) n = draft_fill(s_tok, s_par, s_dep, s_nkid, s_cand, n, n_nodes, max_depth, k, s_fill, n_filler, t.vocab, lane, s_turn, &fail);
        __syncwarp();
        if (lane == 0) {
            s_n = n;
            if (fail) { s_fail = 1; atomicCAS(t.status, 0, (int)ADED_ERR_INVALID_ARG); }
        }
    }
    __syncthreads();
    const int n = s_n;
    for (int i = threadIdx.x; i < n_nodes; i += blockDim.x) {
        out_tok[i] = (i < n && !(s_fail && i == 0)) ? s_tok[i] : -1;
        out_par[i] = i < n ? s_par[i] : -1;
    }
}

// After a verification step: the table learns the windows of (context, emitted tokens), and the last two tokens become the
// context of the next step.  A failed step (accept length < 1) leaves context and table as they are.  One thread per window.
constexpr int FEEDBACK_THREADS = 160;
static_assert(FEEDBACK_THREADS >= ADED_MAX_NODES + 2, "a thread per token of the longest span");
__global__ void __launch_bounds__(FEEDBACK_THREADS)
k_decode_feedback(TgView t, const int32_t* __restrict__ out_tok, int32_t* __restrict__ out_len, int32_t* ctx, int max_emit) {
    pdl_enter();
    __shared__ int32_t s_span[FEEDBACK_THREADS];
    int a = *out_len;
    if (a > max_emit) a = max_emit;
    const int i = threadIdx.x;
    if (i < a + 2) s_span[i] = i < 2 ? ctx[i] : out_tok[i - 2];
    __syncthreads();
    if (a < 1) {
        if (i == 0) *out_len = 0;
        return;
    }
    if (i < 2) ctx[i] = s_span[a + i];
    if (i < a) tg_add_window(t, s_span[i], s_span[i + 1], s_span[i + 2]);
}

__global__ void k_tg_get(TgView t, int a, int b, int c, uint32_t* out) {
    *out = 0;
    if (a < 0 || b < 0 || c < 0 || a >= t.vocab || b >= t.vocab || c >= t.vocab) return;
    const uint32_t* cnt = tg_find(t, a, b, c);
    if (cnt) *out = *cnt;
}

// Stored tri-grams, and buckets in use (home buckets and units of six further entries).
__global__ void k_tg_stats(TgView t, unsigned long long* out) {
    unsigned long long entries = 0, used = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < t.n_home; i += gridDim.x * blockDim.x) {
        const Bucket* bk = t.buckets + i;
        if (bk->key == TG_EMPTY) continue;
        ++used;
        for (int e = 0; e < 6; ++e) entries += bk->e[e].tok >= 0;
        if (bk->more == 0 || bk->more == TG_FAILED) continue;
        if (t.chain) {
            for (uint32_t at = bk->more, hop = 0; at != 0 && at != TG_LOCKED && hop < t.n_over; ++hop) {
                const Bucket* next = t.chain + (at - 1);
                for (int e = 0; e < 6; ++e) entries += next->e[e].tok >= 0;
                ++used;
                at = next->more;
            }
            continue;
        }
        const uint32_t n = bk->n_more & ~TG_CLOSED;
        if (!(bk->n_more & TG_CLOSED)) {
            entries += n;
            used += (n + TG_UNIT - 1) / TG_UNIT;
            continue;
        }
        const uint32_t* dir = reinterpret_cast<const uint32_t*>(t.pool + (size_t)(bk->more - 1) * TG_UNIT);
        for (uint32_t m = 0; m * TG_UNIT < n; ++m) {       // a context that ran out of room: some of its entries are not there
            const int x = tg_extent(m);
            const uint32_t base = x == 0 ? bk->more + TG_DIR_UNITS : x < TG_LINKS ? dir[x] : 0;
            if (base == 0 || base == TG_FAILED) continue;
            int here = 0;
            for (uint32_t e = 0; e < TG_UNIT && m * TG_UNIT + e < n; ++e)
                here += t.pool[((size_t)(base - 1) + (m + 1 - (1u << x))) * TG_UNIT + e].tok >= 0;
            entries += here;
            used += here > 0;
        }
    }
    atomicAdd(out, entries);
    atomicAdd(out + 1, used);
}


// ---- draft maker: Monte Carlo tree search (Eq. 2-3, Algorithm 1) -----------------------------------
// One warp runs the search, in which every iteration reads what the last one left: bound by the latency of its chain of steps.
// The tree is in shared memory; lanes hold the children of the node that is being left, the nodes of the current path, the
// continuations of a looked-up context.  Floating point is IEEE double, one rounded operation at a time (no fused multiply-add
// where the formulas have none), so that the search can be reproduced bit for bit; the exploration factor E of Eq. 3 and the
// square root depend on an integer only and come from tables the host computes; a node's mean score changes only when it is
// visited, a continuation's probability never during a search, so each is divided out once, not at every look.
// A lookup in the table is three dependent reads of memory and took most of an iteration.  The contexts a search can meet are the
// k-ary tree of continuations below the root's, which is small near the root: all warps of the block look up its first MC_AHEAD
// contexts, level by level, before the search begins (85 contexts are all there are for sentences of 4 and k = 4).  Ranking the
// sentences and laying out the result are the block's work too.
// Measured, 150 iterations, sentences of 4, 24 of them, k = 4, the kernel alone with a cold L2, six contexts, us: a warp for everything
// 269 to 389, this 133 to 164 (table of 200,000 tokens); 373 to 492 and 158 to 201 (2,000,000).  Of that the look-ahead is about 25.
constexpr int MC_MAX_ITER = 160, MC_MAX_K = ADED_DRAFT_MAX_K, MC_MAX_LEN = 8;
constexpr int MC_MAX_NODES = 1 + MC_MAX_ITER * MC_MAX_K;
constexpr int MC_WARPS = 16, MC_THREADS = MC_WARPS * 32;
constexpr int MC_AHEAD = 352;          // contexts looked up ahead (all of k = 8 and two words, of k = 4 and four)
constexpr int MC_CACHE_BYTES = 96 * 1024;

struct McParams {
    int iterations, length, n_candidates, k;
    int slots;                         // of the remembered lookups: a power of two
    double e_table[MC_MAX_ITER + 1];   // E for sum N = 0 .. iterations
    double root[MC_MAX_ITER + 1];      // square root of sum N
};
static int mc_slots(int k) {
    int n = 64;
    while (2 * n * (12 + 20 * k) <= MC_CACHE_BYTES) n *= 2;
    return n;
}

// A node of the search tree: visits, token, link, and visits of its children together | the child that is to be visited next << 16.
// link: first child (children are consecutive), number of children << 16, flags.
constexpr int MC_EXPANDED = 1 << 24, MC_CHOSEN = 1 << 25, MC_KEPT = 1 << 26;
__device__ __forceinline__ int mc_first(int link) { return link & 0xFFFF; }
__device__ __forceinline__ int mc_kids(int link) { return link >> 16 & 0xFF; }

// Remembered lookups, each in one of two neighbouring slots.  (The key of an empty slot is that of the context (-1, -1), which a caller
// may pass: no continuations, the right answer for it.)
struct McCache {
    unsigned long long* key;           // [slots]
    unsigned long long* upto;          // [slots][k] sum of the counts of continuations 0 .. j
    double* prob;                      // [slots][k]
    int32_t* word;                     // [slots][k]
    int32_t* n;                        // [slots]
    uint32_t mask;
    int k;
};
// Top-k list of one context: lane j < k holds the j-th continuation, the others nothing of use.
struct McLookup {
    int n;                             // continuations (every lane)
    int32_t word;
    double prob;                       // Eq. 1: count over the sum of ALL the context's counts
    unsigned long long upto;           // sum of the counts of continuations 0 .. j
};
// The k best of a context whose second token is b, and the sum of its counts, as a lookup, into slot `slot` (all 32 lanes).
__device__ __forceinline__ McLookup mc_keep(const TgView& t, int b, unsigned long long best, uint32_t total, int lane, const McCache& c, uint32_t slot) {
    if (lane >= c.k) best = 0;
    McLookup out;
    out.n = __popc(__ballot_sync(0xffffffffu, best != 0));
    out.word = tg_packed_tok(best);
    out.prob = best ? __ddiv_rn((double)tg_packed_cnt(best), (double)total) : 0.0;
    out.upto = tg_packed_cnt(best);
    if (best) {      // one of these is likely the next context: its home bucket comes to L2 meanwhile
        const Bucket* next = t.buckets + (tg_hash(tg_key(b, out.word)) & t.n_home_mask);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(next));
    }
#pragma unroll
    for (int o = 1; o < MC_MAX_K; o <<= 1) {
        const unsigned long long other = __shfl_up_sync(0xffffffffu, out.upto, o);
        if (lane >= o) out.upto += other;
    }
    if (lane < c.k) {
        c.upto[slot * c.k + lane] = out.upto;
        c.prob[slot * c.k + lane] = out.prob;
        c.word[slot * c.k + lane] = out.word;
    }
    if (lane == 0) c.n[slot] = out.n;
    return out;
}
__device__ __forceinline__ McLookup mc_read(const TgView& t, int a, int b, int lane, const McCache& c, uint32_t slot) {
    unsigned long long best = 0;
    uint32_t total = 0;
    tg_scan(t, tg_open(t, a, b, lane), 0, 1, c.k, lane, best, total);
    return mc_keep(t, b, best, __reduce_add_sync(0xffffffffu, total), lane, c, slot);
}
// A slot for a context: -1 when somebody has it already, or both its slots are taken.
__device__ __forceinline__ int mc_claim(const McCache& c, int2 context) {
    const unsigned long long key = tg_key(context.x, context.y);
    const uint32_t h = tg_hash(key) & c.mask;
    for (uint32_t way = 0; way < 2; ++way) {
        const unsigned long long have = atomicCAS(&c.key[h ^ way], TG_EMPTY, key);
        if (have == TG_EMPTY) return (int)(h ^ way);
        if (have == key) return -1;
    }
    return -1;
}
// The searching warp's lookup (all 32 lanes the same context; the table does not change during a search).
__device__ __forceinline__ McLookup mc_lookup(const TgView& t, int a, int b, int lane, const McCache& c) {
    const unsigned long long key = tg_key(a, b);
    const uint32_t h = tg_hash(key) & c.mask;
    const unsigned long long k0 = c.key[h], k1 = c.key[h ^ 1];
    if (k0 == key || k1 == key) {
        const uint32_t slot = k0 == key ? h : h ^ 1, at = slot * c.k + min(lane, c.k - 1);
        McLookup out;
        out.n = c.n[slot];
        out.word = c.word[at];
        out.prob = c.prob[at];
        out.upto = c.upto[at];
        return out;
    }
    const uint32_t slot = k0 == TG_EMPTY || k1 != TG_EMPTY ? h : h ^ 1;
    const McLookup out = mc_read(t, a, b, lane, c, slot);
    __syncwarp();
    if (lane == 0) c.key[slot] = key;
    __syncwarp();
    return out;
}

// a / n for n = 1 .. MC_MAX_ITER + 1, correctly rounded, given the correctly rounded 1 / n: the quotient within one place of the exact
// one, then Markstein's last step ("Computation of elementary functions on the IBM RISC System/6000 processor", 1990).  What could
// overflow or lose bits on the way takes the operator.
__device__ __forceinline__ double mc_div(double a, int n, double rcp) {
    const unsigned hi = (unsigned)__double2hiint(a) & 0x7FFFFFFFu;
    if (hi - 0x06000000u >= 0x78000000u) return a == 0.0 ? a : __ddiv_rn(a, (double)n);      // (zero, |a| < 2^-927, |a| >= 2^993, infinite, NaN)
    const double d = -(double)n;
    double q = __dmul_rn(a, rcp);
    q = __fma_rn(__fma_rn(d, q, a), rcp, q);
    return __fma_rn(__fma_rn(d, q, a), rcp, q);
}

struct McLayout {          // byte offsets in shared memory
    size_t score, prior, mean, er, rcp, list, node, par, queue, key, upto, prob, word, n, u, tok, fpar, dep, nkid, kid, fill, end;
};
__host__ __device__ constexpr McLayout mc_layout(int slots, int k) {
    McLayout l = {};
    size_t at = 0;
    auto take = [&](size_t bytes) { const size_t here = at; at += (bytes + 15) / 16 * 16; return here; };
    l.score = take((size_t)MC_MAX_NODES * 8);                  // sum of scores
    l.prior = take((size_t)MC_MAX_NODES * 8);                  // Eq. 1 probability of the node's token in its parent's context
    l.mean = take((size_t)MC_MAX_NODES * 8);                   // mean score (0 while not visited)
    l.er = take((size_t)(MC_MAX_ITER + 1) * 16);               // E and square root
    l.rcp = take((size_t)(MC_MAX_ITER + 2) * 8);               // 1 / n
    l.list = take((size_t)MC_AHEAD * 8);                       // contexts looked up ahead
    l.node = take((size_t)MC_MAX_NODES * 16);
    l.par = take((size_t)MC_MAX_NODES * 2);
    l.queue = take((size_t)ADED_MAX_NODES * 2);                // breadth-first order of the result
    l.key = take((size_t)slots * 8);
    l.upto = take((size_t)slots * k * 8);
    l.prob = take((size_t)slots * k * 8);
    l.word = take((size_t)slots * k * 4);
    l.n = take((size_t)slots * 4);
    l.u = take((size_t)MC_MAX_ITER * MC_MAX_LEN * 4);          // the caller's uniform numbers
    l.tok = take((size_t)ADED_MAX_NODES * 4);                  // the result (see draft_fill)
    l.fpar = take((size_t)ADED_MAX_NODES * 4);
    l.dep = take((size_t)ADED_MAX_NODES * 4);
    l.nkid = take((size_t)ADED_MAX_NODES * 4);
    l.kid = take((size_t)ADED_MAX_NODES * ADED_DRAFT_MAX_K * 4);
    l.fill = take((size_t)DRAFT_MAX_FILLER * 4);
    l.end = at;
    return l;
}

__global__ void __launch_bounds__(MC_THREADS, 1)
k_mcts_draft(TgView t, const __grid_constant__ McParams p, const int32_t* __restrict__ ctx, const float* __restrict__ u,
             int32_t* __restrict__ out_tok, int32_t* __restrict__ out_par, int32_t* __restrict__ out_n,
             int32_t* __restrict__ sent_tok, double* __restrict__ sent_score, int32_t* __restrict__ out_n_sent,
             int n_target, const int32_t* __restrict__ filler, int n_filler) {
    extern __shared__ __align__(16) uint8_t mc_smem[];
    __shared__ int s_count, s_next, s_nodes;
    __shared__ unsigned long long s_part[MC_WARPS * MC_MAX_K];
    __shared__ uint32_t s_total[MC_WARPS];
    __shared__ int s_slot[MC_WARPS], s_sent[ADED_MAX_NODES];
    __shared__ uint3 s_top[MC_WARPS];
    const McLayout lay = mc_layout(p.slots, p.k);
    double* s_score = reinterpret_cast<double*>(mc_smem + lay.score);
    double* s_prior = reinterpret_cast<double*>(mc_smem + lay.prior);
    double* s_mean = reinterpret_cast<double*>(mc_smem + lay.mean);
    double2* s_er = reinterpret_cast<double2*>(mc_smem + lay.er);
    double* s_rcp = reinterpret_cast<double*>(mc_smem + lay.rcp);
    int2* s_list = reinterpret_cast<int2*>(mc_smem + lay.list);
    int4* s_node = reinterpret_cast<int4*>(mc_smem + lay.node);
    int16_t* s_par = reinterpret_cast<int16_t*>(mc_smem + lay.par);
    int16_t* s_queue = reinterpret_cast<int16_t*>(mc_smem + lay.queue);
    float* s_u = reinterpret_cast<float*>(mc_smem + lay.u);
    int32_t* f_fill = reinterpret_cast<int32_t*>(mc_smem + lay.fill);
    McCache cache;
    cache.key = reinterpret_cast<unsigned long long*>(mc_smem + lay.key);
    cache.upto = reinterpret_cast<unsigned long long*>(mc_smem + lay.upto);
    cache.prob = reinterpret_cast<double*>(mc_smem + lay.prob);
    cache.word = reinterpret_cast<int32_t*>(mc_smem + lay.word);
    cache.n = reinterpret_cast<int32_t*>(mc_smem + lay.n);
    cache.mask = (uint32_t)p.slots - 1;
    cache.k = p.k;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < p.slots; i += MC_THREADS) { cache.key[i] = TG_EMPTY; cache.n[i] = 0; }
    for (int i = tid; i <= MC_MAX_ITER; i += MC_THREADS) {
        s_er[i] = make_double2(p.e_table[i], p.root[i]);
        s_rcp[i + 1] = __ddiv_rn(1.0, (double)(i + 1));
    }
    pdl_enter();
    for (int i = tid; i < p.iterations * p.length; i += MC_THREADS) s_u[i] = u[i];
    if (n_target > 0 && filler)
        for (int i = tid; i < n_filler; i += MC_THREADS) f_fill[i] = filler[i];
    const int prev_token = ctx[0], root_token = ctx[1];
    if (tid == 0) {
        s_node[0] = make_int4(0, root_token, 0, 0);
        s_par[0] = -1;
        s_score[0] = 0.0;
        s_prior[0] = 0.0;
        s_mean[0] = 0.0;
        s_list[0] = make_int2(prev_token, root_token);
        s_count = 1;
        s_next = 1;
    }
    __syncthreads();

    // look up ahead: a level's contexts, by several warps each while they are few (the first may have thousands of continuations)
    for (int lo = 0, level = 0; level < p.length; ++level) {
        const int hi = s_count, n_ctx = hi - lo;
        // A level takes as long as its longest context does, once per MC_WARPS of them; the search meets one of its contexts per iteration.
        // Cold, table of 2,000,000 tokens, three contexts, us: all levels / these / a search by one warp alone.  1 iteration, k = 8: 94, 92, 106 /
        // 41, 70, 22 / 47, 69, 25.  2 iterations, k = 4: 66, 51, 74 / 74, 49, 72 / 64, 92, 39; k = 8: 104, 93, 111 / 62, 57, 29 / 68, 88, 25.
        // 4 iterations, k = 8, sentences of 8: 114, 101, 117 against 211, 189, 209 (these are all levels).
        const int waves = (n_ctx + MC_WARPS - 1) / MC_WARPS;
        if (n_ctx <= 0 || (level > 0 && (p.iterations == 1 || waves > p.iterations))) break;
        const bool deeper = level + 1 < p.length && hi + n_ctx * p.k <= MC_AHEAD;
        auto append = [&](int b, const McLookup& lk) {
            if (!deeper || lk.n == 0) return;
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_next, lk.n);
            at = __shfl_sync(0xffffffffu, at, 0) + lane;
            if (lane < lk.n) s_list[at] = make_int2(b, lk.word);      // (never more than MC_AHEAD: `deeper`)
        };
        int parts = 1;
        while (parts * 2 * n_ctx <= MC_WARPS) parts *= 2;
        if (parts > 1) {
            const int g = warp / parts, part = warp % parts;
            const int2 c = s_list[lo + min(g, n_ctx - 1)];
            if (tid < n_ctx) s_slot[tid] = mc_claim(cache, s_list[lo + tid]);
            unsigned long long best = 0;
            uint32_t total = 0;
            if (g < n_ctx) tg_scan(t, tg_open(t, c.x, c.y, lane), part, parts, p.k, lane, best, total);
            total = __reduce_add_sync(0xffffffffu, total);
            if (lane < MC_MAX_K) s_part[warp * MC_MAX_K + lane] = lane < p.k ? best : 0ull;
            if (lane == 0) s_total[warp] = total;
            __syncthreads();
            if (g < n_ctx && part == 0 && s_slot[g] >= 0) {
                best = 0;
                draft_merge(s_part + warp * MC_MAX_K, parts, p.k, lane, best);
                total = __reduce_add_sync(0xffffffffu, lane < parts ? s_total[warp + lane] : 0u);
                append(c.y, mc_keep(t, c.y, best, total, lane, cache, (uint32_t)s_slot[g]));
            }
        } else {
            for (int i = lo + warp; i < hi; i += MC_WARPS) {
                const int2 c = s_list[i];
                int slot = -1;
                if (lane == 0) slot = mc_claim(cache, c);
                slot = __shfl_sync(0xffffffffu, slot, 0);
                if (slot >= 0) append(c.y, mc_read(t, c.x, c.y, lane, cache, (uint32_t)slot));
            }
        }
        __syncthreads();
        if (tid == 0) s_count = s_next;
        lo = hi;
        __syncthreads();
    }

    if (warp == 0) {
        const int kid_bits = p.k <= 4 ? 2 : 3;              // lanes per node of the path
        int n_nodes = 1;
        for (int it = 0; it < p.iterations; ++it) {
            // the sentence so far: its last two tokens, its score (1 + the probabilities in order), and the tree nodes on it --
            // lane d holds the node at depth d
            int node = 0, len = 1, on_path = 0, depth = 0;
            int before = prev_token, last = root_token;
            double sc = 1.0;
            int4 nd = s_node[0];
            // selection: every node knows which child is next (see below)
            while (mc_kids(nd.z) > 0 && len <= p.length) {      // (a node has children only once it is expanded)
                node = nd.w >> 16;
                nd = s_node[node];
                sc = __dadd_rn(sc, s_prior[node]);
                ++depth;
                if (lane == depth) on_path = node;
                before = last;
                last = nd.y;
                ++len;
            }
            const int link = nd.z;
            // expansion
            if (!(link & MC_EXPANDED) && len <= p.length) {
                const McLookup lk = mc_lookup(t, before, last, lane, cache);
                if (lane == 0) s_node[node].z = n_nodes | lk.n << 16 | MC_EXPANDED;
                if (lane < lk.n) {
                    const int c = n_nodes + lane;
                    s_node[c] = make_int4(0, lk.word, 0, 0);
                    s_par[c] = (int16_t)node;
                    s_score[c] = 0.0;
                    s_mean[c] = 0.0;
                    s_prior[c] = lk.prob;
                }
                __syncwarp();
                if (lk.n > 0) {
                    n_nodes += lk.n;
                    node = n_nodes - 1;                       // the last child created
                    ++depth;
                    if (lane == depth) on_path = node;
                    before = last;
                    last = __shfl_sync(0xffffffffu, lk.word, lk.n - 1);
                    sc = __dadd_rn(sc, __shfl_sync(0xffffffffu, lk.prob, lk.n - 1));
                    ++len;
                }
            }
            // simulation
            for (int draws = 0; len <= p.length; ++draws, ++len) {
                const McLookup lk = mc_lookup(t, before, last, lane, cache);
                if (lk.n == 0) break;
                const unsigned long long total = __shfl_sync(0xffffffffu, lk.upto, lk.n - 1);
                unsigned long long u24 = __float2uint_rd(__fmul_rn(s_u[it * p.length + draws], 16777216.f));
                if (u24 > 16777215ull) u24 = 16777215ull;
                const unsigned long long target = (total * u24) >> 24;
                const unsigned past = __ballot_sync(0xffffffffu, lane < lk.n && lk.upto > target);
                const int pick = past ? __ffs((int)past) - 1 : lk.n - 1;
                before = last;
                last = __shfl_sync(0xffffffffu, lk.word, pick);
                sc = __dadd_rn(sc, __shfl_sync(0xffffffffu, lk.prob, pick));
            }
            // Back propagation, and every path node's next choice.  A choice depends on the node's children and their visits alone, which
            // change only when the node is on the path: it is made now, for all nodes of the path side by side (a lane per child), not one
            // after the other when they are met again (450 cycles a level, nearly all of them the chain of double-precision operations).
            for (int d0 = 0; d0 < depth; d0 += 32 >> kid_bits) {
                const int d = d0 + (lane >> kid_bits), j = lane & ((1 << kid_bits) - 1);
                const int parent = __shfl_sync(0xffffffffu, on_path, d & 31), visited = __shfl_sync(0xffffffffu, on_path, (d + 1) & 31);
                const int4 up = s_node[parent];
                const int first = mc_first(up.z), below = (up.w & 0xFFFF) + 1;
                const bool mine = d < depth && j < mc_kids(up.z);
                const int c = mine ? first + j : 0;
                const double2 er = s_er[min(below, MC_MAX_ITER)];
                double mean = s_mean[c];
                int visits = s_node[c].x;
                const double explore = __dmul_rn(__dmul_rn(er.x, s_prior[c]), er.y);
                if (mine && c == visited) {
                    const double total = __dadd_rn(s_score[c], sc);
                    ++visits;
                    mean = mc_div(total, visits, s_rcp[visits]);
                    s_node[c].x = visits;
                    s_score[c] = total;
                    s_mean[c] = mean;
                }
                const double score = __dadd_rn(mean, mc_div(explore, visits + 1, s_rcp[visits + 1]));
                // the largest score, the earliest child among equals: bits of a double in an order that integers have
                const unsigned long long bits = (unsigned long long)__double_as_longlong(score);
                unsigned long long best = mine ? bits ^ ((bits >> 63) ? ~0ull : 1ull << 63) : 0ull;
                int pick = j;
                for (int o = 1 << kid_bits >> 1; o > 0; o >>= 1) {
                    const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
                    const int who = __shfl_xor_sync(0xffffffffu, pick, o);
                    if (other > best || (other == best && who < pick)) { best = other; pick = who; }
                }
                if (j == 0 && d < depth) s_node[parent].w = below | (first + pick) << 16;
            }
            __syncwarp();
        }
        if (lane == 0) s_nodes = n_nodes;
    }
    __syncthreads();
    const int n_nodes = s_nodes;

    // ranking: leaves of the search tree by mean score (descending), earlier nodes first on ties
    int n_sent = 0;
    auto order = [&](int i) {                        // bits of a leaf's mean in an order that integers have; 0 for other nodes
        const unsigned long long bits = (unsigned long long)__double_as_longlong(s_mean[i] + 0.0);
        return mc_kids(s_node[i].z) != 0 ? 0ull : bits ^ ((bits >> 63) ? ~0ull : 1ull << 63);
    };
    if (n_nodes <= MC_THREADS) {                     // a thread per node counts the leaves in front of it (a round per sentence, below, takes about 0.5 us)
        unsigned long long* s_order = reinterpret_cast<unsigned long long*>(s_score);     // (the sums are not needed any more)
        const unsigned long long mine = tid >= 1 && tid < n_nodes ? order(tid) : 0ull;
        __syncthreads();
        s_order[tid] = mine;
        const int leaves = __syncthreads_count(mine != 0);
        n_sent = min(leaves, p.n_candidates);
        if (mine != 0) {
            int before = 0;
            for (int i = 1; i < n_nodes; ++i) before += s_order[i] > mine || (s_order[i] == mine && i < tid);
            if (before < n_sent) s_sent[before] = tid;
        }
        __syncthreads();
    } else
    for (; n_sent < p.n_candidates; ++n_sent) {
        unsigned long long best = 0;                 // (bits of the mean in an order that integers have: 0 is none)
        int best_i = MC_MAX_NODES;
        for (int i = 1 + tid; i < n_nodes; i += MC_THREADS) {
            const unsigned long long ord = s_node[i].z & MC_CHOSEN ? 0ull : order(i);
            if (ord > best) { best = ord; best_i = i; }     // i ascends within a thread: first wins ties
        }
        auto top = [&]() {                           // over the warp, in every lane
            const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32));
            const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
            const unsigned long long all = (unsigned long long)hi << 32 | lo;
            best_i = (int)__reduce_min_sync(0xffffffffu, best == all ? (unsigned)best_i : (unsigned)MC_MAX_NODES);
            best = all;
        };
        top();
        if (lane == 0) s_top[warp] = make_uint3((unsigned)(best >> 32), (unsigned)best, (unsigned)best_i);
        __syncthreads();
        const uint3 other = s_top[lane & (MC_WARPS - 1)];
        best = (unsigned long long)other.x << 32 | other.y;
        best_i = (int)other.z;
        top();
        if (best == 0) break;                        // (every thread has the same answer)
        if (tid == 0) {
            s_node[best_i].z |= MC_CHOSEN;
            s_sent[n_sent] = best_i;
        }
        __syncthreads();
    }
    for (int r = tid; r < n_sent; r += MC_THREADS) {
        int d = 0;
        for (int j = s_sent[r]; j > 0; j = s_par[j]) { atomicOr(&s_node[j].z, MC_KEPT); ++d; }
        for (int e = d; e < p.length; ++e) sent_tok[r * p.length + e] = -1;
        for (int j = s_sent[r]; j > 0; j = s_par[j]) sent_tok[r * p.length + --d] = s_node[j].y;
        sent_score[r] = s_mean[s_sent[r]];
    }
    __syncthreads();
    if (warp != 0) return;
    // prefix tree of the chosen sentences, breadth first, children in creation order: 32 nodes' children at a time
    int32_t* f_tok = reinterpret_cast<int32_t*>(mc_smem + lay.tok);          // [ADED_MAX_NODES] each
    int32_t* f_par = reinterpret_cast<int32_t*>(mc_smem + lay.fpar);
    int32_t* f_dep = reinterpret_cast<int32_t*>(mc_smem + lay.dep);
    int32_t* f_nkid = reinterpret_cast<int32_t*>(mc_smem + lay.nkid);
    int32_t* f_kid = reinterpret_cast<int32_t*>(mc_smem + lay.kid);          // [ADED_MAX_NODES][ADED_DRAFT_MAX_K]
    if (lane == 0) {
        s_queue[0] = 0;
        f_tok[0] = root_token;
        f_par[0] = -1;
        f_dep[0] = 0;
    }
    __syncwarp();
    int count = 1;
    for (int head0 = 0; head0 < count; ) {
        const int head = head0 + lane, heads = min(32, count - head0);
        int first = 0, nk = 0, mine = 0;
        if (lane < heads) {
            const int link = s_node[s_queue[head]].z;
            first = mc_first(link);
            nk = mc_kids(link);
            for (int c = 0; c < nk; ++c) mine += (s_node[first + c].z & MC_KEPT) != 0;
        }
        int upto = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int other = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += other;
        }
        int at = count + upto - mine, kept = 0;
        if (lane < heads) {
            for (int c = 0; c < nk; ++c) {
                const int4 nd = s_node[first + c];
                if (!(nd.z & MC_KEPT) || at >= ADED_MAX_NODES) continue;
                s_queue[at] = (int16_t)(first + c);
                f_tok[at] = nd.y;
                f_par[at] = head;
                f_dep[at] = f_dep[head] + 1;
                f_kid[head * ADED_DRAFT_MAX_K + kept++] = nd.y;
                ++at;
            }
            f_nkid[head] = kept;
        }
        count = min(ADED_MAX_NODES, count + __shfl_sync(0xffffffffu, upto, 31));
        head0 += heads;
        __syncwarp();
    }
    bool fail = false;
    if (n_target > count && filler) {
        // complete the prefix tree to a fixed number of nodes, by the rule of the draft-tree kernel
        count = draft_fill(f_tok, f_par, f_dep, f_nkid, f_kid, count, n_target, p.length, p.k, f_fill, n_filler, t.vocab, lane, reinterpret_cast<int16_t*>(s_list), &fail);
        __syncwarp();
        if (fail && lane == 0) { atomicCAS(t.status, 0, (int)ADED_ERR_INVALID_ARG); f_tok[0] = -1; }
        __syncwarp();
    }
    for (int i = lane; i < count; i += 32) {
        out_tok[i] = f_tok[i];
        out_par[i] = f_par[i];
    }
    if (lane == 0) {
        *out_n = count;
        *out_n_sent = n_sent;
    }
}

static int mc_smem_bytes(int slots, int k) { return (int)mc_layout(slots, k).end; }
static int mc_smem_most() {
    int most = 0;
    for (int k = 1; k <= MC_MAX_K; ++k) most = mc_smem_bytes(mc_slots(k), k) > most ? mc_smem_bytes(mc_slots(k), k) : most;
    return most;
}

}  // namespace aded

struct aded_trigram {
    aded_trigram_config cfg;
    int device;
    aded::TgView view;
    int32_t* stage_i;    // staging for the _host entry points
    uint32_t* stage_u;
    size_t stage_n;
    unsigned long long* stats_dev;
    int32_t* step_i;     // decoding step: see STEP_SENT
    mutable bool search_prepared;   // the tree search's shared-memory limit has been raised on this device
    uint64_t counted;    // windows and entries given to update and import since the table was empty (a decoding step's few are left out)
};

using namespace aded;

static constexpr size_t TG_STAGE = 1 << 16;
// step_i layout: sentences of the search, nodes from the table, filler staging
static constexpr int STEP_SENT = 0, STEP_REAL = 1, STEP_FILL = 2;
static constexpr int STEP_INTS = STEP_FILL + DRAFT_MAX_FILLER;

// Tokens of text that the table holds, as far as a call knows without asking the device: what it was given, but no more than its home buckets
// are meant for (half as many).  By its size alone, a table of 2^24 buckets that held 10^5 tokens took 21 us instead of 10 for 4096 lookups.
static uint64_t topk_text(const aded_trigram* t) {
    const uint64_t room = t->view.n_home / 2;
    return t->counted < room ? t->counted : room;
}

// An empty table: home buckets and index.  The pool needs no clearing: see tg_place.
static aded_status tg_reset(aded_trigram* t, cudaStream_t st) {
    t->counted = 0;
    const size_t buckets = (size_t)t->view.n_home + (t->view.chain ? t->view.n_over : 0);     // (chain buckets follow the home buckets)
    static_assert(sizeof(TgIndexSlot) == sizeof(uint4), "a slot per store");
    const size_t parts = buckets * (sizeof(Bucket) / sizeof(uint4)), slots = t->view.index ? (size_t)(t->view.index_mask + 1) : 0;
    const size_t blocks = ((parts > slots ? parts : slots) + 511) / 512;
    k_tg_init<<<(unsigned)(blocks < 2048 ? blocks : 2048), 512, 0, st>>>(reinterpret_cast<uint4*>(t->view.buckets), parts, reinterpret_cast<uint4*>(t->view.index),
                                                                       slots, t->view.used);
    ADED_CUDA_TRY(cudaGetLastError());
    return ADED_OK;
}

extern "C" {

aded_status aded_trigram_create(const aded_trigram_config* cfg, aded_trigram** out) {
    if (!cfg || !out) return ADED_ERR_INVALID_ARG;
    *out = nullptr;
    if (cfg->vocab < 1 || cfg->log2_buckets < 4 || cfg->log2_buckets > 28 || cfg->overflow_buckets < 0)
        return ADED_ERR_INVALID_ARG;
    if (cfg->cap > 0x7fffffffu) return ADED_ERR_INVALID_ARG;     // counts are kept below 2^31 so that concurrent adds cannot wrap
    aded_trigram* t = new (std::nothrow) aded_trigram();
    if (!t) return ADED_ERR_OOM;
    t->cfg = *cfg;
    t->stage_i = nullptr;
    t->stage_u = nullptr;
    t->stats_dev = nullptr;
    t->step_i = nullptr;
    t->search_prepared = false;
    t->view = TgView();
    const size_t n_home = (size_t)1 << cfg->log2_buckets, n_over = (size_t)cfg->overflow_buckets;
    bool ok = cudaGetDevice(&t->device) == cudaSuccess;
    cudaError_t e = cudaSuccess;
    // one allocation: home buckets, index and pool (or, where the device has no room for those, or they number more than 32-bit
    // units, chain buckets), then the small arrays (every part a multiple of 64 bytes)
    size_t n_units = (size_t)tg_pool_units(n_over), n_index = (size_t)tg_index_slots(n_over), at[9] = {0};
    bool chained = n_units > 0xFFFFFFF0ull;
    char* block = nullptr;
    for (;; chained = true) {
        if (chained) n_units = n_index = 0;
        const size_t parts[8] = {(n_home + (chained ? n_over : 0)) * sizeof(Bucket), n_index * sizeof(TgIndexSlot), n_units * TG_UNIT * sizeof(TgSlot),
                                 TG_STAGE * sizeof(int32_t), TG_STAGE * sizeof(uint32_t), STEP_INTS * sizeof(int32_t),
                                 2 * sizeof(unsigned long long), 4 * sizeof(uint32_t)};
        for (int i = 0; i < 8; ++i) at[i + 1] = at[i] + (parts[i] + 63) / 64 * 64;
        if (ok) { e = cudaMalloc((void**)&block, at[8]); ok = e == cudaSuccess; }
        if (ok || chained || e != cudaErrorMemoryAllocation) break;
        cudaGetLastError();
        ok = true;
    }
    if (ok) {
        t->view.buckets = reinterpret_cast<Bucket*>(block + at[0]);
        if (chained) {
            t->view.chain = t->view.buckets + n_home;
        } else {
            t->view.index = reinterpret_cast<TgIndexSlot*>(block + at[1]);
            t->view.pool = reinterpret_cast<TgSlot*>(block + at[2]);
        }
        t->stage_i = reinterpret_cast<int32_t*>(block + at[3]);
        t->stage_u = reinterpret_cast<uint32_t*>(block + at[4]);
        t->step_i = reinterpret_cast<int32_t*>(block + at[5]);
        t->stats_dev = reinterpret_cast<unsigned long long*>(block + at[6]);
        t->view.used = reinterpret_cast<uint32_t*>(block + at[7]);
        t->view.status = reinterpret_cast<int32_t*>(t->view.used + 2);
    }
    if (!ok) {
        cudaGetLastError();
        aded_trigram_destroy(t);
        return e == cudaErrorMemoryAllocation ? ADED_ERR_OOM : ADED_ERR_CUDA;
    }
    t->view.n_home = (uint32_t)n_home;
    t->view.n_home_mask = (uint32_t)n_home - 1;
    t->view.n_over = (uint32_t)cfg->overflow_buckets;
    t->view.n_units = (uint32_t)n_units;
    t->view.index_mask = chained ? 0 : n_index - 1;
    t->view.vocab = cfg->vocab;
    t->view.cap = cfg->cap == 0 ? 0x7fffffffu : cfg->cap;
    t->view.min_count = cfg->min_count;
    ok = tg_reset(t, nullptr) == ADED_OK &&
         cudaMemset(t->view.status, 0, sizeof(int32_t)) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        aded_trigram_destroy(t);
        return ADED_ERR_CUDA;
    }
    *out = t;
    return ADED_OK;
}

aded_status aded_trigram_destroy(aded_trigram* t) {
    if (!t) return ADED_ERR_INVALID_ARG;
    if (t->view.buckets) cudaFree(t->view.buckets);     // (the first part of the handle's one allocation)
    delete t;
    return ADED_OK;
}

aded_status aded_trigram_update(aded_trigram* t, const int32_t* tokens_dev, int32_t n, void* stream) {
    if (!t || n < 0 || (n > 0 && !tokens_dev)) return ADED_ERR_INVALID_ARG;
    if (n < 3) return ADED_OK;
    const int windows = n - 2;
    t->counted += (uint64_t)windows;
    note_launch();
    if (windows >= BULK_MIN)
        k_tg_update_bulk<<<(unsigned)(((int64_t)windows + BULK_WINDOWS - 1) / BULK_WINDOWS), BULK_THREADS, (BULK_WINDOWS + 2 + 2 * BULK_SLOTS) * sizeof(int32_t),
                           static_cast<cudaStream_t>(stream)>>>(t->view, tokens_dev, windows);
    else
        k_tg_update<<<(windows + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(t->view, tokens_dev, n);
    ADED_CUDA_TRY(cudaGetLastError());
    return ADED_OK;
}

aded_status aded_trigram_update_host(aded_trigram* t, const int32_t* tokens_host, int32_t n, void* stream) {
    if (!t || n < 0 || (n > 0 && !tokens_host)) return ADED_ERR_INVALID_ARG;
    if (n < 3) return ADED_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // long spans go through the staging buffer in pieces that overlap by two tokens
    for (int64_t lo = 0; lo + 2 < n; lo += (int64_t)TG_STAGE - 2) {
        const int64_t m = n - lo < (int64_t)TG_STAGE ? n - lo : (int64_t)TG_STAGE;
        ADED_CUDA_TRY(cudaMemcpyAsync(t->stage_i, tokens_host + lo, m * sizeof(int32_t), cudaMemcpyHostToDevice, st));
        aded_status s = aded_trigram_update(t, t->stage_i, (int32_t)m, stream);
        if (s != ADED_OK) return s;
        ADED_CUDA_TRY(cudaStreamSynchronize(st));
    }
    return ADED_OK;
}

aded_status aded_trigram_topk(const aded_trigram* t, const int32_t* ctx_dev, int32_t q, int32_t k,
                              int32_t* out_tokens_dev, uint32_t* out_counts_dev, uint32_t* out_total_dev,
                              void* stream) {
    if (!t || q < 0 || k < 1 || k > 32) return ADED_ERR_INVALID_ARG;
    if (q == 0) return ADED_OK;
    if (!ctx_dev || !out_tokens_dev || !out_counts_dev) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // As many queries per block as fill the device's block slots once (three blocks per SM).
    const int wave = ws_grid_limit(t->device) / 2 * 3;
    int per_block = (int)(((int64_t)q + wave - 1) / wave);
    if (q >= topk_bulk_min(topk_text(t)) && k >= 2) {
        uint32_t slots = 1;
        while ((uint64_t)slots * 2 < (uint64_t)q) slots *= 2;
        const int deferred = (int)((slots + k - 1) / k);             // rows whose counts the hash table lies in
        per_block = per_block > TOPK_LEAD_QUERIES ? TOPK_LEAD_QUERIES : per_block;
        ADED_CUDA_TRY(cudaMemsetAsync(out_counts_dev, 0xFF, (size_t)slots * sizeof(uint32_t), st));
        note_launch(3);
        const int lead_blocks = (int)(((int64_t)q + per_block - 1) / per_block);
        const uintptr_t low = reinterpret_cast<uintptr_t>(out_tokens_dev) | reinterpret_cast<uintptr_t>(out_counts_dev);
        const int vec = k % 4 == 0 && low % 16 == 0 ? 4 : k % 2 == 0 && low % 8 == 0 ? 2 : 1;      // words of a row that one load or store takes
        launch_k(k_topk_mark, dim3((unsigned)(((int64_t)q + MARK_THREADS - 1) / MARK_THREADS)), dim3(MARK_THREADS), 0, st, t->view, ctx_dev, q, k, vec, slots - 1,
                 deferred, out_tokens_dev, out_counts_dev, out_total_dev);
        launch_k(k_topk_lead, dim3(lead_blocks), dim3(TOPK_THREADS), 0, st, t->view, q, k, vec, per_block, out_tokens_dev, out_counts_dev, out_total_dev);
        const dim3 grid((unsigned)(((int64_t)q + 255) / 256));
        if (vec == 4)
            launch_k(k_topk_copy<int4>, grid, dim3(256), 0, st, q, k, reinterpret_cast<int4*>(out_tokens_dev), reinterpret_cast<int4*>(out_counts_dev), out_total_dev);
        else if (vec == 2)
            launch_k(k_topk_copy<int2>, grid, dim3(256), 0, st, q, k, reinterpret_cast<int2*>(out_tokens_dev), reinterpret_cast<int2*>(out_counts_dev), out_total_dev);
        else
            launch_k(k_topk_copy<int32_t>, grid, dim3(256), 0, st, q, k, out_tokens_dev, reinterpret_cast<int32_t*>(out_counts_dev), out_total_dev);
        ADED_CUDA_TRY(cudaGetLastError());
        return ADED_OK;
    }
    per_block = per_block > TOPK_MAX_QUERIES ? TOPK_MAX_QUERIES : per_block;
    // (the limit is the device's, not the process's; blocks of so many queries come from k = 1 and some 700,000 of them only)
    if (topk_smem(per_block) > 40 * 1024)
        ADED_CUDA_TRY(cudaFuncSetAttribute(k_tg_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)topk_smem(TOPK_MAX_QUERIES)));
    note_launch();
    k_tg_topk<<<(unsigned)(((int64_t)q + per_block - 1) / per_block), TOPK_THREADS, topk_smem(per_block), st>>>(
        t->view, ctx_dev, q, k, per_block, out_tokens_dev, out_counts_dev, out_total_dev);
    ADED_CUDA_TRY(cudaGetLastError());
    return ADED_OK;
}

aded_status aded_trigram_topk_host(const aded_trigram* t, const int32_t* ctx_host, int32_t q, int32_t k,
                                   int32_t* out_tokens_host, uint32_t* out_counts_host, uint32_t* out_total_host,
                                   void* stream) {
    if (!t || q < 0 || k < 1 || k > 32) return ADED_ERR_INVALID_ARG;
    if (q == 0) return ADED_OK;
    if (!ctx_host || !out_tokens_host || !out_counts_host) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // staging: [ctx 2*qq | tokens qq*k] in stage_i, [counts qq*k | totals qq] in stage_u
    const int per = (int)(TG_STAGE / (size_t)(k + 2));
    for (int lo = 0; lo < q; lo += per) {
        const int qq = q - lo < per ? q - lo : per;
        int32_t* ctx_d = t->stage_i;
        int32_t* tok_d = t->stage_i + 2 * qq;
        uint32_t* cnt_d = t->stage_u;
        uint32_t* tot_d = t->stage_u + (size_t)qq * k;
        ADED_CUDA_TRY(cudaMemcpyAsync(ctx_d, ctx_host + 2 * (size_t)lo, 2 * (size_t)qq * sizeof(int32_t), cudaMemcpyHostToDevice, st));
        aded_status s = aded_trigram_topk(t, ctx_d, qq, k, tok_d, cnt_d, tot_d, stream);
        if (s != ADED_OK) return s;
        ADED_CUDA_TRY(cudaMemcpyAsync(out_tokens_host + (size_t)lo * k, tok_d, (size_t)qq * k * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        ADED_CUDA_TRY(cudaMemcpyAsync(out_counts_host + (size_t)lo * k, cnt_d, (size_t)qq * k * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
        if (out_total_host)
            ADED_CUDA_TRY(cudaMemcpyAsync(out_total_host + lo, tot_d, (size_t)qq * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
        ADED_CUDA_TRY(cudaStreamSynchronize(st));
    }
    return ADED_OK;
}

aded_status aded_draft_tree(const aded_trigram* t, const int32_t* context_dev, int32_t n_nodes, int32_t max_depth,
                            int32_t k, const int32_t* filler_dev, int32_t n_filler, int32_t* tree_tokens_dev,
                            int32_t* tree_parents_dev, int32_t* n_from_table_dev, void* stream) {
    if (!t || !context_dev || !tree_tokens_dev || !tree_parents_dev) return ADED_ERR_INVALID_ARG;
    if (n_nodes < 1 || n_nodes > ADED_MAX_NODES || max_depth < 0 || k < 1 || k > ADED_DRAFT_MAX_K) return ADED_ERR_INVALID_ARG;
    if (n_filler < 0 || n_filler > DRAFT_MAX_FILLER || (n_filler > 0 && !filler_dev)) return ADED_ERR_INVALID_ARG;
    note_launch();
    ADED_CUDA_TRY(launch_k(k_draft_tree, 1, 1024, 0, static_cast<cudaStream_t>(stream), t->view, context_dev, n_nodes, max_depth, k,
                           n_filler > 0 ? filler_dev : nullptr, n_filler, tree_tokens_dev, tree_parents_dev, n_from_table_dev));
    return ADED_OK;
}

aded_status aded_mcts_draft(const aded_trigram* t, const int32_t* context_dev, int32_t iterations, int32_t length,
                            int32_t n_candidates, int32_t k, float c1, float c2, const float* u_dev, int32_t* tree_tokens_dev,
                            int32_t* tree_parents_dev, int32_t* n_nodes_dev, int32_t* sentence_tokens_dev,
                            double* sentence_scores_dev, int32_t* n_sentences_dev, int32_t n_nodes_target,
                            const int32_t* filler_dev, int32_t n_filler, void* stream) {
    if (!t || !context_dev || !u_dev || !tree_tokens_dev || !tree_parents_dev || !n_nodes_dev || !sentence_tokens_dev ||
        !sentence_scores_dev || !n_sentences_dev)
        return ADED_ERR_INVALID_ARG;
    if (n_nodes_target < 0 || n_nodes_target > ADED_MAX_NODES || n_filler < 0 || n_filler > DRAFT_MAX_FILLER ||
        (n_nodes_target > 0 && (!filler_dev || n_filler < 1)))
        return ADED_ERR_INVALID_ARG;
    if (iterations < 1 || iterations > MC_MAX_ITER || length < 1 || length > MC_MAX_LEN || k < 1 || k > MC_MAX_K ||
        n_candidates < 1 || n_candidates * length + 1 > ADED_MAX_NODES || !(c2 > 0.f))
        return ADED_ERR_INVALID_ARG;
    if (!t->search_prepared) {      // (per handle: the limit is the device's, and a handle belongs to one)
        ADED_CUDA_TRY(cudaFuncSetAttribute(k_mcts_draft, cudaFuncAttributeMaxDynamicSharedMemorySize, mc_smem_most()));
        t->search_prepared = true;
    }
    McParams p;
    p.iterations = iterations;
    p.length = length;
    p.n_candidates = n_candidates;
    p.k = k;
    p.slots = mc_slots(k);
    for (int n = 0; n <= MC_MAX_ITER; ++n) p.e_table[n] = (double)c1 + std::log(((double)n + (double)c2 + 1.0) / (double)c2);   // Eq. 3
    for (int n = 0; n <= MC_MAX_ITER; ++n) p.root[n] = std::sqrt((double)n);
    note_launch();
    ADED_CUDA_TRY(launch_k(k_mcts_draft, 1, MC_THREADS, mc_smem_bytes(p.slots, k), static_cast<cudaStream_t>(stream), t->view, p, context_dev, u_dev, tree_tokens_dev,
                           tree_parents_dev, n_nodes_dev, sentence_tokens_dev, sentence_scores_dev, n_sentences_dev, n_nodes_target,
                           n_nodes_target > 0 ? filler_dev : nullptr, n_filler));
    return ADED_OK;
}

aded_status aded_decode_step(aded_model* m, aded_kv* kv, aded_trigram* t, int32_t* context_dev, int32_t n_nodes,
                             int32_t max_depth, int32_t k, const int32_t* filler_dev, int32_t n_filler,
                             int32_t* out_tokens_dev, int32_t* out_accept_len_dev, int32_t* n_from_table_dev,
                             void* stream) {
    if (!m || !kv || !t || !context_dev || !out_tokens_dev || !out_accept_len_dev) return ADED_ERR_INVALID_ARG;
    if (n_nodes < 1 || n_nodes > ADED_MAX_NODES || n_nodes > m->cfg.max_rows) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    aded_status s = aded_draft_tree(t, context_dev, n_nodes, max_depth, k, filler_dev, n_filler, m->tokens, m->parents,
                                    n_from_table_dev ? n_from_table_dev : t->step_i + STEP_REAL, stream);
    if (s != ADED_OK) return s;
    s = aded_verify(m, kv, m->tokens, m->parents, n_nodes, out_tokens_dev, out_accept_len_dev, stream);
    if (s != ADED_OK) return s;
    note_launch();
    ADED_CUDA_TRY(launch_k(k_decode_feedback, 1, FEEDBACK_THREADS, 0, st, t->view, out_tokens_dev, out_accept_len_dev, context_dev, n_nodes));
    return ADED_OK;
}

aded_status aded_decode_step_mcts(aded_model* m, aded_kv* kv, aded_trigram* t, int32_t* context_dev, int32_t n_nodes,
                                  int32_t iterations, int32_t length, int32_t n_candidates, int32_t k, float c1, float c2,
                                  const float* u_dev, const int32_t* filler_dev, int32_t n_filler, int32_t* out_tokens_dev,
                                  int32_t* out_accept_len_dev, void* stream) {
    if (!m || !kv || !t || !context_dev || !out_tokens_dev || !out_accept_len_dev) return ADED_ERR_INVALID_ARG;
    if (n_nodes < 1 || n_nodes > ADED_MAX_NODES || n_nodes > m->cfg.max_rows) return ADED_ERR_INVALID_ARG;
    if (!m->step_mcts) {      // sentences and counts of the search, which a decoding step does not hand out
        void* p = nullptr;
        ADED_CUDA_TRY(cudaMalloc(&p, (size_t)ADED_MAX_NODES * (sizeof(int32_t) + sizeof(double)) + 64));
        m->step_mcts = p;
        m->owned.push_back(p);
    }
    double* scores = reinterpret_cast<double*>(m->step_mcts);
    int32_t* sent = reinterpret_cast<int32_t*>(scores + ADED_MAX_NODES);
    int32_t* counts = t->step_i + STEP_REAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    aded_status s = aded_mcts_draft(t, context_dev, iterations, length, n_candidates, k, c1, c2, u_dev, m->tokens, m->parents, counts,
                                    sent, scores, t->step_i + STEP_SENT, n_nodes, filler_dev, n_filler, stream);
    if (s != ADED_OK) return s;
    s = aded_verify(m, kv, m->tokens, m->parents, n_nodes, out_tokens_dev, out_accept_len_dev, stream);
    if (s != ADED_OK) return s;
    note_launch();
    ADED_CUDA_TRY(launch_k(k_decode_feedback, 1, FEEDBACK_THREADS, 0, st, t->view, out_tokens_dev, out_accept_len_dev, context_dev, n_nodes));
    return ADED_OK;
}

aded_status aded_decode_step_host(aded_model* m, aded_kv* kv, aded_trigram* t, int32_t* context_dev, int32_t n_nodes,
                                  int32_t max_depth, int32_t k, const int32_t* filler_host, int32_t n_filler,
                                  int32_t* out_tokens_host, int32_t* out_accept_len_host, void* stream) {
    if (!m || !t || !out_tokens_host || !out_accept_len_host) return ADED_ERR_INVALID_ARG;
    if (n_filler < 0 || n_filler > DRAFT_MAX_FILLER || (n_filler > 0 && !filler_host)) return ADED_ERR_INVALID_ARG;
    if (n_nodes < 1 || n_nodes > m->cfg.max_rows) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (n_filler > 0)
        ADED_CUDA_TRY(cudaMemcpyAsync(t->step_i + STEP_FILL, filler_host, (size_t)n_filler * sizeof(int32_t),
                                      cudaMemcpyHostToDevice, st));
    const aded_status s = aded_decode_step(m, kv, t, context_dev, n_nodes, max_depth, k, t->step_i + STEP_FILL, n_filler,
                                           m->out_tokens, m->out_len, nullptr, stream);
    if (s != ADED_OK) return s;
    ADED_CUDA_TRY(cudaMemcpyAsync(out_tokens_host, m->out_tokens, (size_t)n_nodes * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    ADED_CUDA_TRY(cudaMemcpyAsync(out_accept_len_host, m->out_len, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    ADED_CUDA_TRY(cudaStreamSynchronize(st));
    return ADED_OK;
}

// ---- persistence and pruning -----------------------------------------------------------------------
aded_status aded_trigram_export(const aded_trigram* t, uint32_t min_count, int32_t* keys_dev, uint32_t* counts_dev,
                                uint64_t max_entries, uint64_t* n_out_host, void* stream) {
    if (!t || !n_out_host || (max_entries > 0 && (!keys_dev || !counts_dev))) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned long long n = 0;
    ADED_CUDA_TRY(cudaMemsetAsync(t->stats_dev, 0, sizeof n, st));
    note_launch();
    k_tg_export<<<1024, EXPORT_THREADS, 0, st>>>(t->view, min_count, keys_dev, counts_dev, max_entries, t->stats_dev);
    ADED_CUDA_TRY(cudaMemcpyAsync(&n, t->stats_dev, sizeof n, cudaMemcpyDeviceToHost, st));
    ADED_CUDA_TRY(cudaStreamSynchronize(st));
    *n_out_host = n;
    return ADED_OK;
}

aded_status aded_trigram_import(aded_trigram* t, const int32_t* keys_dev, const uint32_t* counts_dev, uint64_t n, void* stream) {
    if (!t || (n > 0 && (!keys_dev || !counts_dev))) return ADED_ERR_INVALID_ARG;
    if (n == 0) return ADED_OK;
    t->counted += n;
    note_launch();
    k_tg_import<<<(unsigned int)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(t->view, keys_dev, counts_dev, n);
    ADED_CUDA_TRY(cudaGetLastError());
    return ADED_OK;
}

aded_status aded_trigram_clear(aded_trigram* t, void* stream) {
    if (!t) return ADED_ERR_INVALID_ARG;
    note_launch();
    return tg_reset(t, static_cast<cudaStream_t>(stream));
}

// Scratch copy of the entries with count >= min_count; the caller frees *keys / *counts.
static aded_status tg_snapshot(const aded_trigram* t, uint32_t min_count, int32_t** keys, uint32_t** counts, uint64_t* n, void* stream) {
    *keys = nullptr;
    *counts = nullptr;
    uint64_t total = 0;
    aded_status s = aded_trigram_export(t, min_count, nullptr, nullptr, 0, &total, stream);
    if (s != ADED_OK) return s;
    *n = total;
    if (total == 0) return ADED_OK;
    if (cudaMalloc((void**)keys, total * 3 * sizeof(int32_t)) != cudaSuccess || cudaMalloc((void**)counts, total * sizeof(uint32_t)) != cudaSuccess) {
        cudaGetLastError();
        if (*keys) cudaFree(*keys);
        *keys = nullptr;
        return ADED_ERR_OOM;
    }
    uint64_t again = 0;
    s = aded_trigram_export(t, min_count, *keys, *counts, total, &again, stream);
    if (s == ADED_OK && again != total) s = ADED_ERR_INVALID_ARG;     // the table changed between the two passes
    if (s != ADED_OK) { cudaFree(*keys); cudaFree(*counts); *keys = nullptr; *counts = nullptr; }
    return s;
}

aded_status aded_trigram_prune(aded_trigram* t, uint32_t min_count, void* stream) {
    if (!t) return ADED_ERR_INVALID_ARG;
    int32_t* keys;
    uint32_t* counts;
    uint64_t n;
    aded_status s = tg_snapshot(t, min_count, &keys, &counts, &n, stream);
    if (s != ADED_OK) return s;
    s = aded_trigram_clear(t, stream);
    if (s == ADED_OK) s = aded_trigram_import(t, keys, counts, n, stream);
    cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (keys) cudaFree(keys);
    if (counts) cudaFree(counts);
    return s;
}

static const char TG_MAGIC[8] = {'A', 'D', 'E', 'D', 'T', 'G', '0', '1'};

aded_status aded_trigram_save(const aded_trigram* t, const char* path, void* stream) {
    if (!t || !path) return ADED_ERR_INVALID_ARG;
    int32_t* keys;
    uint32_t* counts;
    uint64_t n;
    aded_status s = tg_snapshot(t, 0, &keys, &counts, &n, stream);
    if (s != ADED_OK) return s;
    std::vector<int32_t> hk(n * 3);
    std::vector<uint32_t> hc(n);
    bool ok = true;
    if (n) {
        ok = cudaMemcpy(hk.data(), keys, n * 3 * sizeof(int32_t), cudaMemcpyDeviceToHost) == cudaSuccess &&
             cudaMemcpy(hc.data(), counts, n * sizeof(uint32_t), cudaMemcpyDeviceToHost) == cudaSuccess;
        cudaFree(keys);
        cudaFree(counts);
    }
    if (!ok) { cudaGetLastError(); return ADED_ERR_CUDA; }
    FILE* f = fopen(path, "wb");
    if (!f) return ADED_ERR_INVALID_ARG;
    const int32_t vocab = t->cfg.vocab;
    ok = fwrite(TG_MAGIC, 1, 8, f) == 8 && fwrite(&vocab, sizeof vocab, 1, f) == 1 && fwrite(&n, sizeof n, 1, f) == 1 &&
         (n == 0 || (fwrite(hk.data(), sizeof(int32_t), n * 3, f) == n * 3 && fwrite(hc.data(), sizeof(uint32_t), n, f) == n));
    ok = (fclose(f) == 0) && ok;
    return ok ? ADED_OK : ADED_ERR_INVALID_ARG;
}

aded_status aded_trigram_load(aded_trigram* t, const char* path, void* stream) {
    if (!t || !path) return ADED_ERR_INVALID_ARG;
    FILE* f = fopen(path, "rb");
    if (!f) return ADED_ERR_INVALID_ARG;
    char magic[8];
    int32_t vocab = 0;
    uint64_t n = 0;
    bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, TG_MAGIC, 8) == 0 && fread(&vocab, sizeof vocab, 1, f) == 1 &&
              fread(&n, sizeof n, 1, f) == 1 && vocab == t->cfg.vocab && n <= ((uint64_t)1 << 34);
    std::vector<int32_t> hk;
    std::vector<uint32_t> hc;
    if (ok && n) {
        hk.resize(n * 3);
        hc.resize(n);
        ok = fread(hk.data(), sizeof(int32_t), n * 3, f) == n * 3 && fread(hc.data(), sizeof(uint32_t), n, f) == n;
    }
    fclose(f);
    if (!ok) return ADED_ERR_INVALID_ARG;
    if (n == 0) return ADED_OK;
    int32_t* keys = nullptr;
    uint32_t* counts = nullptr;
    if (cudaMalloc((void**)&keys, n * 3 * sizeof(int32_t)) != cudaSuccess || cudaMalloc((void**)&counts, n * sizeof(uint32_t)) != cudaSuccess) {
        cudaGetLastError();
        if (keys) cudaFree(keys);
        return ADED_ERR_OOM;
    }
    aded_status s = ADED_OK;
    if (cudaMemcpy(keys, hk.data(), n * 3 * sizeof(int32_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(counts, hc.data(), n * sizeof(uint32_t), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        s = ADED_ERR_CUDA;
    }
    if (s == ADED_OK) s = aded_trigram_import(t, keys, counts, n, stream);
    cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    cudaFree(keys);
    cudaFree(counts);
    return s;
}

aded_status aded_trigram_get(const aded_trigram* t, int32_t a, int32_t b, int32_t c, uint32_t* out_count_host, void* stream) {
    if (!t || !out_count_host) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_tg_get<<<1, 1, 0, st>>>(t->view, a, b, c, t->stage_u);
    ADED_CUDA_TRY(cudaMemcpyAsync(out_count_host, t->stage_u, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    ADED_CUDA_TRY(cudaStreamSynchronize(st));
    return ADED_OK;
}

aded_status aded_trigram_stats(const aded_trigram* t, uint64_t* out_entries_host, uint64_t* out_buckets_host, void* stream) {
    if (!t || !out_entries_host || !out_buckets_host) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned long long res[2] = {0, 0};
    ADED_CUDA_TRY(cudaMemsetAsync(t->stats_dev, 0, sizeof res, st));
    k_tg_stats<<<1024, 256, 0, st>>>(t->view, t->stats_dev);
    ADED_CUDA_TRY(cudaMemcpyAsync(res, t->stats_dev, sizeof res, cudaMemcpyDeviceToHost, st));
    ADED_CUDA_TRY(cudaStreamSynchronize(st));
    *out_entries_host = res[0];
    *out_buckets_host = res[1];
    return ADED_OK;
}

aded_status aded_trigram_poll_status(aded_trigram* t, aded_status* out_host, void* stream) {
    if (!t || !out_host) return ADED_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t v = 0;
    ADED_CUDA_TRY(cudaMemcpyAsync(&v, t->view.status, sizeof v, cudaMemcpyDeviceToHost, st));
    ADED_CUDA_TRY(cudaStreamSynchronize(st));
    if (v != 0) {
        ADED_CUDA_TRY(cudaMemsetAsync(t->view.status, 0, sizeof v, st));
        ADED_CUDA_TRY(cudaStreamSynchronize(st));
    }
    *out_host = static_cast<aded_status>(v);
    return ADED_OK;
}

}  // extern "C"
