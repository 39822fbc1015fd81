// The tri-gram store in device memory: layout, insertion and lookup (device code shared by the kernels of trigram.cu).
//
// Three arrays:
//   * home buckets (64 bytes, 2^log2_buckets of them), found by hashing the two-token context (a, b) and probing
//     linearly; a bucket holds its context, six (token, count) entries that fill front to back, and where the
//     context's further entries are;
//   * a pool of (token, count) entries in units of six (48 bytes).  A context's entries beyond six lie in extents of
//     1, 2, 4, ... units, each contiguous, handed out by a bump allocator when the extent before is full; the first
//     extent starts with a directory: where the others are, and how many units the context has been given.  Every
//     entry of a context, however many there are, is therefore two dependent reads behind its home bucket, and a lookup
//     reads them with coalesced 16-byte loads that are all independent.  (Chains of single buckets, as before, cost
//     one dependent read per six entries: a lookup of a frequent context -- thousands of continuations -- was a chain of
//     hundreds to thousands of memory round trips.)
//   * an index over the pool entries: (home bucket, token) -> entry, open addressing, at most three quarters full.
//     Raising a count is one probe of the home buckets, one of the index and one atomic add, wherever the entry is.
//     Measured, 10^6 tokens into an empty table: 0.30 ms (13.6 ms with chains that every insertion walked from the front);
//     lookups: see k_tg_topk and k_topk_mark; a 64-node draft tree from that table 32 us (490).
//
// Entries are never moved or removed.  The configured number of overflow buckets limits the units of six entries in use: as long
// as one is left any context can grow by it, and a unit that was given out can be filled.  The pool has room for the unused ends
// of the extents on top: a context opens extent s only once it has been given 2^s units, so that with d units it takes
// 2 + 1 + 2 + 4 + .. <= 3 d.  (What waiting for that costs: 20,000 tokens into an empty table 32 -> 36 us, 10^6 0.30 -> 0.31 ms, 4 x 10^6 no
// difference, against extents that were opened on a thread's own unit alone, with which a table at its limit could exceed its pool.)
//
// Pool and index take 272-400 bytes per overflow bucket.  Where the device has no room for them the further entries lie in
// chains of buckets instead (TgView::chain, 64 bytes each): an insertion walks its context's chain from the front and a lookup reads it
// bucket by bucket -- the same answers, at the speeds named in brackets above, for tables that would otherwise not exist.
#pragma once

#include <cstddef>

#include "aded_internal.cuh"

namespace aded {

struct TgSlot { int32_t tok; uint32_t cnt; };
struct __align__(64) Bucket {
    unsigned long long key;   // context
    uint32_t more;            // first extent: pool unit + 1 (0 none yet, TG_FAILED: there was no room for it); chained: next bucket + 1
    uint32_t n_more;          // entries beyond six; bit 31 (TG_CLOSED): no room for further ones; chained: places in the chain
    TgSlot e[6];
};
static_assert(sizeof(Bucket) == 64, "bucket must be 64 bytes");
struct __align__(16) TgIndexSlot {
    unsigned long long key;   // home bucket and token (tg_index_key), 0 empty
    unsigned long long at;    // pool entry + 1; 0 while its thread is still placing it, TG_DEAD: there was no room
};

constexpr unsigned long long TG_EMPTY = ~0ull, TG_DEAD = ~0ull;
constexpr int TG_MAX_PROBE = 4096;
constexpr uint32_t TG_FAILED = 0xFFFFFFFFu, TG_CLOSED = 0x80000000u;
constexpr uint32_t TG_LOCKED = TG_FAILED;      // chained: the next bucket is being taken
constexpr int TG_MAX_SPIN = 1 << 20;
constexpr int TG_UNIT = 6;            // entries of a pool unit
constexpr int TG_DIR_UNITS = 2;       // units the directory takes in front of the first extent's entries
constexpr int TG_DIR_WORDS = TG_DIR_UNITS * TG_UNIT * 2;
constexpr int TG_GRANTED = 0;         // directory word: units beyond the first that the limit allowed
constexpr int TG_REFUSED = TG_DIR_WORDS - 1;   // and those it did not
constexpr int TG_LINKS = TG_REFUSED;  // words 1 .. TG_LINKS - 1: extent s (2^s units) is word s

struct TgView {
    Bucket* buckets;
    TgSlot* pool;                // [n_units][TG_UNIT]
    TgIndexSlot* index;
    Bucket* chain;               // [n_over] where the device has no room for pool and index (then unused), else NULL
    uint32_t n_home_mask;
    uint32_t n_home;
    uint32_t n_over;             // configured limit on units of entries in use
    uint32_t n_units;            // units the pool has
    unsigned long long index_mask;
    uint32_t* used;              // [0] units of entries in use (counts on past n_over), [1] pool units handed out
    int32_t* status;
    int32_t vocab;
    uint32_t cap;
    uint32_t min_count;
};

// Pool units for a limit of n_over units in use (see above).
__host__ __device__ constexpr unsigned long long tg_pool_units(unsigned long long n_over) { return 3 * n_over; }
// Index slots: at most three quarters full with every unit filled, and room for the slots of entries that were refused after they had
// taken one -- threads under way when the limit is reached, of which a device holds some 300,000.
constexpr unsigned long long tg_index_slots(unsigned long long n_over) {
    unsigned long long n = 16;
    while (n < 8 * n_over || n < 6 * n_over + (1ull << 19)) n *= 2;
    return n;
}

__device__ __forceinline__ uint32_t tg_hash(unsigned long long k) {
    k ^= k >> 30; k *= 0xBF58476D1CE4E5B9ull;
    k ^= k >> 27; k *= 0x94D049BB133111EBull;
    k ^= k >> 31;
    return (uint32_t)k;
}
__device__ __forceinline__ unsigned long long tg_key(int a, int b) {
    return ((unsigned long long)(uint32_t)a << 32) | (uint32_t)b;
}
// Home buckets number at most 2^28 and tokens are below 2^31: exact, and never 0.
__device__ __forceinline__ unsigned long long tg_index_key(uint32_t home, int tok) {
    return (((unsigned long long)home << 31) | (uint32_t)tok) + 1ull;
}
__device__ __forceinline__ unsigned long long tg_index_start(unsigned long long key) {
    key ^= key >> 29; key *= 0x9E3779B97F4A7C15ull;
    key ^= key >> 32; key *= 0xBF58476D1CE4E5B9ull;
    return key ^ (key >> 31);
}
// Extent of the unit with ordinal m (0-based among a context's units beyond the home bucket): 2^s units from ordinal 2^s - 1.
__device__ __forceinline__ int tg_extent(uint32_t m) { return 31 - __clz((int)(m + 1)); }

// Home bucket of a context; claims an empty one when `insert`.  Returns -1 if absent / no room.
__device__ __forceinline__ int64_t tg_find_home(const TgView& t, unsigned long long key, bool insert) {
    const uint32_t h = tg_hash(key);
    const int limit = t.n_home < (uint32_t)TG_MAX_PROBE ? (int)t.n_home : TG_MAX_PROBE;
    for (int probe = 0; probe < limit; ++probe) {
        const uint32_t idx = (h + probe) & t.n_home_mask;
        unsigned long long k = *reinterpret_cast<volatile unsigned long long*>(&t.buckets[idx].key);
        if (k == key) return idx;
        if (k == TG_EMPTY) {
            if (!insert) return -1;
            k = atomicCAS(&t.buckets[idx].key, TG_EMPTY, key);
            if (k == TG_EMPTY || k == key) return idx;
        }
    }
    return -1;
}

// ---- insertion ------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void tg_report(const TgView& t, int what) { atomicCAS(t.status, 0, what); }

// Raises an entry's count by inc (>= 1), saturating at the cap.  `windows`: the increments of the launch number the
// windows of one span.
__device__ __forceinline__ void tg_raise(const TgView& t, uint32_t* cnt, uint32_t inc, bool windows) {
    if (windows || inc == 1) {
        // cap <= 2^31 - 1 and a span has fewer than 2^31 windows: even if all of them are added before the minimum
        // below takes effect, the 32-bit count cannot wrap
        const uint32_t old = atomicAdd(cnt, inc);
        if (old + inc > t.cap) atomicMin(cnt, t.cap);
        return;
    }
    // imports add arbitrary counts: saturate in one step, so that two large additions to one
    // tri-gram cannot carry the count past 2^32 between an add and a later minimum
    uint32_t seen = *reinterpret_cast<volatile uint32_t*>(cnt);
    for (;;) {
        const uint32_t want = seen >= t.cap || inc > t.cap - seen ? t.cap : seen + inc;
        const uint32_t prev = atomicCAS(cnt, seen, want);
        if (prev == seen) break;
        seen = prev;      // (another thread moved the count; every retry follows a change made by someone else)
    }
}

// Publishing a link or an index entry is a release, reading one an acquire.  (With full fences in their places threads spent as
// long in the fences as in waiting for memory: 35 against 51 of 98 stalled cycles per instruction of the bulk update.)
__device__ __forceinline__ uint32_t tg_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long tg_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void tg_release(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Publishes an extent (or TG_FAILED), unless a thread that ran out of patience has given it up.  Returns what the link says now.
__device__ __forceinline__ uint32_t tg_publish(uint32_t* link, uint32_t base) {
    uint32_t seen;
    asm volatile("atom.release.gpu.global.cas.b32 %0, [%1], 0, %2;" : "=r"(seen) : "l"(link), "r"(base) : "memory");
    return seen == 0 ? base : seen;
}

// Waits (bounded) until another thread has published an extent.  When the wait runs out the extent is given up for everybody
// (TG_FAILED, reported): an entry of it that is not written will never be read, whatever its owner does later.
__device__ __forceinline__ uint32_t tg_wait_link(const TgView& t, uint32_t* link) {
    uint32_t v = tg_acquire(link);
    for (int spin = 0; v == 0 && spin < TG_MAX_SPIN; ++spin) {
        __nanosleep(32);
        v = tg_acquire(link);
    }
    if (v == 0) {
        v = tg_publish(link, TG_FAILED);
        if (v == TG_FAILED) tg_report(t, (int)ADED_ERR_TIMEOUT);
        else v = tg_acquire(link);
    }
    return v;
}

// A new extent: its first unit + 1, or TG_FAILED.  (The pool is sized so that there is room; if not, nothing is written.)
__device__ __forceinline__ uint32_t tg_new_extent(const TgView& t, uint32_t units) {
    const uint32_t at = atomicAdd(&t.used[1], units);
    return (unsigned long long)at + units <= t.n_units ? at + 1 : TG_FAILED;
}

// Whether unit m >= 1 of a context exists: it does once m units beyond the first have been granted, whichever of the threads that
// asked for one got it.  It does not when all that have asked are answered and fewer were granted: a refusal means that the
// limit is reached, so that whoever asks later is refused too.  (Granted, then refused, then asked for are read, none of which
// falls: granted + refused == asked for says that granted was complete when refused was read.)
__device__ __forceinline__ bool tg_wait_room(const TgView& t, const Bucket* bk, const uint32_t* dir, uint32_t m) {
    for (int spin = 0; spin < TG_MAX_SPIN; ++spin) {
        const uint32_t granted = tg_acquire(dir + TG_GRANTED);
        if (granted >= m) return true;
        const uint32_t refused = tg_acquire(dir + TG_REFUSED);
        if (refused != 0 && granted + refused == ((tg_acquire(&bk->n_more) & ~TG_CLOSED) - 1) / TG_UNIT) return false;
        __nanosleep(32);
    }
    tg_report(t, (int)ADED_ERR_TIMEOUT);
    return false;
}

// Takes the next entry of a context beyond its home bucket and writes the token with count 0.  Returns the entry's
// number in the pool plus one, or 0 (reported) when there is no room.  The thread that takes the first entry of a unit asks for
// the unit; all that take one of its entries act on the same answer (tg_wait_room; for the first unit the link in the home bucket).
// The thread that takes the first entry of an extent allocates the extent and publishes it; the others of that
// extent wait for it.  `first`: see tg_full.  Threads only ever wait for owners of earlier entries, so the waits cannot form a
// cycle.  The pool is never cleared: every path leaves the entry written -- with the token, or without one where it was refused or
// a wait ran out -- or in an extent that no reader will find.
__device__ __forceinline__ unsigned long long tg_place(const TgView& t, Bucket* bk, uint32_t first, int c) {
    const uint32_t p = atomicAdd(&bk->n_more, 1u) & ~TG_CLOSED;
    const uint32_t m = p / TG_UNIT, e = p % TG_UNIT;
    const int s = tg_extent(m);
    const uint32_t in_extent = m + 1 - (1u << s);             // the unit's place in its extent
    bool room = true;
    uint32_t base = TG_FAILED;                                // extent's first unit + 1
    if (m == 0) {
        if (e == 0) {
            if (atomicAdd(&t.used[0], 1u) < t.n_over) base = tg_new_extent(t, TG_DIR_UNITS + 1);
            if (base != TG_FAILED) {
                uint4* dir = reinterpret_cast<uint4*>(t.pool + (size_t)(base - 1) * TG_UNIT);
                for (int i = 0; i < TG_DIR_WORDS / 4; ++i) dir[i] = make_uint4(0u, 0u, 0u, 0u);
            }
            base = tg_publish(&bk->more, base);
        } else {
            base = tg_wait_link(t, &bk->more);
        }
    } else {
        if (first == 0) first = tg_wait_link(t, &bk->more);
        if (first != TG_FAILED && s < TG_LINKS) {             // (asked only now: what a context is given it can use)
            uint32_t* dir = reinterpret_cast<uint32_t*>(t.pool + (size_t)(first - 1) * TG_UNIT);
            // (link and count in one round trip; nothing is read through them)
            const uint32_t link = *reinterpret_cast<volatile uint32_t*>(dir + s);
            uint32_t granted = 0;
            if (e != 0) granted = *reinterpret_cast<volatile uint32_t*>(dir + TG_GRANTED);
            else if (atomicAdd(&t.used[0], 1u) < t.n_over) granted = atomicAdd(dir + TG_GRANTED, 1u) + 1u;
            else atomicAdd(dir + TG_REFUSED, 1u);
            room = granted >= m || tg_wait_room(t, bk, dir, m);
            if (e == 0 && in_extent == 0) {
                if (room) base = tg_new_extent(t, 1u << s);
                base = tg_publish(dir + s, base);
            } else {
                base = link != 0 ? link : tg_wait_link(t, dir + s);
            }
        }
    }
    unsigned long long at = 0;
    if (base != TG_FAILED) {
        at = ((unsigned long long)(base - 1) + (s == 0 ? TG_DIR_UNITS : 0) + in_extent) * TG_UNIT + e;
        if (!ADED_IN_RANGE(at < (unsigned long long)t.n_units * TG_UNIT, t.status)) return 0;
        t.pool[at] = TgSlot{room ? c : -1, 0u};               // (an entry without a token is skipped by every reader)
        if (room) return at + 1;
    }
    atomicOr(&bk->n_more, TG_CLOSED);
    tg_report(t, (int)ADED_ERR_TABLE_FULL);
    return 0;
}

// Whether a context can take no further entry: it has been refused one, or its next one would open a unit and the limit is reached.
// (Asked before an index slot is taken: what a full table refuses should leave no trace in the index.)
// `first`: the context's first extent as seen on the way, 0 if it was not there yet.
__device__ __forceinline__ bool tg_full(const TgView& t, const Bucket* bk, uint32_t& first) {
    static_assert(offsetof(Bucket, more) == 8 && offsetof(Bucket, n_more) == 12, "one load for both");
    const unsigned long long both = tg_acquire(reinterpret_cast<const unsigned long long*>(&bk->more));
    first = (uint32_t)both;
    uint32_t n = (uint32_t)(both >> 32);
    for (;;) {
        if (n & TG_CLOSED) return true;
        if (n % TG_UNIT != 0 || tg_acquire(&t.used[0]) < t.n_over) return false;
        // (still the next entry: whoever takes it asks after the limit was reached; if not, somebody else may have been given the last unit for it)
        const uint32_t now = tg_acquire(&bk->n_more);
        if (now == n) return true;
        n = now;
    }
}

// Count cell of the token in a bucket, claiming the first free entry for it; NULL when others have all six.
__device__ __forceinline__ uint32_t* tg_entry(Bucket* bk, int c) {
    // the six tokens at once (they are only ever written from -1 to their final value)
    const int4 e01 = __ldcg(reinterpret_cast<const int4*>(bk) + 1), e23 = __ldcg(reinterpret_cast<const int4*>(bk) + 2), e45 = __ldcg(reinterpret_cast<const int4*>(bk) + 3);
    const int32_t seen[6] = {e01.x, e01.z, e23.x, e23.z, e45.x, e45.z};
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        int32_t have = seen[e];
        if (have == -1) {
            have = atomicCAS(&bk->e[e].tok, -1, c);
            if (have == -1) have = c;
        }
        if (have == c) return &bk->e[e].cnt;
    }
    return nullptr;
}

// The count cell of a token beyond a context's home bucket, in its chain; NULL (reported) when there is none and no room.  The thread
// that finds no next bucket takes one under a one-word lock, the others wait for it.
__device__ __forceinline__ uint32_t* tg_chained_entry(const TgView& t, Bucket* home, int c) {
    Bucket* bk = home;
    for (uint32_t hop = 0; hop < t.n_over; ++hop) {           // (a chain cannot be longer)
        uint32_t next = tg_acquire(&bk->more);
        if (next == 0) {
            next = atomicCAS(&bk->more, 0u, TG_LOCKED);
            if (next == 0) {
                const uint32_t fresh = tg_acquire(&t.used[0]) < t.n_over ? atomicAdd(&t.used[0], 1u) : t.n_over;
                if (fresh < t.n_over) {
                    atomicAdd(&home->n_more, (uint32_t)TG_UNIT);
                    next = fresh + 1;
                }
                atomicExch(&bk->more, next);
            }
        }
        for (int spin = 0; next == TG_LOCKED && spin < TG_MAX_SPIN; ++spin) {
            __nanosleep(64);
            next = tg_acquire(&bk->more);
        }
        if (next == 0 || next == TG_LOCKED) {
            tg_report(t, next == 0 ? (int)ADED_ERR_TABLE_FULL : (int)ADED_ERR_TIMEOUT);
            return nullptr;
        }
        bk = t.chain + (next - 1);
        uint32_t* cnt = tg_entry(bk, c);
        if (cnt) return cnt;
    }
    tg_report(t, (int)ADED_ERR_TABLE_FULL);
    return nullptr;
}

// Raises the count of tri-gram (a, b, c) by `inc` (see tg_raise), inserting it if absent; counts
// saturate at the cap.  Independent atomic adds: the result does not depend on the thread order.
__device__ __forceinline__ void tg_add(const TgView& t, int a, int b, int c, uint32_t inc, bool windows) {
    const int64_t home = tg_find_home(t, tg_key(a, b), true);
    if (home < 0) { tg_report(t, (int)ADED_ERR_TABLE_FULL); return; }
    if (!ADED_IN_RANGE((uint64_t)home < (uint64_t)t.n_home, t.status)) return;
    Bucket* bk = t.buckets + home;
    uint32_t* cnt = tg_entry(bk, c);
    if (!cnt && t.chain) {
        cnt = tg_chained_entry(t, bk, c);
        if (!cnt) return;
    }
    if (cnt) { tg_raise(t, cnt, inc, windows); return; }
    const unsigned long long key = tg_index_key((uint32_t)home, c);
    unsigned long long at_index = tg_index_start(key) & t.index_mask;
    const int limit = t.index_mask < TG_MAX_PROBE ? (int)t.index_mask + 1 : TG_MAX_PROBE;
    for (int probe = 0; probe < limit; ++probe, at_index = (at_index + 1) & t.index_mask) {
        TgIndexSlot* slot = t.index + at_index;
        unsigned long long k = *reinterpret_cast<volatile unsigned long long*>(&slot->key);
        if (k == 0) {
            uint32_t first;
            if (tg_full(t, bk, first)) {
                k = tg_acquire(&slot->key);                   // (unless the last entry has gone to this very token)
                if (k == 0) { tg_report(t, (int)ADED_ERR_TABLE_FULL); return; }
            } else {
                k = atomicCAS(&slot->key, 0ull, key);
            }
            if (k == 0) {
                const unsigned long long at = tg_place(t, bk, first, c);
                tg_release(&slot->at, at ? at : TG_DEAD);
                if (at) tg_raise(t, &t.pool[at - 1].cnt, inc, windows);
                return;
            }
        }
        if (k == key) {
            unsigned long long at = tg_acquire(&slot->at);
            for (int spin = 0; at == 0 && spin < TG_MAX_SPIN; ++spin) {
                __nanosleep(32);
                at = tg_acquire(&slot->at);
            }
            if (at == 0) { tg_report(t, (int)ADED_ERR_TIMEOUT); return; }
            if (at == TG_DEAD) { tg_report(t, (int)ADED_ERR_TABLE_FULL); return; }
            tg_raise(t, &t.pool[at - 1].cnt, inc, windows);
            return;
        }
    }
    tg_report(t, (int)ADED_ERR_TABLE_FULL);
}

// ---- lookup ---------------------------------------------------------------------------------------------------------
// A context's entries as one warp holds them.
struct TgWalk {
    uint4 part;            // lanes 0..3: the home bucket's 16-byte parts (header, then two entries each); elsewhere no entries
    uint32_t n;            // entries beyond the home bucket
    uint32_t extent;       // lane s: where extent s has its entries (first unit + 1, 0 none)
    uint32_t chain;        // first bucket of the chain + 1, 0 none
    bool found;            // the context is stored
};

// Lane s gets extent s of the context whose home bucket `w.part` holds.
__device__ __forceinline__ void tg_open_extents(const TgView& t, TgWalk& w, int lane) {
    const uint32_t more = __shfl_sync(0xffffffffu, w.part.z, 0), n = __shfl_sync(0xffffffffu, w.part.w, 0);
    if (lane == 0 || lane > 3) { w.part.x = 0xFFFFFFFFu; w.part.y = 0u; w.part.z = 0xFFFFFFFFu; w.part.w = 0u; }
    w.n = 0;
    w.extent = 0;
    w.chain = 0;
    if (more == 0 || more == TG_FAILED) return;
    if (t.chain) { w.chain = more; return; }
    w.n = n & ~TG_CLOSED;
    if (lane == 0) {
        w.extent = more + TG_DIR_UNITS;
    } else if (lane < TG_LINKS && w.n > (uint32_t)TG_UNIT * ((1u << lane) - 1u)) {
        const uint32_t link = reinterpret_cast<const uint32_t*>(t.pool + (size_t)(more - 1) * TG_UNIT)[lane];
        w.extent = link == TG_FAILED ? 0u : link;
    }
}

// By home bucket (all lanes the same, stored).
__device__ __forceinline__ TgWalk tg_open(const TgView& t, uint32_t home, int lane) {
    TgWalk w;
    w.found = ADED_IN_RANGE(home < t.n_home, t.status);
    w.part = make_uint4(0u, 0u, 0u, 0u);
    if (w.found && lane < 4) w.part = reinterpret_cast<const uint4*>(t.buckets + home)[lane];
    tg_open_extents(t, w, lane);
    return w;
}

// By context (all lanes the same): a bucket's key and entries come with one read.
__device__ __forceinline__ TgWalk tg_open(const TgView& t, int a, int b, int lane) {
    TgWalk w;
    w.part = make_uint4(0u, 0u, 0u, 0u);
    w.found = false;
    if (a >= 0 && b >= 0 && a < t.vocab && b < t.vocab) {
        const unsigned long long key = tg_key(a, b);
        const uint32_t h = tg_hash(key);
        const int limit = t.n_home < (uint32_t)TG_MAX_PROBE ? (int)t.n_home : TG_MAX_PROBE;
        for (int probe = 0; probe < limit; ++probe) {
            const uint32_t idx = (h + probe) & t.n_home_mask;
            if (lane < 4) w.part = reinterpret_cast<const uint4*>(t.buckets + idx)[lane];
            const unsigned long long k = ((unsigned long long)__shfl_sync(0xffffffffu, w.part.y, 0) << 32) | __shfl_sync(0xffffffffu, w.part.x, 0);
            w.found = k == key;
            if (k == key || k == TG_EMPTY) break;
        }
    }
    if (!w.found) w.part = make_uint4(0u, 0u, 0u, 0u);
    tg_open_extents(t, w, lane);
    return w;
}

// The best entries of a context, largest packed (count, ~token) first: lane r holds the r-th, lanes from k on nothing of use.
// Packed keys are distinct (a context holds a token once); 0 = none.
__device__ __forceinline__ unsigned long long tg_pack(const TgView& t, int32_t tok, uint32_t cnt) {
    return tok >= 0 && cnt > 0 && cnt >= t.min_count ? ((unsigned long long)cnt << 32) | (0xFFFFFFFFu - (uint32_t)tok) : 0ull;
}
__device__ __forceinline__ int32_t tg_packed_tok(unsigned long long key) { return key ? (int32_t)(0xFFFFFFFFu - (uint32_t)key) : -1; }
__device__ __forceinline__ uint32_t tg_packed_cnt(unsigned long long key) { return (uint32_t)(key >> 32); }

// Every lane offers one key; those that beat the k-th best so far are inserted one by one, which is rare after the first
// few (entries lie in order of first appearance, so the frequent tokens come early).
__device__ __forceinline__ void tg_offer(unsigned long long cand, int k, int lane, unsigned long long& best) {
    unsigned m = __ballot_sync(0xffffffffu, cand > __shfl_sync(0xffffffffu, best, k - 1));
    while (m) {
        const unsigned long long c = __shfl_sync(0xffffffffu, cand, __ffs((int)m) - 1);
        const int rank = __popc(__ballot_sync(0xffffffffu, lane < k && best > c));
        const unsigned long long up = __shfl_up_sync(0xffffffffu, best, 1);
        if (lane == rank) best = c;
        else if (lane > rank) best = up;
        m &= m - 1;
        m &= __ballot_sync(0xffffffffu, cand > __shfl_sync(0xffffffffu, best, k - 1));
    }
}

// Every lane offers two keys.  Where few beat the k-th best so far they are inserted one by one (about 100 cycles each);
// where k or more do -- the first entries of a context, the merge of several warps' lists -- the new list is picked in k
// rounds of warp-wide maxima instead.
__device__ __forceinline__ void tg_offer2(unsigned long long c0, unsigned long long c1, int k, int lane, unsigned long long& best) {
    const unsigned long long top = c0 > c1 ? c0 : c1;
    const unsigned m = __ballot_sync(0xffffffffu, top > __shfl_sync(0xffffffffu, best, k - 1));
    if (m == 0) return;
    if (__popc(m) < k) {
        tg_offer(c0, k, lane, best);
        tg_offer(c1, k, lane, best);
        return;
    }
    unsigned long long have = lane < k ? best : 0ull, out = 0;
    for (int r = 0; r < k; ++r) {
        unsigned long long v = c0 > c1 ? c0 : c1;
        v = v > have ? v : have;
        const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32));
        if (hi == 0) break;                     // (counts are at least 1)
        const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
        const unsigned long long pick = ((unsigned long long)hi << 32) | lo;
        if (lane == r) out = pick;
        if (have == pick) have = 0;
        if (c0 == pick) c0 = 0;
        if (c1 == pick) c1 = 0;
    }
    best = out;
}

// Two entries per lane (token -1: none) into the running list and sum.
__device__ __forceinline__ void tg_take(const TgView& t, uint4 v, int k, int lane, unsigned long long& best, uint32_t& total) {
    if ((int32_t)v.x >= 0) total += v.y;
    if ((int32_t)v.z >= 0) total += v.w;
    tg_offer2(tg_pack(t, (int32_t)v.x, v.y), tg_pack(t, (int32_t)v.z, v.w), k, lane, best);
}

// The buckets of a chain, one after the other: `f` gets their 16-byte parts as tg_take takes them.
template <typename F>
__device__ __forceinline__ void tg_each_chained(const TgView& t, uint32_t at, int lane, F f) {
    for (uint32_t hop = 0; at != 0 && at != TG_LOCKED && hop < t.n_over; ++hop) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (lane < 4 && ADED_IN_RANGE(at <= t.n_over, t.status)) v = reinterpret_cast<const uint4*>(t.chain + (at - 1))[lane];
        at = __shfl_sync(0xffffffffu, v.z, 0);
        if (lane == 0 || lane > 3) v = make_uint4(0xFFFFFFFFu, 0u, 0xFFFFFFFFu, 0u);
        f(v);
    }
}

// Part `part` of `parts` of a context's entries (each part by one warp, all lanes): the k <= 32 best of them in `best`, and this
// lane's share of the sum of the counts in `total` (both are carried on from the caller's values).
__device__ __forceinline__ void tg_scan(const TgView& t, const TgWalk& w, int part, int parts, int k, int lane, unsigned long long& best, uint32_t& total) {
    if (part == 0) {
        tg_take(t, w.part, k, lane, best, total);
        if (w.chain) tg_each_chained(t, w.chain, lane, [&](uint4 v) { tg_take(t, v, k, lane, best, total); });
    }
    // The entries beyond, two per lane and load, BATCH loads in flight.  Pair g is the (g % 3)-th of the unit with ordinal g / 3.
    constexpr int BATCH = 4;
    const uint32_t pairs = (w.n + 1) / 2;
    for (uint32_t g0 = (uint32_t)part * 32; g0 < pairs; g0 += (uint32_t)parts * 32 * BATCH) {
        uint4 v[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            const uint32_t g = g0 + (uint32_t)i * parts * 32 + lane;
            const uint32_t m = g / 3;
            const int s = tg_extent(m);
            const uint32_t base = __shfl_sync(0xffffffffu, w.extent, s & 31);
            v[i] = make_uint4(0xFFFFFFFFu, 0u, 0xFFFFFFFFu, 0u);
            if (g < pairs && base != 0) {
                const size_t unit = (size_t)(base - 1) + (m + 1 - (1u << s));
                if (ADED_IN_RANGE(unit < t.n_units, t.status)) v[i] = reinterpret_cast<const uint4*>(t.pool + unit * TG_UNIT)[g % 3];
                if (2 * g + 1 >= w.n) { v[i].z = 0xFFFFFFFFu; v[i].w = 0u; }
            }
        }
#pragma unroll
        for (int i = 0; i < BATCH; ++i) tg_take(t, v[i], k, lane, best, total);
    }
}

// Count cell of a stored tri-gram, or NULL.
__device__ __forceinline__ const uint32_t* tg_find(const TgView& t, int a, int b, int c) {
    const int64_t home = tg_find_home(t, tg_key(a, b), false);
    if (home < 0) return nullptr;
    const Bucket* bk = t.buckets + home;
    for (int e = 0; e < 6; ++e)
        if (bk->e[e].tok == c) return &bk->e[e].cnt;
    if (t.chain) {
        uint32_t at = bk->more;
        for (uint32_t hop = 0; at != 0 && at != TG_LOCKED && hop < t.n_over; ++hop) {
            bk = t.chain + (at - 1);
            for (int e = 0; e < 6; ++e)
                if (bk->e[e].tok == c) return &bk->e[e].cnt;
            at = bk->more;
        }
        return nullptr;
    }
    const unsigned long long key = tg_index_key((uint32_t)home, c);
    unsigned long long i = tg_index_start(key) & t.index_mask;
    const int limit = t.index_mask < TG_MAX_PROBE ? (int)t.index_mask + 1 : TG_MAX_PROBE;
    for (int probe = 0; probe < limit; ++probe, i = (i + 1) & t.index_mask) {
        if (t.index[i].key == 0) return nullptr;
        if (t.index[i].key == key) {
            const unsigned long long at = t.index[i].at;
            return at == 0 || at == TG_DEAD ? nullptr : &t.pool[at - 1].cnt;
        }
    }
    return nullptr;
}

}  // namespace aded
