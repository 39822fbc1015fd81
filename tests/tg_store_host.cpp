// The insertion code of the tri-gram store (csrc/tg_store.cuh, turned into a host header by test_tg_store_host.py) under random
// interleavings of its atomic steps: every simulated thread is a coroutine that gives way at each atomic operation and load, and
// the next one to run is drawn.  The pool has guard words behind it and is filled with entries that nobody inserted.
//   tg_store_host <seed> <runs> <late> <chained>    late = 1: threads are held back for long stretches, so that bounded waits run out;
//                                                   chained = 1: the layout without pool and index
#include <ucontext.h>

#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <random>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
#define __align__(n) alignas(n)
struct int4 { int x, y, z, w; };
struct uint4 { unsigned x, y, z, w; };
static uint4 make_uint4(unsigned x, unsigned y, unsigned z, unsigned w) { return {x, y, z, w}; }
static int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
enum { ADED_ERR_TABLE_FULL = 4, ADED_ERR_TIMEOUT = 8, ADED_ERR_INTERNAL = 9 };
#define ADED_IN_RANGE(cond, status) ((cond) ? true : (*(status) = (int)ADED_ERR_INTERNAL, false))

static void give_way();
template <typename T> static T model_load(const T* p) { give_way(); return *p; }
template <typename T> static void model_store(T* p, T v) { give_way(); *p = v; }
template <typename T, typename U> static T atomicAdd(T* p, U v) { give_way(); const T old = *p; *p += (T)v; return old; }
template <typename T, typename U> static T atomicExch(T* p, U v) { give_way(); const T old = *p; *p = (T)v; return old; }
template <typename T, typename U> static T atomicOr(T* p, U v) { give_way(); const T old = *p; *p |= (T)v; return old; }
template <typename T, typename U> static T atomicMin(T* p, U v) { give_way(); const T old = *p; if ((T)v < old) *p = (T)v; return old; }
template <typename T, typename U, typename V> static T atomicCAS(T* p, U cmp, V v) { give_way(); const T old = *p; if (old == (T)cmp) *p = (T)v; return old; }
template <typename T> static T __ldcg(const T* p) { return model_load(p); }
static void __nanosleep(unsigned) { give_way(); }

#include "tg_store_host.h"
using namespace aded;

// ---- coroutines -------------------------------------------------------------------------------------------------------
struct Thread { ucontext_t ctx; std::vector<char> stack; bool done; long wake; };
static ucontext_t g_main;
static std::vector<Thread> g_threads;
static Thread* g_cur = nullptr;
static std::mt19937_64 g_rng;
static bool g_late, g_stalls;              // held back beyond the spin limit; for a while
static long g_step;
struct Job { int a, b, c; };
static std::vector<Job> g_jobs;
static TgView g_view;

static void give_way() {
    if (!g_cur) return;
    if (g_late && g_rng() % 64 == 0) g_cur->wake = g_step + (long)(g_rng() % 60000);
    if (g_stalls && g_rng() % 4 == 0) g_cur->wake = g_step + (long)(g_rng() % 3000);
    swapcontext(&g_cur->ctx, &g_main);
}
static void entry(int i) {
    tg_add(g_view, g_jobs[i].a, g_jobs[i].b, g_jobs[i].c, 1u, true);
    g_threads[i].done = true;
    swapcontext(&g_threads[i].ctx, &g_main);
}
static void run_all() {
    const int n = (int)g_jobs.size();
    g_threads.assign(n, Thread());
    std::vector<int> live;
    for (int i = 0; i < n; ++i) {
        Thread& t = g_threads[i];
        t.stack.resize(32768);
        t.done = false;
        t.wake = 0;
        getcontext(&t.ctx);
        t.ctx.uc_stack.ss_sp = t.stack.data();
        t.ctx.uc_stack.ss_size = t.stack.size();
        t.ctx.uc_link = &g_main;
        makecontext(&t.ctx, (void (*)())entry, 1, i);
        live.push_back(i);
    }
    // one thread in a few runs ahead of the others for a while
    while (!live.empty()) {
        const size_t at = g_rng() % live.size();
        Thread& t = g_threads[live[at]];
        for (int burst = 1 + (int)(g_rng() % 4) * (g_rng() % 4 == 0 ? 40 : 1); burst > 0 && !t.done; --burst) {
            ++g_step;
            if (t.wake > g_step) break;
            g_cur = &t;
            swapcontext(&g_main, &t.ctx);
            g_cur = nullptr;
        }
        if (t.done) { live[at] = live.back(); live.pop_back(); }
    }
}

#define CHECK(cond, ...) do { if (!(cond)) { printf("run %d (n_over %u): " #cond " failed: ", run, n_over); printf(__VA_ARGS__); printf("\n"); return 1; } } while (0)

int main(int argc, char** argv) {
    g_rng.seed(strtoull(argv[1], nullptr, 10));
    const int runs = atoi(argv[2]);
    g_late = argc > 3 && atoi(argv[3]) != 0;
    const bool chained = argc > 4 && atoi(argv[4]) != 0;
    long timeouts = 0, refusals = 0;
    for (int run = 0; run < runs; ++run) {
        static const unsigned limits[] = {0, 1, 2, 3, 4, 5, 8, 9, 10, 17, 40, 64};
        const unsigned n_over = limits[g_rng() % 12];
        g_stalls = g_rng() % 2;
        const int contexts = 1 + (int)(g_rng() % 4), threads = 20 + (int)(g_rng() % 240), tokens = 1 + (int)(g_rng() % threads) + threads / 2;
        const size_t n_units = (size_t)tg_pool_units(n_over), guard = 64, n_index = (size_t)tg_index_slots(n_over);
        std::vector<Bucket> home(16);
        auto clear = [](Bucket& b) {
            b.key = TG_EMPTY; b.more = 0; b.n_more = 0;
            for (TgSlot& e : b.e) e = TgSlot{-1, 0u};
        };
        for (Bucket& b : home) clear(b);
        std::vector<Bucket> chain(n_over + guard);
        for (size_t i = 0; i < chain.size(); ++i) { clear(chain[i]); if (i >= n_over) chain[i].more = 77u; }
        std::vector<uint4> pool((n_units + guard) * TG_UNIT / 2 + 2);
        TgSlot* cells = reinterpret_cast<TgSlot*>(pool.data());
        for (size_t i = 0; i < (n_units + guard) * TG_UNIT; ++i) cells[i] = TgSlot{1000000 + (int)i, 777u};
        TgIndexSlot* index = static_cast<TgIndexSlot*>(calloc(n_index, sizeof(TgIndexSlot)));
        uint32_t used[2] = {0, 0};
        int32_t status = 0;
        g_view = TgView();
        g_view.buckets = home.data(); g_view.pool = cells; g_view.index = index;
        if (chained) { g_view.chain = chain.data(); g_view.pool = nullptr; g_view.index = nullptr; }
        g_view.n_home = 16; g_view.n_home_mask = 15; g_view.n_over = n_over; g_view.n_units = (uint32_t)n_units; g_view.index_mask = n_index - 1;
        g_view.used = used; g_view.status = &status; g_view.vocab = 1 << 20; g_view.cap = 0x7fffffffu; g_view.min_count = 0;
        std::map<std::pair<int, int>, uint32_t> added;      // (context, token) -> how often
        for (int round = 0; round < 3; ++round) {
            g_jobs.clear();
            for (int i = 0; i < threads; ++i) {
                const Job j = {(int)(g_rng() % contexts), 7, (int)(g_rng() % tokens)};
                g_jobs.push_back(j);
                ++added[{j.a, j.c}];
            }
            status = 0;
            run_all();
            for (size_t i = n_units * TG_UNIT; i < (n_units + guard) * TG_UNIT; ++i)
                CHECK(cells[i].tok == 1000000 + (int)i && cells[i].cnt == 777u, "the pool of %zu units was written %zu entries past its end", n_units, i - n_units * TG_UNIT);
            for (size_t i = n_over; i < chain.size(); ++i) CHECK(chain[i].more == 77u && chain[i].e[0].tok == -1 && chain[i].n_more == 0, "chain bucket %zu of %u", i, n_over);
            CHECK(status != ADED_ERR_INTERNAL, "an index out of range");
            timeouts += status == ADED_ERR_TIMEOUT;
            refusals += status == ADED_ERR_TABLE_FULL;
            // what a reader sees (as tg_open_extents and tg_scan walk it)
            unsigned long long units = 0;
            bool refused = false;
            for (const Bucket& b : home) {
                if (b.key == TG_EMPTY) continue;
                const int a = (int)(b.key >> 32);
                std::map<int, uint32_t> seen;
                for (const TgSlot& e : b.e)
                    if (e.tok >= 0) { CHECK(seen.count(e.tok) == 0, "token %d twice", e.tok); seen[e.tok] = e.cnt; }
                const size_t at_home = seen.size();
                for (uint32_t at = chained ? b.more : 0u; at != 0 && at != TG_LOCKED; at = chain[at - 1].more) {
                    CHECK(at <= n_over, "chain bucket %u", at - 1);
                    for (const TgSlot& e : chain[at - 1].e)
                        if (e.tok >= 0) { CHECK(seen.count(e.tok) == 0, "token %d twice", e.tok); seen[e.tok] = e.cnt; }
                }
                const uint32_t n = chained || b.more == 0 || b.more == TG_FAILED ? 0u : b.n_more & ~TG_CLOSED;
                for (uint32_t p = 0; p < n; ++p) {
                    const uint32_t m = p / TG_UNIT;
                    const int s = tg_extent(m);
                    uint32_t base = b.more + TG_DIR_UNITS;
                    if (s > 0) base = s < TG_LINKS ? reinterpret_cast<const uint32_t*>(cells + (size_t)(b.more - 1) * TG_UNIT)[s] : 0u;
                    if (base == 0 || base == TG_FAILED) continue;
                    const size_t unit = (size_t)(base - 1) + (m + 1 - (1u << s));
                    CHECK(unit < n_units, "unit %zu of %zu", unit, n_units);
                    const TgSlot e = cells[unit * TG_UNIT + p % TG_UNIT];
                    if (e.tok < 0) continue;
                    CHECK(seen.count(e.tok) == 0, "token %d twice", e.tok);
                    seen[e.tok] = e.cnt;
                }
                for (const auto& it : seen) {
                    CHECK(added.count({a, it.first}), "token %d of context %d was never inserted", it.first, a);
                    const uint32_t want = added[{a, it.first}];
                    CHECK(g_late ? it.second <= want : it.second == want, "token %d of context %d counted %u times instead of %u", it.first, a, it.second, want);
                }
                size_t distinct = 0;
                for (const auto& it : added) distinct += it.first.first == a;
                const size_t beyond = seen.size() - at_home;
                units += (beyond + TG_UNIT - 1) / TG_UNIT;
                if (!g_late) {
                    CHECK(seen.size() == distinct || ((b.n_more & TG_CLOSED) && beyond % TG_UNIT == 0) || (beyond % TG_UNIT == 0 && used[0] >= n_over),
                          "context %d holds %zu of %zu tokens", a, seen.size(), distinct);
                    refused = refused || seen.size() < distinct;
                }
            }
            CHECK(units <= n_over, "%llu units in use", units);
            if (!g_late) {
                CHECK(!refused || units == n_over, "refused with %llu units in use", units);
                CHECK((status == ADED_ERR_TABLE_FULL) == refused || !refused, "status %d", status);
                CHECK(status == 0 || status == ADED_ERR_TABLE_FULL, "status %d", status);
            }
        }
        free(index);
    }
    printf("ok: %d runs, %ld full, %ld timed out\n", runs, refusals, timeouts);
    return 0;
}
