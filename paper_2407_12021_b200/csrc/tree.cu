// Draft-tree bookkeeping around the forward pass ("Draft Construction and Verification"):
// validation + depths + ancestor masks before it, draft approval and cache compaction after it.
#include <type_traits>

#include "aded_internal.cuh"

namespace aded {

// The start of a pass: a block per row.  Every block checks its sequence's tree, a thread per node: node 0 is the only root and every
// other node points at an earlier node, tokens are in the vocabulary, the cache has room.  Then its row's ancestor bit set and depth
// (a climb to the root, bounded as parents decrease strictly), embedding, first RMSNorm and rotary tables (made by the last warps
// while the row is on its way).  One kernel: as two, a check per sequence and then the rows, a pass took 3.5 us more.
//
// The call's record and row offsets come as kernel arguments (two small copies ahead of the pass cost it about 10 us) and are
// published here for the kernels that follow.
struct PrologueArgs {
    CallPtrs call;
    int32_t row_off[PROLOGUE_MAX_BATCH + 1];
    int batch;
    int given;             // 0: call and row_off have been copied to their places instead
};
__device__ __forceinline__ float4 begin_load4(const float* p, int vec) { return vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]); }
__device__ __forceinline__ float4 begin_load4(const bf16* p, int) { return unpack4_bf16(*reinterpret_cast<const uint2*>(p)); }
__device__ __forceinline__ void begin_store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void begin_store4(bf16* p, float4 v) { *reinterpret_cast<uint2*>(p) = pack4_bf16(v.x, v.y, v.z, v.w); }

// Four columns per thread and pass, two passes: d <= 8 x the block's threads.  vec: table and gain of an fp32 model lie on 16-byte boundaries.
template <typename T>
__global__ void __launch_bounds__(1024) k_pass_begin(const __grid_constant__ PrologueArgs pa, CallPtrs* call_dev, int32_t* row_off_dev, int32_t* order,
                                                     const int32_t* __restrict__ len, const int32_t* __restrict__ cap, int vocab, int chain_mode, RowMeta rows,
                                                     const T* __restrict__ table, const T* __restrict__ gain, T* __restrict__ h, T* __restrict__ x, int d,
                                                     float eps, RopeArgs rope, int vec, int32_t* status) {
    pdl_launch_dependents();
    __shared__ float red[32];
    __shared__ int s_bad, s_pending, s_par[ADED_MAX_NODES];
    const int r = blockIdx.x, tid = threadIdx.x, threads = blockDim.x;
    float4 gv[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int c = (e * threads + tid) * 4;
        if (c < d) gv[e] = begin_load4(gain + c, vec);
    }
    pdl_wait();
    if (tid == 0) {                                // (read once: another block may be reporting)
        s_bad = 0;
        s_pending = *status;
    }
    if (first_thread_of_grid()) trace_mark(status, TK_OTHER);
    const int32_t* __restrict__ offsets = pa.given ? pa.row_off : row_off_dev;
    const int32_t* __restrict__ tokens = pa.given ? pa.call.tokens : call_dev->tokens;
    const int32_t* __restrict__ parents = pa.given ? pa.call.parents : call_dev->parents;
    int b = 0;                                     // the row's sequence: the last that begins at or before it
    for (int hi = pa.batch; hi - b > 1; ) {
        const int mid = (b + hi) >> 1;
        if (offsets[mid] <= r) b = mid;
        else hi = mid;
    }
    const int off = offsets[b], T_nodes = offsets[b + 1] - off, i = r - off, L = len[b];
    int tok = tokens[r];
    if (pa.given && r == 0) {
        if (tid == 0) *call_dev = pa.call;
        if (tid <= pa.batch) row_off_dev[tid] = pa.row_off[tid];
    }
    if (tok < 0 || tok >= vocab) tok = 0;          // (reported below)
    const T* src = table + (size_t)tok * d;
    float4 v[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int c = (e * threads + tid) * 4;
        if (c < d) v[e] = begin_load4(src + c, vec);
    }
    __syncthreads();
    if (pa.batch > 1 && i == 0) {                  // this sequence's place by falling length
        int place = 0;
        for (int o0 = 0; o0 < pa.batch; o0 += threads) {
            const int o = o0 + tid, other = o < pa.batch ? len[o] : -1;
            place += __syncthreads_count(o < pa.batch && (other > L || (other == L && o < b)));
        }
        if (tid == 0) order[place] = b;
    }
    if (s_pending != 0) return;                    // an earlier error is still pending: do nothing
    if (tid < T_nodes) {
        const int p = chain_mode ? tid - 1 : parents[off + tid], t = tokens[off + tid];
        s_par[tid] = p;
        if (t < 0 || t >= vocab) atomicMax(&s_bad, (int)ADED_ERR_INVALID_ARG);
        if (tid == 0 ? (p != -1) : (p < 0 || p >= tid)) atomicMax(&s_bad, (int)ADED_ERR_BAD_TREE);
        if (tid == 0 && L + T_nodes > cap[b]) atomicMax(&s_bad, (int)ADED_ERR_KV_CAPACITY);
    }
    __syncthreads();
    if (s_bad != 0) {
        if (tid == 0) atomicCAS(status, 0, s_bad);
        return;
    }
    float sq = 0.f;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int c = (e * threads + tid) * 4;
        if (c < d) {
            begin_store4(h + (size_t)r * d + c, v[e]);
            sq += v[e].x * v[e].x + v[e].y * v[e].y + v[e].z * v[e].z + v[e].w * v[e].w;
        }
    }
    const int last = threads - 1 - tid;
    if (last < max(rope.half, 1)) {                // each of these threads climbs
        uint64_t lo, hi;
        int depth;
        if (chain_mode) {
            depth = i;
            lo = i < 63 ? (2ull << i) - 1ull : ~0ull;
            hi = i < 64 ? 0ull : i < 127 ? (2ull << (i - 64)) - 1ull : ~0ull;
        } else {
            lo = hi = 0;
            depth = -1;
            for (int cur = i; cur >= 0; cur = s_par[cur]) {
                if (cur < 64) lo |= 1ull << cur;
                else hi |= 1ull << (cur - 64);
                ++depth;
            }
        }
        if (last == 0) {
            rows.seq[r] = b;
            rows.local[r] = i;
            rows.pos[r] = L + depth;
            rows.anc[2 * r] = lo;
            rows.anc[2 * r + 1] = hi;
        }
        for (int e = last; e < rope.half; e += threads) {
            double s, c;
            sincos((double)(L + depth) * rope.freq[e], &s, &c);
            rope.cs[r * rope.half + e] = (float)c;
            rope.sn[r * rope.half + e] = (float)s;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((tid & 31) == 0) red[tid >> 5] = sq;
    __syncthreads();
    float total = 0.f;
    for (int e = 0; e < threads / 32; ++e) total += red[e];
    const float inv = rsqrtf(total / (float)d + eps);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int c = (e * threads + tid) * 4;
        if (c < d)
            begin_store4(x + (size_t)r * d + c, make_float4(v[e].x * inv * gv[e].x, v[e].y * inv * gv[e].y, v[e].z * inv * gv[e].z, v[e].w * inv * gv[e].w));
    }
}

// Draft approval for tokens that are already chosen (sampling mode); a block per sequence.
__global__ void k_accept(const CallPtrs* __restrict__ call,
                         const int32_t* __restrict__ row_off, const int32_t* __restrict__ best,
                         const uint64_t* __restrict__ anc, int32_t* __restrict__ len,
                         int32_t* __restrict__ path, int32_t* __restrict__ moves,
                         const int32_t* status, int batch) {
    pdl_enter();
    if (first_thread_of_grid()) trace_mark(status, TK_PICK);
    const int32_t* __restrict__ tokens = call->tokens;
    const int32_t* __restrict__ parents = call->parents;
    int32_t* __restrict__ out_tokens = call->out_tokens;
    int32_t* __restrict__ out_len = call->out_len;
    const int out_stride = call->out_stride;
    const int b = blockIdx.x;
    if (b >= batch) return;
    __shared__ int32_t s_par[ADED_MAX_NODES], s_tok[ADED_MAX_NODES], s_best[ADED_MAX_NODES];
    const int pass_status = *status;
    const int off = row_off[b];
    const int T = min(row_off[b + 1] - off, (int)ADED_MAX_NODES);
    for (int i = threadIdx.x; i < T; i += blockDim.x) {
        s_par[i] = parents[off + i];
        s_tok[i] = tokens[off + i];
        s_best[i] = best[off + i];
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    approval_warp(threadIdx.x, s_par, s_tok, s_best, anc + 2 * (size_t)off, T, pass_status, out_tokens + (size_t)b * out_stride, out_len + b,
                  path + b * ADED_MAX_NODES, moves + 2 * b, len + b);
}

// Compaction: the tree's K/V were written at slots L + node index; the accepted path p_0 = 0 <
// p_1 < ... moves to slots L + 0, L + 1, ...  Because p_j >= j and the p_j increase, the source of a
// later move is never the destination of an earlier one, and a thread that owns one 16-byte column of a plane and walks j
// upwards, COMPACT_BATCH moves at a time, reads every slot before it overwrites it.  Latency-bound: all reads of a batch are in
// flight together, and a block takes several planes.
constexpr int COMPACT_THREADS = 128, COMPACT_BATCH = 8;
__global__ void __launch_bounds__(COMPACT_THREADS)
k_compact(char* const* __restrict__ base, const int32_t* __restrict__ cap, const int32_t* __restrict__ moves,
          const int32_t* __restrict__ path, int planes, int chunks, const int32_t* status) {
    pdl_enter();
    if (first_thread_of_grid()) trace_mark(status, TK_STEP_END);
    if (*status != 0) return;
    const int b = blockIdx.y;
    const int L = moves[2 * b], n_acc = moves[2 * b + 1];
    if (n_acc <= 1) return;
    const int plane = blockIdx.x * (COMPACT_THREADS / chunks) + (int)threadIdx.x / chunks;      // (layer * 2 + k|v) * H + head
    if (plane >= planes) return;
    uint4* p = reinterpret_cast<uint4*>(base[b]) + ((size_t)plane * cap[b] + L) * chunks + threadIdx.x % chunks;
    for (int j0 = 1; j0 < n_acc; j0 += COMPACT_BATCH) {
        int src[COMPACT_BATCH];
        uint4 v[COMPACT_BATCH];
#pragma unroll
        for (int i = 0; i < COMPACT_BATCH; ++i) {
            const int j = j0 + i;
            src[i] = j < n_acc ? path[b * ADED_MAX_NODES + j] : j;
            if (!ADED_IN_RANGE(j >= n_acc || (src[i] >= j && src[i] < ADED_MAX_NODES && L + src[i] < cap[b]), status)) src[i] = j;
        }
#pragma unroll
        for (int i = 0; i < COMPACT_BATCH; ++i)
            if (src[i] != j0 + i) v[i] = p[(size_t)src[i] * chunks];
#pragma unroll
        for (int i = 0; i < COMPACT_BATCH; ++i)
            if (src[i] != j0 + i) p[(size_t)(j0 + i) * chunks] = v[i];
    }
}

// Prefill: every row is kept.
__global__ void k_commit_chain(int32_t* len, const int32_t* __restrict__ row_off, const int32_t* status, int batch) {
    pdl_enter();
    if (first_thread_of_grid()) trace_mark(status, TK_STEP_END);
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= batch || *status != 0) return;
    len[b] += row_off[b + 1] - row_off[b];
}

// Rows [pos0, pos0 + n) of all heads of a layer's K and V planes, to or from the caller's two [head][n] arrays; chunks of 16 bytes.
// Grid (parts of a head's rows, heads, K and V).
constexpr int KV_COPY_THREADS = 256, KV_COPY_PER = 4;
template <bool LOAD>
__global__ void __launch_bounds__(KV_COPY_THREADS)
k_kv_copy(uint4* cache_k, uint4* cache_v, size_t head_stride, uint4* user_k, uint4* user_v, size_t n) {
    uint4* cache = (blockIdx.z ? cache_v : cache_k) + blockIdx.y * head_stride;
    uint4* user = (blockIdx.z ? user_v : user_k) + blockIdx.y * n;
    const size_t i0 = (size_t)blockIdx.x * (KV_COPY_THREADS * KV_COPY_PER) + threadIdx.x;
    uint4 v[KV_COPY_PER];
#pragma unroll
    for (int j = 0; j < KV_COPY_PER; ++j)
        if (i0 + j * KV_COPY_THREADS < n) v[j] = (LOAD ? user : cache)[i0 + j * KV_COPY_THREADS];
#pragma unroll
    for (int j = 0; j < KV_COPY_PER; ++j)
        if (i0 + j * KV_COPY_THREADS < n) (LOAD ? cache : user)[i0 + j * KV_COPY_THREADS] = v[j];
}

void launch_kv_copy(char* cache_k, char* cache_v, size_t head_bytes, void* user_k, void* user_v, size_t bytes, int heads, bool load, cudaStream_t st) {
    const size_t n = bytes / sizeof(uint4), per = KV_COPY_THREADS * KV_COPY_PER;
    const dim3 grid((unsigned)((n + per - 1) / per), heads, 2);
    auto* ck = reinterpret_cast<uint4*>(cache_k);
    auto* cv = reinterpret_cast<uint4*>(cache_v);
    auto* uk = static_cast<uint4*>(user_k);
    auto* uv = static_cast<uint4*>(user_v);
    if (load) k_kv_copy<true><<<grid, KV_COPY_THREADS, 0, st>>>(ck, cv, head_bytes / sizeof(uint4), uk, uv, n);
    else k_kv_copy<false><<<grid, KV_COPY_THREADS, 0, st>>>(ck, cv, head_bytes / sizeof(uint4), uk, uv, n);
}

void launch_pass_begin(aded_model* m, aded_kv* kv, const CallPtrs& call, const int32_t* offsets_host, int batch, int rows, int chain_mode, cudaStream_t st) {
    PrologueArgs pa = {};
    pa.given = batch <= PROLOGUE_MAX_BATCH;
    pa.batch = batch;
    if (pa.given) {
        pa.call = call;
        for (int b = 0; b <= batch; ++b) pa.row_off[b] = offsets_host[b];
    }
    const aded_model_config& c = m->cfg;
    const void* gain = m->layers[0].norm1;
    static_assert(PROLOGUE_MAX_BATCH < 256 && ADED_MAX_NODES <= 256, "a thread per row offset and per node");
    auto go = [&](auto* kernel, auto* type, int threads, int vec) {
        using T = std::remove_pointer_t<decltype(type)>;
        launch_k(kernel, dim3(rows), dim3(threads), 0, st, pa, m->call_dev, m->seqs.row_off, m->seqs.order, kv->len_dev, kv->cap_dev, c.vocab, chain_mode, m->rows,
                 (const T*)m->top.embed, (const T*)gain, (T*)m->h, (T*)m->x, c.d_model, c.rms_eps, rope_args(m), vec, m->status);
    };
    if (c.dtype == ADED_BF16) go(k_pass_begin<bf16>, (bf16*)nullptr, 1024, 1);
    else go(k_pass_begin<float>, (float*)nullptr, c.d_model <= 1024 ? 256 : 1024, (reinterpret_cast<uintptr_t>(m->top.embed) | reinterpret_cast<uintptr_t>(gain)) % 16 == 0);
}

void launch_accept(aded_model* m, aded_kv* kv, int batch, cudaStream_t st) {
    launch_k(k_accept, batch, 128, 0, st, m->call_dev, m->seqs.row_off, m->best, m->rows.anc,
                                               kv->len_dev, m->seqs.path, m->seqs.moves, m->status, batch);
}

void launch_compact(aded_model* m, aded_kv* kv, int batch, cudaStream_t st) {
    // a row of a plane is head_dim (64 or 128) elements of 2 or 4 bytes: 8, 16 or 32 chunks of 16
    const int chunks = (int)(m->cfg.head_dim * m->elem / sizeof(uint4)), planes = m->cfg.n_layers * 2 * m->cfg.n_heads, per = COMPACT_THREADS / chunks;
    launch_k(k_compact, dim3((planes + per - 1) / per, batch), COMPACT_THREADS, 0, st, kv->base_dev, kv->cap_dev, m->seqs.moves, m->seqs.path, planes,
             chunks, m->status);
}

void launch_commit_chain(aded_model* m, aded_kv* kv, int batch, cudaStream_t st) {
    launch_k(k_commit_chain, (batch + 31) / 32, 32, 0, st, kv->len_dev, m->seqs.row_off, m->status, batch);
}

}  // namespace aded
