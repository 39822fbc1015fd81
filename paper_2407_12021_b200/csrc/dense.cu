// Row-wise pieces of the Llama-style decoder around the projections: embedding gather, residual
// add + RMSNorm, rotary embedding + K/V write, SwiGLU, per-row greedy choice, and a plain
// shared-memory GEMM used for fp32 models and for shapes the tensor-core path does not take.
//
// Rounding: activations are stored in the model dtype (bf16 models round to nearest even at
// every store below); all sums are fp32.  Kernels that consume a projection read it through
// GemmOut (gemm_out.cuh): either a plain fp32 matrix or per-CTA partial tiles added in CTA order.
// These are the kernels of fp32 models; bf16 models on the tensor-core path use the four-columns-per-thread
// versions in dense_ws.cu.
#include "aded_internal.cuh"

namespace aded {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Frequencies of the rotary embedding, theta^(-2i/hd), in double (once per model; the angles are made per pass, k_pass_begin).
__global__ void k_rope_freq(double* __restrict__ freq, int half, double theta) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < half) freq[i] = pow(theta, -(double)i / (double)half);
}

// h = round(h + y) (y may be absent);  x = round(h * rsqrt(mean(h^2) + eps) * gain).  One block
// per row, columns strided over the threads and kept in registers between the sum of squares and the scaling; the sum's
// order is fixed.  fp32 models; of bf16 models those whose widths the tensor-core GEMM does not take.
constexpr int NORM_COLS = 8;           // columns per thread: d_model <= 8 x 1024
template <typename T>
__global__ void __launch_bounds__(1024) k_add_rmsnorm(T* __restrict__ h, const float* __restrict__ y, const T* __restrict__ gain, T* __restrict__ x, int d,
                                                      float eps, const int32_t* status) {
    pdl_launch_dependents();
    __shared__ float red[32];
    const int r = blockIdx.x;
    float g[NORM_COLS], v[NORM_COLS];
#pragma unroll
    for (int i = 0; i < NORM_COLS; ++i) {
        const int c = threadIdx.x + i * blockDim.x;
        g[i] = c < d ? to_f32(gain[c]) : 0.f;
    }
    pdl_wait();
    if (first_thread_of_grid()) trace_mark(status, TK_NORM);
    if (*status != 0) return;
    float sq = 0.f;
#pragma unroll
    for (int i = 0; i < NORM_COLS; ++i) {
        const int c = threadIdx.x + i * blockDim.x;
        v[i] = 0.f;
        if (c < d) {
            v[i] = to_f32(h[(size_t)r * d + c]);
            if (y) v[i] = to_f32(from_f32<T>(v[i] + y[(size_t)r * d + c]));
            h[(size_t)r * d + c] = from_f32<T>(v[i]);
        }
        sq += v[i] * v[i];
    }
    sq = warp_sum(sq);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
    __syncthreads();
    float total = 0.f;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) total += red[i];
    const float inv = rsqrtf(total / (float)d + eps);
#pragma unroll
    for (int i = 0; i < NORM_COLS; ++i) {
        const int c = threadIdx.x + i * blockDim.x;
        if (c < d) x[(size_t)r * d + c] = from_f32<T>(v[i] * inv * g[i]);
    }
}

// y[r, n] = sum_k x[r, k] * w[n, k] in fp32.  A block computes BM rows x BN columns: the operands of a chunk of k are staged in
// shared memory as they lie (rows padded by four words: the lanes of a warp then read different banks), 4 x 4 outputs per
// thread, four k per step; the threads beyond one per 4 x 4 split the chunk's k among them, and their sums are added at the end
// in a fixed order.
// These are the GEMMs of small models and a handful of rows: bound by latency, not by arithmetic.  So the chunk is all of k where
// that fits -- one round of loads, of which the weights' are issued before the previous kernel has finished -- and the split of
// k keeps eight warps busy on 16 rows.  (Blocks of 64 x 64 outputs with 16 k at a time took 23 to 65 us per GEMM of the 256-wide
// fp32 model at 16 rows, two barriers and one exposed load per 16 k; this: 3.9 to 6.5 us.)
constexpr int GP_THREADS = 256;
template <typename T, bool VEC>
__device__ __forceinline__ float4 gp_load4(const T* p) {
    if (!VEC) return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
    if (sizeof(T) == 4) return *reinterpret_cast<const float4*>(p);
    return unpack4_bf16(*reinterpret_cast<const uint2*>(p));
}

template <typename T, int BM, int BN, bool VEC>
__global__ void __launch_bounds__(GP_THREADS) k_gemm_plain(const T* __restrict__ x, const T* __restrict__ w,
                                                           float* __restrict__ y, int rows, int n, int k, int chunk,
                                                           const int32_t* status, int trace_kind) {
    pdl_launch_dependents();
    constexpr int RG = BM / 4, CG = BN / 4, SLICES = GP_THREADS / (CG * RG), STEP = 4 * SLICES;
    extern __shared__ __align__(16) float gp_smem[];
    const int ld = (chunk + 31) / 32 * 32 + 4;
    float* sw = gp_smem;                       // [BN][ld]
    float* sx = gp_smem + BN * ld;             // [BM][ld]
    const int n0 = blockIdx.x * BN, r0 = blockIdx.y * BM;
    const int cg = threadIdx.x % CG, rg = threadIdx.x / CG % RG, slice = threadIdx.x / (CG * RG);
    // rows [from, from + count) of m, columns [k0, k0 + len), zero beyond `limit` rows and beyond k (k % 4 == 0)
    auto stage = [&](float* dst, const T* m, int from, int count, int limit, int k0, int len) {
        const int quads = len / 4;
        for (int i = threadIdx.x; i < count * quads; i += GP_THREADS) {
            const int rr = i / quads, kk = (i % quads) * 4;
            const bool there = from + rr < limit && k0 + kk < k;
            const T* src = m + (there ? (size_t)(from + rr) * k + k0 + kk : 0);
            float* to = dst + (size_t)rr * ld + kk;
            if (VEC && sizeof(T) == 4) {       // all of a thread's copies in flight, without registers; zeros where there is nothing
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(src), "r"(there ? 16 : 0) : "memory");
            } else {
                *reinterpret_cast<float4*>(to) = there ? gp_load4<T, VEC>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    };
    float acc[4][4] = {};
    for (int k0 = 0; k0 < k; k0 += chunk) {
        const int here = k - k0 < chunk ? k - k0 : chunk, len = (here + STEP - 1) / STEP * STEP;      // (chunk % STEP == 0 unless it is all of k)
        if (k0 > 0) __syncthreads();
        stage(sw, w, n0, BN, n, k0, len);
        if (k0 == 0) {
            pdl_wait();
            if (first_thread_of_grid()) trace_mark(status, trace_kind);
            if (*status != 0) {
                asm volatile("cp.async.wait_all;" ::: "memory");
                return;
            }
        }
        stage(sx, x, r0, BM, rows, k0, len);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        const int per = len / SLICES;
        for (int kk = slice * per; kk < (slice + 1) * per; kk += 4) {
            float4 a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = *reinterpret_cast<const float4*>(sx + (size_t)(rg + RG * i) * ld + kk);
                b[i] = *reinterpret_cast<const float4*>(sw + (size_t)(cg + CG * i) * ld + kk);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
                    acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
                    acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
                    acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
                }
        }
    }
    __syncthreads();
    float* part = gp_smem;                     // [SLICES][BM][BN]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) part[(slice * BM + rg + RG * i) * BN + cg + CG * j] = acc[i][j];
    __syncthreads();
    for (int o = threadIdx.x; o < BM * BN; o += GP_THREADS) {
        float sum = part[o];
#pragma unroll
        for (int sl = 1; sl < SLICES; ++sl) sum += part[sl * BM * BN + o];
        const int r = r0 + o / BN, c = n0 + o % BN;
        if (r < rows && c < n) y[(size_t)r * n + c] = sum;
    }
}

// Rotary embedding of q and k (pairs (i, i + hd/2), angle from the table), then q -> q buffer and
// k, v -> the cache at slot committed length + local node index.  Block = (row, head).
// bf16 models release the next kernel only after this one's wait: see attn_sequence (fp32 attention reads nothing early).
template <typename T>
__global__ void k_rope_kv(GemmOut qkv, const float* __restrict__ cs, const float* __restrict__ sn,
                          T* __restrict__ q, char* const* __restrict__ base, const int32_t* __restrict__ cap,
                          const int32_t* __restrict__ len, const int32_t* __restrict__ row_seq,
                          const int32_t* __restrict__ row_local, int layer, int H, int hd, const int32_t* status) {
    if (sizeof(T) == 4) pdl_launch_dependents();
    pdl_wait();
    if (sizeof(T) != 4) pdl_launch_dependents();
    if (first_thread_of_grid()) trace_mark(status, TK_ROPE);
    if (*status != 0) return;
    const int r = blockIdx.x, hh = blockIdx.y, half = hd >> 1, d = H * hd;
    const int b = row_seq[r];
    const size_t slot = (size_t)len[b] + row_local[r];
    const size_t cp = cap[b];
    T* kdst = reinterpret_cast<T*>(base[b]) + ((((size_t)layer * 2 + 0) * H + hh) * cp + slot) * hd;
    T* vdst = reinterpret_cast<T*>(base[b]) + ((((size_t)layer * 2 + 1) * H + hh) * cp + slot) * hd;
    // the head's q, k and v columns each lie inside one 128-column tile of the projection result
    const int cq = hh * hd, ck = d + hh * hd, cv = 2 * d + hh * hd;
    TileRef tq = {0, 0}, tk = {0, 0}, tv = {0, 0};
    if (qkv.mode == 1) { tq = qkv.tiles[cq >> 7]; tk = qkv.tiles[ck >> 7]; tv = qkv.tiles[cv >> 7]; }
    auto at = [&](const TileRef& t, int col) {
        return qkv.mode == 0 ? qkv.y[(size_t)r * 3 * d + col] : gemm_out_at(qkv, t, r, col & 127);
    };
    for (int i = threadIdx.x; i < half; i += blockDim.x) {
        const float c = cs[r * half + i], s = sn[r * half + i];
        const float q0 = at(tq, cq + i), q1 = at(tq, cq + i + half);
        const float k0 = at(tk, ck + i), k1 = at(tk, ck + i + half);
        q[(size_t)r * d + hh * hd + i] = from_f32<T>(q0 * c - q1 * s);
        q[(size_t)r * d + hh * hd + i + half] = from_f32<T>(q1 * c + q0 * s);
        kdst[i] = from_f32<T>(k0 * c - k1 * s);
        kdst[i + half] = from_f32<T>(k1 * c + k0 * s);
        vdst[i] = from_f32<T>(at(tv, cv + i));
        vdst[i + half] = from_f32<T>(at(tv, cv + i + half));
    }
}

// act = round(silu(gate) * up), gate = gu[:, :F], up = gu[:, F:].
template <typename T>
__global__ void k_swiglu(GemmOut gu, T* __restrict__ act, int F, const int32_t* status) {
    pdl_enter();
    if (first_thread_of_grid()) trace_mark(status, TK_SWIGLU);
    if (*status != 0) return;
    const int r = blockIdx.y;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= F) return;
    const float g = gemm_out_load(gu, r, c), u = gemm_out_load(gu, r, F + c);
    act[(size_t)r * F + c] = from_f32<T>(g / (1.f + expf(-g)) * u);
}

// Greedy choice per row: largest fp32 logit, lowest index among equals.  Stage 1: grid (chunks, rows),
// every block scans `chunk` columns of one row and leaves (value, index) of its best, which the approval kernel
// (k_pick_accept) takes up like the LM head's per-tile candidates.
__global__ void __launch_bounds__(256) k_argmax_chunks(GemmOut logits, float* __restrict__ pv, int32_t* __restrict__ pi,
                                                       int V, int chunk, const int32_t* status) {
    pdl_enter();
    if (first_thread_of_grid()) trace_mark(status, TK_PICK);
    if (*status != 0) return;
    __shared__ float sv[8];
    __shared__ int si[8];
    const int r = logits.row0 + blockIdx.y;
    const int c0 = blockIdx.x * chunk, c1 = min(V, c0 + chunk);
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    if (logits.mode == 1 && (V & 3) == 0) {
        // partial tiles: four adjacent columns per thread and step, all contributors fetched at once
        for (int c = c0 + threadIdx.x * 4; c < c1; c += 1024) {
            const float4 v = gemm_out_at4(logits, logits.tiles[c >> 7], r, c & 127);
            if (v.x > bv) { bv = v.x; bi = c; }       // columns ascend per thread: first maximum kept
            if (v.y > bv) { bv = v.y; bi = c + 1; }
            if (v.z > bv) { bv = v.z; bi = c + 2; }
            if (v.w > bv) { bv = v.w; bi = c + 3; }
        }
    } else {
        for (int c = c0 + threadIdx.x; c < c1; c += 256) {
            const float v = gemm_out_load(logits, r, c);
            if (v > bv) { bv = v; bi = c; }   // c ascends per thread: first maximum kept
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) { sv[w] = bv; si[w] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i)
            if (sv[i] > bv || (sv[i] == bv && si[i] < bi)) { bv = sv[i]; bi = si[i]; }
        pv[r * gridDim.x + blockIdx.x] = bv;
        pi[r * gridDim.x + blockIdx.x] = bi;
    }
}

// A projection result as a plain matrix.  Four columns per thread where it lies in partial tiles (n is then a multiple of 128)
// and the destination's rows start on 16-byte boundaries.
__global__ void k_materialize(GemmOut src, float* __restrict__ dst, int n, int vec, const int32_t* status) {
    pdl_enter();
    if (first_thread_of_grid()) trace_mark(status, TK_OTHER);
    if (*status != 0) return;
    const int r = src.row0 + blockIdx.y;
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) * (vec ? 4 : 1);
    if (c >= n) return;
    if (vec) *reinterpret_cast<float4*>(dst + (size_t)r * n + c) = gemm_out_at4(src, src.tiles[c >> 7], r, c & 127);
    else dst[(size_t)r * n + c] = gemm_out_load(src, r, c);
}

// ---- launchers --------------------------------------------------------------------------
#define BY_DTYPE(m, CALL_BF16, CALL_F32) \
    do { if ((m)->cfg.dtype == ADED_BF16) { CALL_BF16; } else { CALL_F32; } } while (0)

void launch_rope_freq(double* freq, int half, double theta) { k_rope_freq<<<1, half>>>(freq, half, theta); }

static int norm_threads(int d) { return d >= 1024 ? 1024 : (d + 31) / 32 * 32; }

void launch_add_rmsnorm(aded_model* m, const GemmOut& y, const void* gain, cudaStream_t st) {
    const int d = m->cfg.d_model;
    if (y.mode == 1) { launch_add_rmsnorm_ws(m, y, gain, st); return; }
    BY_DTYPE(m, (launch_k(k_add_rmsnorm<bf16>, y.rows, norm_threads(d), 0, st, (bf16*)m->h, y.y, (const bf16*)gain, (bf16*)m->x, d, m->cfg.rms_eps, m->status)),
             (launch_k(k_add_rmsnorm<float>, y.rows, norm_threads(d), 0, st, (float*)m->h, y.y, (const float*)gain, (float*)m->x, d, m->cfg.rms_eps, m->status)));
}

constexpr int GP_SMEM = 160 * 1024, GP_CHUNK = 256;

template <typename T, int BM, int BN>
static void launch_gemm_plain_bm(aded_model* m, const T* x, const T* w, float* y, int rows, int n, int k, int trace_kind, cudaStream_t st) {
    // all of k at once where it fits (and only few blocks run), else pieces that leave room for more than one block per SM
    auto bytes = [](int c) { return (size_t)(BN + BM) * ((c + 31) / 32 * 32 + 4) * sizeof(float); };
    const int piece = BN == 32 ? GP_CHUNK : sizeof(T) == 4 ? GP_CHUNK / 2 : GP_CHUNK / 4;
    const int chunk = k <= piece || (BM == 16 && bytes(k) <= GP_SMEM) ? k : piece;
    const size_t sums = (size_t)GP_THREADS * 16 * sizeof(float);       // the partial sums take the operands' place
    const size_t smem = bytes(chunk) > sums ? bytes(chunk) : sums;
    const bool vec = k % 4 == 0 && (reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w)) % (4 * sizeof(T)) == 0;
    launch_k(vec ? k_gemm_plain<T, BM, BN, true> : k_gemm_plain<T, BM, BN, false>, dim3((n + BN - 1) / BN, (rows + BM - 1) / BM), GP_THREADS, smem, st,
             x, w, y, rows, n, k, chunk, m->status, trace_kind);
}

template <typename T>
static void launch_gemm_plain(aded_model* m, const T* x, const T* w, float* y, int rows, int n, int k, int trace_kind, cudaStream_t st) {
    // The fewest rows per block that still leave no more than about two waves of blocks: more rows per block read the weights fewer
    // times from L2, fewer spread a small GEMM over more SMs.  What is larger than that takes blocks of 64 x 64, which stage each
    // operand for twice as many outputs as 64 x 32, a thread per 4 x 4 of them over all of k, and pieces of k that let several blocks
    // share an SM.  Measured, the five projections of a layer and LM head of width 4096, us: bf16, 256 rows 7560 (9830 with 64 x 32
    // and 256 k at a time; 512 rows 13500 and 19200), fp32 6450 (7300; 12400 and 14000).
    const long long cols = (n + 31) / 32, limit = 2ll * ws_grid_limit(m->device);
    if (cols * ((rows + 15) / 16) <= limit) launch_gemm_plain_bm<T, 16, 32>(m, x, w, y, rows, n, k, trace_kind, st);
    else if (cols * ((rows + 31) / 32) <= limit) launch_gemm_plain_bm<T, 32, 32>(m, x, w, y, rows, n, k, trace_kind, st);
    else launch_gemm_plain_bm<T, 64, 64>(m, x, w, y, rows, n, k, trace_kind, st);
}

template <typename T>
static bool gemm_plain_prepare_t() {
    bool ok = true;
    auto set = [&](auto* f) { ok = ok && cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, GP_SMEM) == cudaSuccess; };
    set(k_gemm_plain<T, 16, 32, true>); set(k_gemm_plain<T, 16, 32, false>);
    set(k_gemm_plain<T, 32, 32, true>); set(k_gemm_plain<T, 32, 32, false>);
    set(k_gemm_plain<T, 64, 64, true>); set(k_gemm_plain<T, 64, 64, false>);
    return ok;
}
// (For the models that use it: the first call on a kernel loads it, which takes the creation of a model milliseconds.)
bool gemm_plain_prepare(bool bf16_model) { return bf16_model ? gemm_plain_prepare_t<bf16>() : gemm_plain_prepare_t<float>(); }

// The tensor-core GEMM runs once per 128 rows (256 in calls with more: half as many trips over W).
int gemm_pass_rows(const aded_model* m, int rows) { return !m->ws_ready ? rows : rows > 128 ? 256 : 128; }

bool gemm_is_many(const aded_model* m, int rows, int n, int k) { return m->many_ok && many_block_rows(m->device, rows, n, k) > 0; }

void launch_gemm_many(aded_model* m, int w_map, int x_map, int rows, int n, int k, const ManyEpilogue& epi, int trace_kind, cudaStream_t st) {
    const int block = many_block_rows(m->device, rows, n, k);
    const int table = w_map < 4 * m->cfg.n_layers ? w_map % 4 : 4;
    many_launch(m->ws_use_tiled ? m->ws_tiled_maps[w_map] : m->ws_half_maps[w_map], m->ws_use_tiled, m->ws_x_maps[x_map], rows, block, n, k,
                ws_grid(m->device, n, k, m->ws_one_per_sm[table]), m->ws_slots, m->many_flags, m->status, epi, trace_kind, m->device, st);
}

void launch_rmsnorm(aded_model* m, int rows, const void* gain, cudaStream_t st) {
    GemmOut none = {};
    none.rows = rows;
    if (m->ws_ready) launch_add_rmsnorm_ws(m, none, gain, st);
    else launch_add_rmsnorm(m, none, gain, st);
}

GemmOut launch_gemm(aded_model* m, int w_map, int x_map, const void* x, const void* w, float* y, int row0, int rows, int n, int k,
                    int epi_mode, int trace_kind, cudaStream_t st) {
    GemmOut out = {};
    out.n = n;
    out.row0 = row0;
    out.rows = rows;
    if (m->ws_ready && w_map >= 0 && x_map >= 0 && ws_supported(n, k)) {
        // tensor-core path; the result stays in slots
        const int table = w_map < 4 * m->cfg.n_layers ? w_map % 4 : 4;
        WsEpilogue e = {};
        e.mode = epi_mode;
        e.tiles = m->ws_tiles[table];
        e.counters = m->ws_counters;
        e.cand_val = m->cand_val;
        e.cand_idx = m->cand_idx;
        if (epi_mode != WS_EPI_SLOTS) e.epoch = ++m->ws_epoch;
        ws_launch(m->ws_maps[w_map], m->ws_use_tiled ? m->ws_tiled[w_map] : nullptr, m->ws_x_maps[x_map][(rows - 1) / 16], rows, row0, n, k, m->ws_slots,
                  m->status, e, trace_kind, m->device, m->ws_one_per_sm[table], st);
        out.mode = 1;
        out.slots = m->ws_slots;
        out.n_tiles = n / 128;
        out.kb = k / 64;
        out.g = ws_grid(m->device, n, k, m->ws_one_per_sm[table]);
        out.tiles = m->ws_tiles[table];
        return out;
    }
    BY_DTYPE(m, (launch_gemm_plain<bf16>(m, (const bf16*)x, (const bf16*)w, y, rows, n, k, trace_kind, st)),
             (launch_gemm_plain<float>(m, (const float*)x, (const float*)w, y, rows, n, k, trace_kind, st)));
    out.mode = 0;
    out.y = y;
    return out;
}

void launch_materialize(aded_model* m, const GemmOut& src, float* dst, cudaStream_t st) {
    const int vec = src.mode == 1 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0, cols = vec ? 1024 : 256;
    dim3 grid((src.n + cols - 1) / cols, src.rows);
    launch_k(k_materialize, grid, 256, 0, st, src, dst, src.n, vec, m->status);
}

void launch_rope_kv(aded_model* m, aded_kv* kv, const GemmOut& qkv, int layer, cudaStream_t st) {
    if (qkv.mode == 1 && m->cfg.dtype == ADED_BF16) { launch_rope_kv_ws(m, kv, qkv, layer, st); return; }
    dim3 grid(qkv.rows, m->cfg.n_heads);
    const int H = m->cfg.n_heads, hd = m->cfg.head_dim;
    BY_DTYPE(m, (launch_k(k_rope_kv<bf16>, grid, 64, 0, st, qkv, m->rope_cos, m->rope_sin, (bf16*)m->q, kv->base_dev, kv->cap_dev, kv->len_dev, m->rows.seq, m->rows.local, layer, H, hd, m->status)),
             (launch_k(k_rope_kv<float>, grid, 64, 0, st, qkv, m->rope_cos, m->rope_sin, (float*)m->q, kv->base_dev, kv->cap_dev, kv->len_dev, m->rows.seq, m->rows.local, layer, H, hd, m->status)));
}

void launch_swiglu(aded_model* m, const GemmOut& gu, cudaStream_t st) {
    if (gu.mode == 1 && m->cfg.dtype == ADED_BF16) { launch_swiglu_ws(m, gu, st); return; }
    const int F = m->cfg.d_ffn;
    dim3 grid((F + 255) / 256, gu.rows);
    BY_DTYPE(m, (launch_k(k_swiglu<bf16>, grid, 256, 0, st, gu, (bf16*)m->act, F, m->status)),
             (launch_k(k_swiglu<float>, grid, 256, 0, st, gu, (float*)m->act, F, m->status)));
}

void launch_argmax(aded_model* m, const GemmOut& logits, cudaStream_t st) {
    const int V = m->cfg.vocab;
    const int chunks = ARGMAX_CHUNKS;
    const int chunk = ((V + chunks - 1) / chunks + 127) / 128 * 128;   // whole 128-column tiles per block
    dim3 grid(chunks, logits.rows);
    launch_k(k_argmax_chunks, grid, 256, 0, st, logits, m->argmax_val, m->argmax_idx, V, chunk, m->status);
}

}  // namespace aded
