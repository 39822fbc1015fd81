// fp32 models of small widths and calls of few rows: a layer in five launches instead of nine.
//
// Such a pass is bound by the latency of its launches: each is a chain of a few L2 round trips, 3 to 5 us, whatever it computes.  So
// the row-wise kernels between the projections are part of them here:
//   * QKV, gate/up and LM head read the residual stream itself: a block stages its rows whole, multiplies them with the norm's gain and
//     sums their squares while they lie in shared memory, and scales its results with 1 / rms at the end;
//   * O and down add to the residual stream, gate/up computes gate and up columns side by side and leaves their SwiGLU product, the
//     LM head leaves the best logit of every 32 columns;
//   * the attention kernel rotates its row's query and its ancestors' keys as it reads them from the QKV result, and writes its row's key
//     and value to the cache (for the calls to come; this one's tree is never read from it).
// Sums are fp32 as in dense.cu; those of a norm are taken in another order and its factors applied in another place.
// Measured, 2 layers of width 256, 16 nodes, 64 positions: 24 launches, 102 us, before; 15 and 78 with
// this, 14 and 72 since a pass begins with one kernel (tree.cu).
#include "aded_internal.cuh"

namespace aded {

constexpr int F32_THREADS = 256, F32_SMEM = 200 * 1024;
enum { F32_QKV = 0, F32_ADD = 1, F32_SWIGLU = 2, F32_HEAD = 3 };       // what is done with a projection's result; all but ADD normalise

struct F32Args {
    const float* x;          // [rows, k]
    const float* w;          // [n, k]
    const float* gain;       // [k] of the norm
    float* y;                // QKV, HEAD: [rows, n]; ADD: the residual stream, [rows, n]; SWIGLU: [rows, n / 2]
    float* x_out;            // HEAD: the normalised rows
    float* cand_val;         // HEAD: [rows][blocks of 32 columns]
    int32_t* cand_idx;
    int rows, n, k;
    float eps;
    const int32_t* status;
    int trace_kind;
};

// k padded to what the slices of a block divide evenly, and the distance of staged rows (the lanes of a warp read different banks).
template <int BM, int BN> __host__ __device__ constexpr int f32_step() { return 4 * F32_THREADS / (BM / 4 * (BN / 4)); }
template <int BM, int BN> __host__ __device__ constexpr int f32_len(int k) { return (k + f32_step<BM, BN>() - 1) / f32_step<BM, BN>() * f32_step<BM, BN>(); }
template <int BM, int BN> static size_t f32_smem(int k) {
    const size_t operands = (size_t)(BM + BN + 1) * (f32_len<BM, BN>(k) + 4) * sizeof(float), sums = (size_t)F32_THREADS * 16 * sizeof(float);
    return operands > sums ? operands : sums;
}

// BM rows x BN columns per block, 4 x 4 outputs per thread, the threads beyond one per 4 x 4 split k (as k_gemm_plain, with all of k staged).
template <int BM, int BN, int MODE>
__global__ void __launch_bounds__(F32_THREADS) k_gemm_f32(const __grid_constant__ F32Args a) {
    pdl_launch_dependents();
    constexpr int RG = BM / 4, CG = BN / 4, SLICES = F32_THREADS / (CG * RG), HALF = BN / 2;
    extern __shared__ __align__(16) float f32_smem_raw[];
    __shared__ float s_inv[BM];
    const int len = f32_len<BM, BN>(a.k), ld = len + 4, quads = len / 4;
    float* sw = f32_smem_raw;                  // [BN][ld]
    float* sx = sw + BN * ld;                  // [BM][ld]
    float* sg = sx + BM * ld;                  // [k] the norm's gain
    const int n0 = blockIdx.x * BN, r0 = blockIdx.y * BM;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cg = tid % CG, rg = tid / CG % RG, slice = tid / (CG * RG);
    auto stage = [&](float* dst, const float* m, int count, int limit, auto&& row_of) {
        for (int i = tid; i < count * quads; i += F32_THREADS) {
            const int rr = i / quads, kk = (i % quads) * 4, from = row_of(rr);
            const bool there = from < limit && kk < a.k;
            const float* src = m + (there ? (size_t)from * a.k + kk : 0);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + rr * ld + kk)), "l"(src), "r"(there ? 16 : 0) : "memory");
        }
    };
    // column c of the block is row column(c) of W (SwiGLU: half of the block gate columns, half the up columns that belong to them)
    auto column = [&](int c) {
        if (MODE != F32_SWIGLU) return n0 + c;
        const int j = (int)blockIdx.x * HALF + c % HALF, F = a.n / 2;
        return j >= F ? a.n : c < HALF ? j : F + j;
    };
    stage(sw, a.w, BN, a.n, column);
    if (MODE != F32_ADD)
        for (int e = tid * 4; e < a.k; e += F32_THREADS * 4)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(sg + e)), "l"(a.gain + e) : "memory");
    pdl_wait();
    if (first_thread_of_grid()) trace_mark(a.status, a.trace_kind);
    if (*a.status != 0) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }
    stage(sx, a.x, BM, a.rows, [&](int r) { return r0 + r; });
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (MODE != F32_ADD) {
        for (int r = warp; r < BM; r += F32_THREADS / 32) {
            float sq = 0.f;
            for (int e = lane * 4; e < a.k; e += 128) {
                float4 v = *reinterpret_cast<float4*>(sx + r * ld + e);
                const float4 g = *reinterpret_cast<const float4*>(sg + e);
                sq += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
                v.x *= g.x; v.y *= g.y; v.z *= g.z; v.w *= g.w;
                *reinterpret_cast<float4*>(sx + r * ld + e) = v;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            const float inv = rsqrtf(sq / (float)a.k + a.eps);
            if (lane == 0) s_inv[r] = inv;
            if (MODE == F32_HEAD && blockIdx.x == 0 && r0 + r < a.rows)
                for (int e = lane * 4; e < a.k; e += 128) {
                    const float4 v = *reinterpret_cast<const float4*>(sx + r * ld + e);
                    *reinterpret_cast<float4*>(a.x_out + (size_t)(r0 + r) * a.k + e) = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
                }
        }
        __syncthreads();
    }
    float acc[4][4] = {};
    const int per = len / SLICES;
    for (int kk = slice * per; kk < (slice + 1) * per; kk += 4) {
        float4 p[4], q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            p[i] = *reinterpret_cast<const float4*>(sx + (rg + RG * i) * ld + kk);
            q[i] = *reinterpret_cast<const float4*>(sw + (cg + CG * i) * ld + kk);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[i][j] = fmaf(p[i].x, q[j].x, acc[i][j]);
                acc[i][j] = fmaf(p[i].y, q[j].y, acc[i][j]);
                acc[i][j] = fmaf(p[i].z, q[j].z, acc[i][j]);
                acc[i][j] = fmaf(p[i].w, q[j].w, acc[i][j]);
            }
    }
    __syncthreads();
    float* part = f32_smem_raw;                // [SLICES][BM][BN]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) part[(slice * BM + rg + RG * i) * BN + cg + CG * j] = acc[i][j];
    __syncthreads();
    auto total = [&](int o) {
        float sum = part[o];
#pragma unroll
        for (int sl = 1; sl < SLICES; ++sl) sum += part[sl * BM * BN + o];
        return MODE == F32_ADD ? sum : sum * s_inv[o / BN];
    };
    if (MODE == F32_SWIGLU) {
        for (int o = tid; o < BM * HALF; o += F32_THREADS) {
            const int rr = o / HALF, cc = o % HALF, r = r0 + rr, c = blockIdx.x * HALF + cc;
            const float g = total(rr * BN + cc), u = total(rr * BN + HALF + cc);
            if (r < a.rows && c < a.n / 2) a.y[(size_t)r * (a.n / 2) + c] = g / (1.f + expf(-g)) * u;
        }
        return;
    }
#pragma unroll
    for (int o = tid; o < BM * BN; o += F32_THREADS) {
        const int r = r0 + o / BN, c = n0 + o % BN;
        const float sum = total(o);
        const bool there = r < a.rows && c < a.n;
        if (there) {
            float* to = a.y + (size_t)r * a.n + c;
            *to = MODE == F32_ADD ? *to + sum : sum;
        }
        if (MODE == F32_HEAD) {
            static_assert(MODE != F32_HEAD || BN == 32, "a warp per row");
            float bv = there && sum > -INFINITY ? sum : -INFINITY;      // (a NaN is no candidate)
            int bi = there && sum > -INFINITY ? c : 0x7fffffff;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, bv, s);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, s);
                if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
            }
            if (lane == 0 && r < a.rows) {
                a.cand_val[(size_t)r * gridDim.x + blockIdx.x] = bv;
                a.cand_idx[(size_t)r * gridDim.x + blockIdx.x] = bi;
            }
        }
    }
}

// Rotary embedding, K/V write and tree attention of one (row, head) per block of four warps, from the QKV result.  As k_tree_attn_plain:
// per chunk of keys a thread per key for the scores, then the threads as (key group, four columns) for the product with V.  Cached keys and
// the tree's are separate loops: with a choice between them in each step the loads of a step waited for the one before.  The tree's few
// are unrolled by four only (all of it: 255 registers with heads of 128, two blocks per SM instead of three).  us per pass, back to
// back, 2 layers of 3 heads of 128, 3000 positions, 1 / 16 / 33 / 64 / 128 rows: rotary kernel and k_tree_attn_plain 268, 306, 354, 525, 560;
// with the choice and without f32_attn_smem 281, 331, 494, 520, 542; now 263, 309, 295, 401, 541.
constexpr int F32_ATTN_THREADS = 128, F32_CHUNK = 512, F32_ATTN_SMEM = 227 * 1024;
template <int HD>
__global__ void __launch_bounds__(F32_ATTN_THREADS) k_attn_rope_f32(
        const float* __restrict__ qkv, const float* __restrict__ cs, const float* __restrict__ sn, float* __restrict__ q, float* __restrict__ out,
        char* const* __restrict__ base, const int32_t* __restrict__ cap, const int32_t* __restrict__ len, const int32_t* __restrict__ row_seq,
        const int32_t* __restrict__ row_local, const uint64_t* __restrict__ anc, int layer, int H, float scale, const int32_t* status) {
    pdl_enter();
    if (first_thread_of_grid()) trace_mark(status, TK_ATTN);
    if (*status != 0) return;
    constexpr int HALF = HD / 2, QUADS = HD / 4, GROUPS = F32_ATTN_THREADS / QUADS;
    __shared__ __align__(16) float s_q[HD];
    __shared__ float s_p[F32_CHUNK], s_red[2][F32_ATTN_THREADS / 32];
    __shared__ int s_anc[ADED_MAX_NODES];
    __shared__ __align__(16) float s_o[GROUPS][HD];
    const int r = blockIdx.x, hh = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, d = H * HD;
    const int b = row_seq[r], local = row_local[r];
    const int L = len[b];
    const size_t cp = cap[b], slot = (size_t)L + local;
    float* kbase = reinterpret_cast<float*>(base[b]) + (((size_t)layer * 2 + 0) * H + hh) * cp * HD;
    float* vbase = reinterpret_cast<float*>(base[b]) + (((size_t)layer * 2 + 1) * H + hh) * cp * HD;
    // row `local` of this tree's QKV result: q, k and v of this head are `part` x d further
    const float* tree = qkv + (size_t)(r - local) * 3 * d + hh * HD;
    const float *tree_cs = cs + (size_t)(r - local) * HALF, *tree_sn = sn + (size_t)(r - local) * HALF;
    if (tid < HALF) {
        const float c = tree_cs[local * HALF + tid], s = tree_sn[local * HALF + tid];
        const float* row = tree + (size_t)local * 3 * d;
        const float q0 = row[tid], q1 = row[tid + HALF], k0 = row[d + tid], k1 = row[d + tid + HALF];
        s_q[tid] = q0 * c - q1 * s;
        s_q[tid + HALF] = q1 * c + q0 * s;
        q[(size_t)r * d + hh * HD + tid] = s_q[tid];
        q[(size_t)r * d + hh * HD + tid + HALF] = s_q[tid + HALF];
        if (ADED_IN_RANGE(slot < cp, status)) {
            kbase[slot * HD + tid] = k0 * c - k1 * s;
            kbase[slot * HD + tid + HALF] = k1 * c + k0 * s;
            vbase[slot * HD + tid] = row[2 * d + tid];
            vbase[slot * HD + tid + HALF] = row[2 * d + tid + HALF];
        }
    }
    // the keys: cache positions 0 .. L - 1, then the row's ancestors in the tree, in index order
    const uint64_t a_lo = anc[2 * r], a_hi = anc[2 * r + 1];
    static_assert(F32_ATTN_THREADS >= ADED_MAX_NODES, "a thread per possible ancestor");
    {
        const bool on = tid < 64 ? (a_lo >> tid) & 1 : (a_hi >> (tid - 64)) & 1;
        const int before = tid < 64 ? __popcll(a_lo & ((1ull << tid) - 1ull)) : __popcll(a_lo) + __popcll(a_hi & ((1ull << (tid - 64)) - 1ull));
        if (on) s_anc[before] = tid;
    }
    const int n = L + __popcll(a_lo) + __popcll(a_hi);
    __syncthreads();
    const int quad = tid % QUADS, group = tid / QUADS;
    float mx = -INFINITY, sum = 0.f;                 // running maximum (all threads) and this thread's share of the sum
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < n; c0 += F32_CHUNK) {
        const int here = min(F32_CHUNK, n - c0), cached = max(0, min(here, L - c0));      // the first `cached` of them lie in the cache
        float m = -INFINITY;
        int i = tid;
        for (; i < cached; i += F32_ATTN_THREADS) {
            float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
            const float* kr = kbase + (size_t)(c0 + i) * HD;
#pragma unroll
            for (int j = 0; j < QUADS; ++j) {
                const float4 kv = *reinterpret_cast<const float4*>(kr + 4 * j), qv = *reinterpret_cast<const float4*>(s_q + 4 * j);
                e.x = fmaf(qv.x, kv.x, e.x); e.y = fmaf(qv.y, kv.y, e.y); e.z = fmaf(qv.z, kv.z, e.z); e.w = fmaf(qv.w, kv.w, e.w);
            }
            const float s = ((e.x + e.y) + (e.z + e.w)) * scale;
            s_p[i] = s;
            m = fmaxf(m, s);
        }
        for (; i < here; i += F32_ATTN_THREADS) {
            float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
            const int node = s_anc[c0 + i - L];
            const float *kr = tree + (size_t)node * 3 * d + d, *c = tree_cs + node * HALF, *s = tree_sn + node * HALF;
#pragma unroll 4
            for (int j = 0; j < HALF; j += 4) {
                const float4 k0 = *reinterpret_cast<const float4*>(kr + j), k1 = *reinterpret_cast<const float4*>(kr + HALF + j);
                const float4 c4 = *reinterpret_cast<const float4*>(c + j), s4 = *reinterpret_cast<const float4*>(s + j);
                const float4 q0 = *reinterpret_cast<const float4*>(s_q + j), q1 = *reinterpret_cast<const float4*>(s_q + HALF + j);
                e.x = fmaf(q0.x, k0.x * c4.x - k1.x * s4.x, fmaf(q1.x, k1.x * c4.x + k0.x * s4.x, e.x));
                e.y = fmaf(q0.y, k0.y * c4.y - k1.y * s4.y, fmaf(q1.y, k1.y * c4.y + k0.y * s4.y, e.y));
                e.z = fmaf(q0.z, k0.z * c4.z - k1.z * s4.z, fmaf(q1.z, k1.z * c4.z + k0.z * s4.z, e.z));
                e.w = fmaf(q0.w, k0.w * c4.w - k1.w * s4.w, fmaf(q1.w, k1.w * c4.w + k0.w * s4.w, e.w));
            }
            const float sc = ((e.x + e.y) + (e.z + e.w)) * scale;
            s_p[i] = sc;
            m = fmaxf(m, sc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) s_red[0][warp] = m;
        __syncthreads();
        float nm = mx;
#pragma unroll
        for (int w = 0; w < F32_ATTN_THREADS / 32; ++w) nm = fmaxf(nm, s_red[0][w]);
        const float corr = expf(mx - nm);            // (0 before the first chunk)
        mx = nm;
        sum *= corr;
        for (int i = tid; i < here; i += F32_ATTN_THREADS) {
            const float pr = expf(s_p[i] - nm);
            s_p[i] = pr;
            sum += pr;
        }
        __syncthreads();
        acc.x *= corr; acc.y *= corr; acc.z *= corr; acc.w *= corr;
        auto add_v = [&](const float* vr, float pr) {
            const float4 vv = *reinterpret_cast<const float4*>(vr + 4 * quad);
            acc.x = fmaf(pr, vv.x, acc.x); acc.y = fmaf(pr, vv.y, acc.y); acc.z = fmaf(pr, vv.z, acc.z); acc.w = fmaf(pr, vv.w, acc.w);
        };
        i = group;
#pragma unroll 4
        for (; i < cached; i += GROUPS) add_v(vbase + (size_t)(c0 + i) * HD, s_p[i]);
#pragma unroll 4
        for (; i < here; i += GROUPS) add_v(tree + (size_t)s_anc[c0 + i - L] * 3 * d + 2 * d, s_p[i]);
        __syncthreads();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_red[1][warp] = sum;
    *reinterpret_cast<float4*>(&s_o[group][4 * quad]) = acc;
    __syncthreads();
    if (tid < HD) {
        float total = 0.f, o = 0.f;
#pragma unroll
        for (int w = 0; w < F32_ATTN_THREADS / 32; ++w) total += s_red[1][w];
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) o += s_o[g][tid];
        out[((size_t)r * H + hh) * HD + tid] = o * (1.f / total);
    }
}

// ---- host side --------------------------------------------------------------------------------
// Blocks of 16 rows while they are few, 32 from where the widest projection would be more than two waves of them (as in dense.cu).
static int f32_block_rows(const aded_model* m, int rows) {
    const aded_model_config& c = m->cfg;
    const int d = c.d_model, widest = c.vocab > 3 * d ? (c.vocab > 2 * c.d_ffn ? c.vocab : 2 * c.d_ffn) : (3 * d > 2 * c.d_ffn ? 3 * d : 2 * c.d_ffn);
    const long long cols = (widest + 31) / 32, limit = 2ll * ws_grid_limit(m->device);
    return cols * ((rows + 15) / 16) <= limit ? 16 : cols * ((rows + 31) / 32) <= limit ? 32 : 0;
}

// Whether a call of `rows` rows goes this way: all of k in shared memory for every projection, rows that start on 16-byte boundaries.
bool f32_fused(const aded_model* m, int rows) {
    if (!m->f32_ok) return false;
    const int bm = f32_block_rows(m, rows), d = m->cfg.d_model, F = m->cfg.d_ffn, k = d > F ? d : F;
    return bm != 0 && (bm == 16 ? f32_smem<16, 32>(k) : f32_smem<32, 32>(k)) <= F32_SMEM;
}

bool f32_prepare(const aded_model* m) {
    const aded_model_config& c = m->cfg;
    if (c.dtype != ADED_F32 || c.d_model % 4 || c.d_ffn % 4) return false;
    uintptr_t low = reinterpret_cast<uintptr_t>(m->top.lm_head) | reinterpret_cast<uintptr_t>(m->top.final_norm);
    for (const aded_layer_weights& w : m->layers)
        low |= reinterpret_cast<uintptr_t>(w.wqkv) | reinterpret_cast<uintptr_t>(w.wo) | reinterpret_cast<uintptr_t>(w.wgu) | reinterpret_cast<uintptr_t>(w.wd) |
               reinterpret_cast<uintptr_t>(w.norm1) | reinterpret_cast<uintptr_t>(w.norm2);
    if (low % 16 || f32_smem<16, 32>(c.d_model > c.d_ffn ? c.d_model : c.d_ffn) > F32_SMEM) return false;
    bool ok = true;
    auto set = [&](auto* f, int bytes = F32_SMEM) { ok = ok && cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess; };
    set(k_gemm_f32<16, 32, F32_QKV>); set(k_gemm_f32<16, 32, F32_SWIGLU>); set(k_gemm_f32<16, 32, F32_HEAD>); set(k_gemm_f32<16, 32, F32_ADD>);
    set(k_gemm_f32<16, 16, F32_ADD>);
    set(k_attn_rope_f32<64>, F32_ATTN_SMEM - 12 * 1024); set(k_attn_rope_f32<128>, F32_ATTN_SMEM - 12 * 1024);
    set(k_gemm_f32<32, 32, F32_QKV>); set(k_gemm_f32<32, 32, F32_SWIGLU>); set(k_gemm_f32<32, 32, F32_HEAD>); set(k_gemm_f32<32, 32, F32_ADD>);
    return ok;
}

template <int BM, int BN, int MODE>
static void f32_launch(const F32Args& a, cudaStream_t st) {
    launch_k(k_gemm_f32<BM, BN, MODE>, dim3((a.n + BN - 1) / BN, (a.rows + BM - 1) / BM), dim3(F32_THREADS), f32_smem<BM, BN>(a.k), st, a);
}

// One projection with its neighbours; `kind` F32_*.
static void f32_project(aded_model* m, int kind, const void* x, const void* w, const void* gain, float* y, int rows, int n, int k, int trace_kind, cudaStream_t st) {
    F32Args a = {};
    a.x = (const float*)x;
    a.w = (const float*)w;
    a.gain = (const float*)gain;
    a.y = y;
    a.x_out = (float*)m->x;
    a.cand_val = m->cand_val;
    a.cand_idx = m->cand_idx;
    a.rows = rows;
    a.n = n;
    a.k = k;
    a.eps = m->cfg.rms_eps;
    a.status = m->status;
    a.trace_kind = trace_kind;
    const bool small = f32_block_rows(m, rows) == 16;
    if (kind == F32_QKV) small ? f32_launch<16, 32, F32_QKV>(a, st) : f32_launch<32, 32, F32_QKV>(a, st);
    else if (kind == F32_SWIGLU) small ? f32_launch<16, 32, F32_SWIGLU>(a, st) : f32_launch<32, 32, F32_SWIGLU>(a, st);
    else if (kind == F32_HEAD) small ? f32_launch<16, 32, F32_HEAD>(a, st) : f32_launch<32, 32, F32_HEAD>(a, st);
    else if (!small) f32_launch<32, 32, F32_ADD>(a, st);
    // O and down have few columns: narrower blocks while that fills SMs that would be idle
    else if ((long long)((n + 15) / 16) * ((rows + 15) / 16) <= ws_grid_limit(m->device) / 2) f32_launch<16, 16, F32_ADD>(a, st);
    else f32_launch<16, 32, F32_ADD>(a, st);
}

// A layer in five launches: QKV, attention, then O, gate/up and down.
void launch_f32_qkv(aded_model* m, int layer, int rows, cudaStream_t st) {
    const int d = m->cfg.d_model;
    f32_project(m, F32_QKV, m->h, m->layers[layer].wqkv, m->layers[layer].norm1, m->y32, rows, 3 * d, d, TK_GEMM_QKV, st);
}
// Shared memory that a block of the attention asks for and does not use: as much as keeps more blocks from an SM than it must take.  The
// blocks start while the QKV projection still holds SMs, and would crowd onto the others (2 layers of 4 heads of 64, 3000 positions, 33 rows:
// 307 us without, 184 with this).  Where they are few for the SMs that are left they spread anyway, and waiting for a whole SM would cost
// 2 us (16 rows of that shape at 64 positions: 67 without, 69 with); beyond what an SM holds by registers there is nothing to keep apart.
static size_t f32_attn_smem(const aded_model* m, int rows) {
    const int sms = ws_grid_limit(m->device) / 2, blocks = rows * m->cfg.n_heads, per_sm = (blocks + sms - 1) / sms;
    const int bm = f32_block_rows(m, rows), projection = (3 * m->cfg.d_model + 31) / 32 * ((rows + bm - 1) / bm);
    if (per_sm > (m->cfg.head_dim == 128 ? 3 : 4) || 3 * blocks <= 2 * (sms - projection)) return 0;
    return F32_ATTN_SMEM / per_sm - 12 * 1024;        // (beside the 5 KB that it uses and what the device keeps)
}
void launch_f32_attention(aded_model* m, aded_kv* kv, int layer, int rows, cudaStream_t st) {
    const int H = m->cfg.n_heads;
    launch_k(m->cfg.head_dim == 128 ? k_attn_rope_f32<128> : k_attn_rope_f32<64>, dim3(rows, H), dim3(F32_ATTN_THREADS), f32_attn_smem(m, rows), st, m->y32, m->rope_cos, m->rope_sin,
             (float*)m->q, (float*)m->attn, kv->base_dev, kv->cap_dev, kv->len_dev, m->rows.seq, m->rows.local, m->rows.anc, layer, H,
             1.f / sqrtf((float)m->cfg.head_dim), m->status);
}
void launch_f32_rest(aded_model* m, int layer, int rows, cudaStream_t st) {
    const aded_layer_weights& w = m->layers[layer];
    const int d = m->cfg.d_model, F = m->cfg.d_ffn;
    f32_project(m, F32_ADD, m->attn, w.wo, nullptr, (float*)m->h, rows, d, d, TK_GEMM_O, st);
    f32_project(m, F32_SWIGLU, m->h, w.wgu, w.norm2, (float*)m->act, rows, 2 * F, d, TK_GEMM_GU, st);
    f32_project(m, F32_ADD, m->act, w.wd, nullptr, (float*)m->h, rows, d, F, TK_GEMM_DOWN, st);
}

// The final norm and the LM head: logits to `logits`, the normalised rows to m->x, candidates of every 32 columns.
void launch_f32_head(aded_model* m, float* logits, int rows, cudaStream_t st) {
    f32_project(m, F32_HEAD, m->h, m->top.lm_head, m->top.final_norm, logits, rows, m->cfg.vocab, m->cfg.d_model, TK_GEMM_HEAD, st);
}
int f32_candidates(const aded_model* m) { return (m->cfg.vocab + 31) / 32; }

}  // namespace aded
