// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "aded.h"
#include "gemm_out.cuh"

#define ADED_CUDA_TRY(expr)                      \
    do {                                         \
        cudaError_t _e = (expr);                 \
        if (_e != cudaSuccess) {                 \
            aded::note_cuda_error(_e, #expr);    \
            return ADED_ERR_CUDA;                \
        }                                        \
    } while (0)

namespace aded {

void note_cuda_error(cudaError_t e, const char* what);
void note_launch(int n = 1);   // bumps the process-wide launch counter

enum { ARGMAX_CHUNKS = 16 };
enum { PROF_GEMM = 0, PROF_ATTN = 1, PROF_OTHER = 2, PROF_GROUPS = 3 };
struct ProfSpan { int group; int launches; cudaEvent_t a, b; };

// ---- element types ---------------------------------------------------------------------
typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f32<bf16>(float v) { return __float2bfloat16_rn(v); }

// ---- programmatic dependent launch ---------------------------------------------------------
// Every kernel of a pass is launched with the programmatic-serialisation attribute and begins with
// pdl_enter(): it lets the next kernel of the stream start launching at once (its blocks become
// resident and run their own preamble) and then waits until the previous kernel has finished and
// its writes are visible.  Nothing may be read from or written to global memory that another kernel
// of the pass touches before pdl_wait().  Done before it: weights, gains and contributor tables, which no kernel
// writes, and the bf16 attention kernels' first blocks of committed keys and values (attn_sequence says why they may).
// Every block waits, also one that has nothing to do: a kernel waits for the one before it alone, so that a launch none of
// whose blocks waited would let the next kernel run beside whatever came earlier on the stream.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() { pdl_launch_dependents(); pdl_wait(); }

// ---- index checks of the debug build -------------------------------------------------------------
// Compiled with -DADED_DEBUG_CHECKS (python -m paper_2407_12021_b200.build --debug -> libaded_debug.so) the
// kernels test the indices they are about to use on slots, cache rows and table buckets; a failed test
// records ADED_ERR_INTERNAL in the status word and the access is skipped.  In the product build the
// macro is the constant true and costs nothing.
#ifdef ADED_DEBUG_CHECKS
#define ADED_IN_RANGE(cond, status) ((cond) ? true : (atomicCAS(const_cast<int32_t*>(status), 0, (int)ADED_ERR_INTERNAL), false))
#else
#define ADED_IN_RANGE(cond, status) true
#endif

// ---- stage trace ---------------------------------------------------------------------------------
// The status word of a model is the first of a small block of device memory:
//   int32 [0] status, [1] trace switch, [2] marks taken, [3] unused; then TRACE_CAP 64-bit times (ns of
//   the global timer) and TRACE_CAP int32 kinds.
// While the switch is on, every kernel of a pass records, from one thread of its first block, the time at
// which its wait for the previous kernel ended.  The difference between two consecutive marks is the
// time the earlier kernel added to the pass (its overlap with its neighbours included), which is what
// a roofline report of a step chained by programmatic dependent launch needs; event pairs around
// launches would serialise the kernels.
enum { TRACE_CAP = 16384, STATUS_WORDS = 4 + 3 * TRACE_CAP };
enum { TK_OTHER = 0, TK_GEMM_QKV = 1, TK_GEMM_O = 2, TK_GEMM_GU = 3, TK_GEMM_DOWN = 4, TK_GEMM_HEAD = 5, TK_ATTN = 6,
       TK_NORM = 7, TK_ROPE = 8, TK_SWIGLU = 9, TK_PICK = 10, TK_STEP_END = 11 };
__device__ __forceinline__ void trace_mark(const int32_t* status, int kind) {
    int32_t* s = const_cast<int32_t*>(status);
    if (__ldcg(s + 1) == 0) return;
    const int i = atomicAdd(s + 2, 1) & (TRACE_CAP - 1);
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    reinterpret_cast<unsigned long long*>(s + 4)[i] = t;
    (s + 4 + 2 * TRACE_CAP)[i] = kind;
}
__device__ __forceinline__ bool first_thread_of_grid() {
    return threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
}

// (`cluster`: blocks of a cluster along x)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_clusters(int cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    return launch_clusters(1, kernel, grid, block, smem, st, args...);
}

// ---- per-call row bookkeeping (device arrays sized for max_rows / max_batch) --------------
struct RowMeta {
    int32_t* seq;      // [R] sequence of the row
    int32_t* local;    // [R] node index inside its tree
    int32_t* pos;      // [R] rotary position = committed length + depth in the tree
    uint64_t* anc;     // [R][2] bit j set <=> local node j is an ancestor of the row's node, or itself
};

// The caller's arrays of one verify/append call.  Kernels read them through this record, which
// lives at a fixed device address and is rewritten before every call, so that a captured launch
// sequence can be replayed with other arrays.
struct CallPtrs {
    const int32_t* tokens;
    const int32_t* parents;
    int32_t* out_tokens;
    int32_t* out_len;
    int32_t out_stride;
};

// Draft approval of one sequence, by one warp (a tree has at most ADED_MAX_NODES nodes; s_* in shared memory).  A node is
// approved when its parent is approved and its token equals the model's token at the parent -- that is, when all its
// ancestors but the root match, which its ancestor set (`anc`, two words per node, the node itself included) answers at
// once; the deepest approved node (lowest index among equals) ends the accepted path, and the nodes of its ancestor set in
// index order are the path.  Emits the model's token of every path node: the approved drafts' successors, ending with the
// model's own next token, and commits the path's length (the compaction that follows works from `moves`).  A failed pass
// emits nothing and keeps the committed length.  (One thread that walked the nodes took about 4 us of a pass.)
__device__ __forceinline__ void approval_warp(int lane, const int32_t* s_par, const int32_t* s_tok, const int32_t* s_best, const uint64_t* __restrict__ anc,
                                              int T, int pass_status, int32_t* out_tokens, int32_t* out_len, int32_t* path, int32_t* moves, int32_t* len) {
    if (pass_status != 0) {
        if (lane == 0) { *out_len = 0; moves[1] = 0; }
        return;
    }
    constexpr int PER = ADED_MAX_NODES / 32;
    static_assert(PER == 4, "two 64-bit words of nodes");
    uint64_t lo[PER], hi[PER], matched[2] = {0, 0};
#pragma unroll
    for (int c = 0; c < PER; ++c) {
        const int i = c * 32 + lane;
        lo[c] = i < T ? anc[2 * i] : 0;
        hi[c] = i < T ? anc[2 * i + 1] : 0;
        const bool match = i < T && (i == 0 || s_tok[i] == s_best[s_par[i]]);
        matched[c >> 1] |= (uint64_t)__ballot_sync(0xffffffffu, match) << ((c & 1) * 32);
    }
    unsigned key = 0;                       // (depth + 1, lowest index first)
#pragma unroll
    for (int c = 0; c < PER; ++c) {
        const int i = c * 32 + lane;
        const bool ok = i < T && ((lo[c] & ~matched[0]) | (hi[c] & ~matched[1])) == 0;
        const unsigned mine = ok ? (unsigned)(__popcll(lo[c]) + __popcll(hi[c])) << 8 | (unsigned)(ADED_MAX_NODES - 1 - i) : 0u;
        key = max(key, mine);
    }
    key = __reduce_max_sync(0xffffffffu, key);
    const int deepest = ADED_MAX_NODES - 1 - (int)(key & 255u), n = (int)(key >> 8);
    uint64_t on_lo = 0, on_hi = 0;
#pragma unroll
    for (int c = 0; c < PER; ++c) {
        const uint64_t l = __shfl_sync(0xffffffffu, lo[c], deepest & 31), h = __shfl_sync(0xffffffffu, hi[c], deepest & 31);
        if (c == deepest >> 5) { on_lo = l; on_hi = h; }
    }
#pragma unroll
    for (int c = 0; c < PER; ++c) {
        const int i = c * 32 + lane;
        const uint64_t word = c < 2 ? on_lo : on_hi, below = (1ull << (i & 63)) - 1ull;
        if ((word >> (i & 63)) & 1) {
            const int at = __popcll(word & below) + (c < 2 ? 0 : __popcll(on_lo));
            path[at] = i;
            out_tokens[at] = s_best[i];
        }
    }
    if (lane == 0) {
        *out_len = n;
        moves[0] = *len;
        moves[1] = n;
        *len += n;
    }
}

// The bf16 attention kernels read before their dependency wait: this order, a sequence's committed length and tree size, and the first
// blocks of committed keys and values.  What a failed pass or another call has left there is caught by reading order, length and
// size again after the wait.  Rows BELOW the length that was read have to be final by then: the approval of a pass
// publishes the new length before the compaction behind it has moved the rows.  So the kernels that launch right before
// attention (rotary and K/V write) release it only after their own wait: when a block of attention starts, every earlier
// kernel on the stream, compaction included, has finished.  (Released at the top of that kernel, a small model whose
// projections do the same would have the whole chain from approval to attention resident at once.)
//
// Sequence of blockIdx.z: z / row_blocks-th in order of work, kept in range.
__device__ __forceinline__ int attn_sequence(const int32_t* order, int z, int row_blocks, int batch) {
    const int place = z / row_blocks;
    return order ? min(max(__ldcg(order + place), 0), batch - 1) : place;
}

struct SeqMeta {
    int32_t* row_off;  // [B+1] first row of each sequence
    int32_t* path;     // [B][ADED_MAX_NODES] accepted path (local node indices), root first
    int32_t* order;    // [B] sequences by falling number of keys (the attention kernel's order of work)
    int32_t* moves;    // [B][2] committed length before this call, and how many nodes of the path were kept (compaction)
};

// The rotary tables of a pass: cos/sin of position * theta^(-2i/hd) for every row, in double, stored as float (the angles reach
// thousands of radians, where float argument reduction would cost several bf16 ulps).
struct RopeArgs {
    const double* freq;      // [half]
    float* cs;               // [R][half]
    float* sn;
    int half;
};
}  // namespace aded

namespace aded {
// What the weight-streaming GEMM leaves behind (gemm_ws.cu): the partial tiles alone, or also -- the LM
// head -- per-row greedy candidates of every tile, reduced in the kernel's tail.
enum { WS_EPI_SLOTS = 0, WS_EPI_ARGMAX = 1 };
struct WsEpilogue {
    int mode;
    const TileRef* tiles;        // contributors of every tile
    uint32_t* counters;          // one arrival counter per tile; never reset: the epoch-th launch waits for
    uint32_t epoch;              //   n x epoch arrivals (modulo 2^32)
    float* cand_val; int32_t* cand_idx;   // best logit and its column per (row, tile): [R][n_tiles]
};

// What the GEMM for calls of many rows (gemm_many.cu) does with its complete results.
enum { MANY_PLAIN = 0, MANY_ROPE = 1, MANY_RESIDUAL = 2, MANY_SWIGLU = 3, MANY_ARGMAX = 4 };
struct ManyEpilogue {
    int kind;
    float* out;              // PLAIN: [tile][rb][128] fp32
    int rb;
    bf16* h;                 // RESIDUAL: h += y
    bf16* act;               // SWIGLU
    float* cand_val;         // ARGMAX: best logit of 32 columns and its column, [R][vocab / 32]
    int32_t* cand_idx;
    // ROPE: rotated q, and k and v to the cache (as k_rope_kv_ws)
    const float* cs;
    const float* sn;
    bf16* q;
    char* const* base;
    const int32_t* cap;
    const int32_t* len;
    const int32_t* row_seq;
    const int32_t* row_local;
    int layer, heads, hd, d;
};
}  // namespace aded

struct aded_kv {
    const aded_model* model;
    int device;
    int batch;
    size_t elem;                  // bytes per element
    std::vector<int32_t> cap;     // host copy of capacities
    std::vector<char*> base;      // host copy of the per-sequence block pointers (device memory)
    char** base_dev;              // [B] device array of the same pointers
    int32_t* cap_dev;             // [B]
    int32_t* len_dev;             // [B] committed lengths
    CUtensorMap* maps_dev;        // [B] TMA descriptors of the blocks (tensor-core attention), or NULL
};

struct aded_model {
    aded_model_config cfg;
    int device;
    aded_weights top;
    std::vector<aded_layer_weights> layers;
    size_t elem;

    // activations, all [max_rows, *]
    void* h;        // residual stream            [R, d]   model dtype
    void* x;        // normalised input of a GEMM [R, d]
    void* q;        // rotated queries            [R, d]
    void* attn;     // attention output           [R, d]
    void* act;      // SwiGLU product             [R, F]
    float* y32;     // fp32 GEMM output, widest of 3d / 2F / d columns
    float* logits;  // [R, V] fp32
    float* rope_cos;  // [R, hd/2]
    float* rope_sin;
    double* rope_freq;  // [hd/2]
    int32_t* best;    // [R] greedy token per row
    int32_t* tokens;  // [R] staging for the _host entry points
    int32_t* parents;
    int32_t* out_tokens;   // [R]
    int32_t* out_len;      // [max_batch]
    int32_t* status;  // device status word
    aded::RowMeta rows;
    aded::SeqMeta seqs;
    aded::CallPtrs* call_dev;   // device copy of the current call's array pointers
    std::vector<void*> owned;   // everything cudaMalloc'ed for this handle

    // sampling-mode verification (aded_verify_sampled): armed for one call
    bool samp_on;
    float samp_temp, samp_top_p;
    const float* samp_u;        // caller's [rows] uniform numbers (device)

    void* step_mcts;            // scratch of aded_decode_step_mcts (allocated on first use)

    float* dbg_logits;
    int32_t* dbg_best;
    void* dbg_hidden;   // [n_layers + 1][rows][d] copies of the residual stream (debug capture)

    bool att_mma;       // bf16 models: tensor-core split-KV attention kernel
    bool att_tc;        // bf16 models with head_dim 128: the tcgen05 attention kernel (tree_attention_tc.cu)
    bool att_tc_ok;     // the tcgen05 kernel can be used (aded_debug_attention_kernel switches between the two)
    CUtensorMap att_q_map;   // TMA descriptor of q for it

    // tensor-core GEMM path (bf16 models): TMA descriptors and split-tile scratch
    bool ws_ready;
    std::vector<CUtensorMap> ws_maps;   // per layer: wqkv, wo, wgu, wd; then lm_head
    CUtensorMap ws_x_maps[3][16];       // x, attn, act in boxes of 16, 32, .. 256 rows: the rows of a pass are one request
    std::vector<void*> ws_tiled;        // the weight matrices re-tiled for the tensor-core GEMM (same indices as ws_maps), model-owned
    std::vector<CUtensorMap> ws_tiled_maps, ws_half_maps;   // calls of many rows: descriptors of the re-tiled copies, and of the caller's matrices, half a tile per box
    bool ws_use_tiled;                  // GEMMs read the re-tiled copies (else the caller's matrices through ws_maps)
    bool many_ok;                       // the kernel for calls of many rows can be used
    aded::TileRef* many_tiles;          // "tile t is slot t, complete" (aded_debug_gemm)
    uint32_t* many_flags;               // its hand-over flags, [many_flag_count]
    float* ws_slots;                    // partial result tiles (see gemm_out.cuh)
    aded::TileRef* ws_tiles[5];         // contributor tables of the wqkv, wo, wgu, wd and LM-head results
    int ws_contributors[5];             // most contributors of any of their tiles
    bool ws_one_per_sm[5];              // which of those five GEMMs launch one CTA per SM instead of two
    uint32_t* ws_counters;              // arrival counters of the LM head's tail, one per tile
    uint32_t ws_epoch;                  // LM-head launches with a tail so far (host side of the counters)
    float* cand_val;                    // [R][vocab / 128] per-tile greedy candidates of the LM head
    int32_t* cand_idx;

    bool f32_ok;            // fp32 model that dense_f32.cu takes, for calls of few rows (f32_fused)
    float* argmax_val;      // [R][ARGMAX_CHUNKS] best logit of each column chunk
    int32_t* argmax_idx;

    bool prof_on;
    float prof_ms[aded::PROF_GROUPS];             // harvested so far
    int32_t prof_n[aded::PROF_GROUPS];
    std::vector<aded::ProfSpan> prof_spans;   // spans recorded by direct launches since aded_profile_begin
    std::vector<cudaEvent_t> prof_pool;       // events kept for reuse
};

namespace aded {

inline RopeArgs rope_args(const aded_model* m) {
    return RopeArgs{m->rope_freq, m->rope_cos, m->rope_sin, m->cfg.head_dim / 2};
}

// ---- launchers (each enqueues on `st`; shapes are validated by the callers) ---------------
// tree.cu
// Calls of up to PROLOGUE_MAX_BATCH sequences pass their record and row offsets to the prologue, which publishes them; larger
// ones have copied them before.
enum { PROLOGUE_MAX_BATCH = 64 };
// checks, row bookkeeping, embedding lookup, the first RMSNorm and the rotary tables
void launch_pass_begin(aded_model* m, aded_kv* kv, const CallPtrs& call, const int32_t* offsets_host, int batch, int rows, int chain_mode, cudaStream_t st);
void launch_accept(aded_model* m, aded_kv* kv, int batch, cudaStream_t st);
void launch_compact(aded_model* m, aded_kv* kv, int batch, cudaStream_t st);
void launch_kv_copy(char* cache_k, char* cache_v, size_t head_bytes, void* user_k, void* user_v, size_t bytes, int heads, bool load, cudaStream_t st);
void launch_commit_chain(aded_model* m, aded_kv* kv, int batch, cudaStream_t st);

// dense.cu
void launch_rope_freq(double* freq, int half, double theta);
// projection result added to the residual stream, then the norm
void launch_add_rmsnorm(aded_model* m, const GemmOut& y, const void* gain, cudaStream_t st);
bool gemm_plain_prepare(bool bf16_model);
// w_map / x_map: index into m->ws_maps / m->ws_x_maps of the operands' TMA descriptors (-1: none, plain kernel).
// `y` is the fp32 buffer the plain kernel writes; the returned descriptor says where the result is.
// `epi_mode` (WS_EPI_*): whether the tensor-core kernel's tail also leaves per-tile greedy candidates (LM head).
// A call is worked in passes of gemm_pass_rows rows: the result of rows [row0, row0 + rows), to be consumed before the next.
int gemm_pass_rows(const aded_model* m, int rows);
// The same for all rows of a call of many rows, result and all, where gemm_is_many.
bool gemm_is_many(const aded_model* m, int rows, int n, int k);
void launch_gemm_many(aded_model* m, int w_map, int x_map, int rows, int n, int k, const ManyEpilogue& epi, int trace_kind, cudaStream_t st);
// The norm alone (h is complete).
void launch_rmsnorm(aded_model* m, int rows, const void* gain, cudaStream_t st);
GemmOut launch_gemm(aded_model* m, int w_map, int x_map, const void* x, const void* w, float* y, int row0, int rows, int n, int k,
                    int epi_mode, int trace_kind, cudaStream_t st);
void launch_rope_kv(aded_model* m, aded_kv* kv, const GemmOut& qkv, int layer, cudaStream_t st);
void launch_swiglu(aded_model* m, const GemmOut& gu, cudaStream_t st);
void launch_argmax(aded_model* m, const GemmOut& logits, cudaStream_t st);
// Writes a projection result as a plain [rows, n] fp32 matrix (debug paths).
void launch_materialize(aded_model* m, const GemmOut& src, float* dst, cudaStream_t st);

// dense_f32.cu: fp32 models of small widths, calls of few rows
bool f32_prepare(const aded_model* m);
bool f32_fused(const aded_model* m, int rows);
int f32_candidates(const aded_model* m);        // per row, of the LM head's result
void launch_f32_qkv(aded_model* m, int layer, int rows, cudaStream_t st);
void launch_f32_attention(aded_model* m, aded_kv* kv, int layer, int rows, cudaStream_t st);
void launch_f32_rest(aded_model* m, int layer, int rows, cudaStream_t st);
void launch_f32_head(aded_model* m, float* logits, int rows, cudaStream_t st);

// dense_ws.cu: bf16 consumers of slot-resident projection results
void launch_add_rmsnorm_ws(aded_model* m, const GemmOut& y, const void* gain, cudaStream_t st);
void launch_swiglu_ws(aded_model* m, const GemmOut& gu, cudaStream_t st);
void launch_rope_kv_ws(aded_model* m, aded_kv* kv, const GemmOut& qkv, int layer, cudaStream_t st);
// greedy token per row from n candidates (value, column) each, then the approval walk (one launch)
void launch_pick_accept(aded_model* m, aded_kv* kv, int batch, const float* cand_val, const int32_t* cand_idx, int n, cudaStream_t st);

// gemm_ws.cu
bool ws_make_map(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows);
bool ws_make_tiled_map(CUtensorMap* map, const void* ptr, uint64_t units);
bool ws_supported(int n, int k);
bool ws_prepare();
bool attn_prepare();
int ws_grid_limit(int device);
int ws_grid(int device, int n, int k, bool one_per_sm);
size_t ws_slot_floats(int device, int max_n, int max_rows);
cudaError_t ws_retile(const void* w, void* out, int n, int k, cudaStream_t st);
cudaError_t ws_launch(const CUtensorMap& map_w, const void* w_tiled, const CUtensorMap& map_x, int rows, int row0,
                      int n, int k,
                      float* slots, int32_t* status, const WsEpilogue& epi, int trace_kind, int device, bool one_per_sm, cudaStream_t st);
// gemm_many.cu: calls of many rows
bool many_prepare();
int many_block_rows(int device, int rows, int n, int k);      // 0: not a call for it
size_t many_flag_count(int device);
cudaError_t many_wait_probe(uint32_t* flag, long long limit, int32_t* status, cudaStream_t st);
cudaError_t many_silu_check(uint32_t first, uint64_t count, uint64_t* differ, cudaStream_t st);
cudaError_t many_launch(const CUtensorMap& map_w, bool tiled, const CUtensorMap* x_maps, int rows, int block_rows, int n, int k, int ws_ctas,
                        float* partial, uint32_t* flags, int32_t* status, const ManyEpilogue& epi, int trace_kind, int device, cudaStream_t st);
enum { WS_MAP_QKV = 0, WS_MAP_O = 1, WS_MAP_GU = 2, WS_MAP_D = 3 };   // per-layer map order
enum { WS_X = 0, WS_X_ATTN = 1, WS_X_ACT = 2 };
cudaError_t ws_wait_probe(int which, long long limit_cycles, const uint32_t* never_raised, int32_t* status, cudaStream_t st);

// sample.cu
bool sample_supported(int vocab);
cudaError_t launch_sample_rows(const float* logits, int rows, int vocab, int ld, float temperature, float top_p, const float* u,
                               int32_t* out, const int32_t* status, cudaStream_t st);

// tree_attention_tc.cu
bool attn_tc_supported(const aded_model_config& c);
bool attn_tc_prepare();
bool attn_tc_make_kv_map(CUtensorMap* map, const void* block, uint64_t capacity, uint64_t planes);
void launch_tree_attention_tc(aded_model* m, aded_kv* kv, int layer, int batch, int max_tree, cudaStream_t st);

// tree_attention.cu
// max_tree: most nodes any sequence's tree has in this call
void launch_tree_attention(aded_model* m, aded_kv* kv, int layer, int batch, int rows, int max_tree, cudaStream_t st);

}  // namespace aded
