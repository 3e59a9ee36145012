// Shared declarations of the folded-MoE CUDA library (sm_100a only).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/exfold.h"

namespace exfold {

// The first 256 bytes of every workspace hold the device status record.
struct DeviceStatus {
    int code;    // 0 or EXFOLD_ERR_DEVICE_TIMEOUT
    int where;   // which wait gave up (kernel-specific tag)
    int detail;  // block index
    int pad0;
    int queue[2];  // work counters of the mixed GEMMs, cleared by the call's routing kernel
    int pad[58];
};
static_assert(sizeof(DeviceStatus) == 256, "status record is 256 bytes");

constexpr int kMaxExperts = 256;  // routed experts
constexpr int kMaxTopK = 32;
constexpr int kMaxGroups = kMaxExperts + 1;  // + shared expert
constexpr int kTileM = 128;                  // token rows per prefill GEMM tile
constexpr int kGemmBK = 64;  // K elements per pipeline stage of the tensor-core GEMMs: 128-byte rows, 128-byte swizzle
constexpr int kMaxDecodeBatch = 256;
constexpr int kMaxCtas = 160;                // persistent grids never exceed this (148 SMs on B200)

__device__ __forceinline__ void report_timeout(DeviceStatus* st, int where) {
    if (atomicCAS(&st->code, 0, EXFOLD_ERR_DEVICE_TIMEOUT) == 0) {
        st->where = where;
        st->detail = (int)blockIdx.x;
    }
}

// host-side launch accounting
void count_launch(int n = 1);
// Synchronises the stream, decodes and clears the device status record at `rec`
int read_status_record(void* rec, cudaStream_t s);

// Programmatic dependent launch: every kernel of the library is launched with the "programmatic stream
// serialization" attribute, lets its successor be scheduled early (grid_dep_launch) and waits for its
// predecessor's results (grid_dep_wait) before it touches global memory. This removes the several
// microseconds of launch latency between dependent kernels of one call. Both are no-ops when the
// kernel was launched without the attribute.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Raises a kernel's dynamic shared memory limit on the current device to the most a block may have, once per host thread
// (a driver call for each launch cost ~0.4 us of a 12 us call); an error if `bytes` is more
cudaError_t ensure_smem_bytes(const void* kernel, size_t bytes);
template <typename... KArgs>
cudaError_t ensure_smem(void (*kernel)(KArgs...), size_t bytes) {
    return ensure_smem_bytes(reinterpret_cast<const void*>(kernel), bytes);
}

// Programmatic launch is requested per call chain: it pays for chains of short, latency-bound kernels and measured slower
// where prefill runs CTA pairs (early-resident successors compete with the running kernel).
void set_pdl(bool on);
bool pdl_enabled();

// Order-preserving map float -> uint32 (larger float <=> larger key), so warp arg-max / arg-min can use
// the hardware integer reductions (redux.sync) instead of shuffle trees.
// -0.0 and +0.0 compare equal as floats, so they get one key (a tie, which the lower expert id then wins).
__device__ __forceinline__ uint32_t float_order_key(float f) {
    uint32_t b = __float_as_uint(f);
    if (b == 0x80000000u) b = 0u;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float float_from_order_key(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
// The same for the doubles that pools are ranked by. Any two images compare, those of NaN too, so ranks counted on them are
// places that no two experts share and none leaves out.
__device__ __forceinline__ long long score_order_key(double score) {
    const long long b = __double_as_longlong(score + 0.0);  // -0.0 as +0.0
    return b < 0 ? b ^ 0x7FFFFFFFFFFFFFFFll : b;            // negative: larger magnitude = smaller
}
// Warp-wide (value desc, id asc) arg-max. Lanes without a candidate pass has = false. Returns the
// winning id to every lane and its key through *key_out. At least one lane must have a candidate.
__device__ __forceinline__ int warp_argmax(bool has, uint32_t key, int id, uint32_t* key_out) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, has ? key : 0u);
    const int best = __reduce_min_sync(0xffffffffu, (has && key == m) ? id : 0x7fffffff);
    *key_out = m;
    return best;
}
// Warp-wide (value asc, id asc) arg-min over lanes with has = true.
__device__ __forceinline__ int warp_argmin(bool has, uint32_t key, int id) {
    const uint32_t m = __reduce_min_sync(0xffffffffu, has ? key : 0xffffffffu);
    return __reduce_min_sync(0xffffffffu, (has && key == m) ? id : 0x7fffffff);
}

// A token's Top-K and its softmax weights in double, by one warp: v[q] = score of expert lane + 32 q (NPL = ceil(N / 32) or
// more). Lane k < K returns the weight of route k (router order, ties -> lower id) and its expert through *id.
template <int NPL>
__device__ __forceinline__ double warp_topk_softmax(const float (&v)[NPL], int N, int K, int lane, int* id) {
    uint32_t key_q[NPL];
    uint32_t used = 0;
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
        key_q[q] = float_order_key(v[q]);
        if (lane + 32 * q >= N) used |= 1u << q;
    }
    int my_id = -1;
    float my_r = 0.f;
    for (int k = 0; k < K; ++k) {
        uint32_t bk = 0;
        int be = 0x7fffffff;
#pragma unroll
        for (int q = 0; q < NPL; ++q) {
            const bool free_q = !((used >> q) & 1u);
            if (free_q && (be == 0x7fffffff || key_q[q] > bk)) {
                bk = key_q[q];
                be = lane + 32 * q;
            }
        }
        uint32_t mk;
        be = warp_argmax(be != 0x7fffffff, bk, be, &mk);
        if ((be & 31) == lane) used |= 1u << (be >> 5);
        if (lane == k) {
            my_id = be;
            my_r = float_from_order_key(mk);
        }
    }
    const float rmax = __shfl_sync(0xffffffffu, my_r, 0);
    const double ex = lane < K ? exp((double)my_r - (double)rmax) : 0.0;
    double sum = 0.0;
    for (int k = 0; k < K; ++k) sum += __shfl_sync(0xffffffffu, ex, k);  // slot order, like the definition
    *id = my_id;
    return ex / sum;
}

// Programmatic launch; cluster > 1: the grid split into thread-block clusters (distributed shared memory)
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, unsigned cluster,
                               cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    if (pdl_enabled()) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
    count_launch();
    return e;
}
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
    return launch_pdl_cluster(kernel, grid, block, smem, 1, s, args...);
}

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) / 16 * 16; }
inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// ---------------------------------------------------------------- routing (prefill)
struct PrefillRouteParams {
    const float* logits;  // [T][N]
    const float* S;       // [N][N]
    const float* L;       // [N][N]
    const float* lnh;     // [N], or null: ranked by the scores alone
    int64_t T;
    int N, K, Kp;
    float loss_thr;     // pairs with loss above it are not admissible targets (+inf: off)
    int rescale;        // keep the original routed-weight sum after folding
    int confidence;     // confidence-aware split of the folded weight
    int32_t* ids;       // [T][Kp]
    float* w;           // [T][Kp]
    int32_t* omit_src;  // [T][K-Kp] or null
    int32_t* omit_tgt;  // [T][K-Kp] or null
    int32_t* block_hist;  // [nblk][N]
    int32_t* sb_hist;     // [ceil(nblk / kRouteSuperBlock)][N] retained routes per (super-block, expert); the
                          //   launcher clears it, the blocks add to it (not with a single super-block)
    DeviceStatus* status; // cleared by block 0 (first kernel of a call); may be null
    int* queue;           // DeviceStatus::queue, cleared by block 0; may be null
};
constexpr int kRouteTokensPerBlock = 32;
constexpr int kRouteThreads = 512;
constexpr int kRouteMaxThreads = 1024;  // a warp per token of the block
constexpr int kRouteFewBlocks = 148;    // up to this many blocks the kernels spread them over more threads or blocks
constexpr int kRouteSuperBlock = 64;  // blocks per super-block of the two-level histogram

// Row tiles of a group for the mixed GEMMs (gemm_mixed.cu): whole 256-row items, and one ragged item of the rest. A rest above
// kRaggedMax rows takes a whole item's time as it is: masked rows of a whole item.
constexpr int kRaggedMax = 224;
constexpr int kMixedTiles = 0;  // as tile_rows: the work list counts these
__host__ __device__ inline int whole_items(int rows) { return rows / 256 + (rows % 256 > kRaggedMax ? 1 : 0); }
__host__ __device__ inline int ragged_rows(int rows) { return rows % 256 > kRaggedMax ? 0 : rows % 256; }
__host__ __device__ inline int row_tiles(int rows, int tile_rows) {
    return tile_rows == kMixedTiles ? whole_items(rows) + (ragged_rows(rows) > 0 ? 1 : 0) : (rows + tile_rows - 1) / tile_rows;
}

struct PrefillScatterParams {
    int64_t T;
    int N, n_shared, Kp, d_bytes;  // d_bytes: bytes of one x row (0: no gather)
    int nblk;                   // blocks of the route kernel (= blocks of this kernel)
    int tile_rows;              // rows per tile of the work list (kTileM, the fp32 FFN's, or kMixedTiles)
    int split;                  // blocks per token block (set by the launcher)
    const int32_t* ids;         // [T][Kp]
    const float* w;             // [T][Kp]
    const int32_t* block_hist;  // [nblk][N] retained routes per (block, expert)
    const int32_t* sb_hist;     // [ceil(nblk / kRouteSuperBlock)][N] the same per super-block
    int32_t* offsets;           // [G+1] out: first sorted row of each group
    int32_t* work_start;        // [G+1] out: prefix of row tiles per group
    const void* x;      // [T][d]
    void* xs;           // [R][d] gathered rows (may be null)
    int32_t* perm;      // [R]
    int32_t* row_tok;   // [R + T*n_shared]
    float* row_w;       // [R + T*n_shared]
    int32_t* inv_pos;   // [R] sorted row of each route (inverse of perm); may be null
    int32_t* zero;      // words to clear on the way (calibration: the pair sums); may be null
    int zero_words;
};

cudaError_t launch_prefill_route(PrefillRouteParams p, cudaStream_t s);
cudaError_t launch_prefill_scatter(PrefillScatterParams p, cudaStream_t s);

// ---------------------------------------------------------------- routing (decode)
struct DecodeRouteParams {
    const float* logits;  // [B][N]
    const float* S;
    const float* L;
    const float* h;
    int B, N, K, M, n_shared;
    int tile_rows;              // rows per tile of grp_tiles
    // static pool (all null for the dynamic pool of Eq. 11): precomputed pool, targets and scalars
    const int32_t* st_pool;    // [M]
    const int32_t* st_target;  // [N]
    const float* st_scale;     // [N]
    // metadata (workspace copies)
    int32_t* pool_ids;    // [N] (-1 padded)
    int32_t* pool_size;   // [1]
    uint32_t* pool_mask;  // [8]
    int32_t* ids;         // [B][K]
    float* w;             // [B][K]
    int32_t* target;      // [N]
    float* scale;         // [N]
    // execution lists: rows sorted by pool rank (then shared expert), duplicates merged
    int32_t* row_tok;     // [B*K + B]
    float* row_w;         // [B*K + B]
    int32_t* grp_expert;  // [N+1] expert id of each group (pool order; shared last)
    int32_t* grp_off;     // [N+2] first row of each group
    int32_t* grp_tiles;   // [N+2] prefix of row tiles per group (work list of the expert FFN)
    int32_t* slot_row;    // [B][K] row of each routed slot, -1 for a slot merged into an earlier one
    int32_t* n_groups;    // [3]: number of groups, total rows, first row of the shared expert's group
    DeviceStatus* status; // cleared here (first kernel of a decode call)
};
cudaError_t launch_decode_route(const DecodeRouteParams& p, cudaStream_t s);

// Token-parallel half of decode routing for bf16 layers (one CTA per token): optional router scores, Top-K,
// softmax weights in double; clears the status record
struct DecodeTopkParams {
    const float* logits;            // [B][N] (w_router == null)
    const __nv_bfloat16* x;         // [B][d]  (w_router != null)
    const __nv_bfloat16* w_router;  // [N][d] or null
    float* logits_out;              // [B][N] (w_router != null)
    int B, N, K, d;
    int32_t* ids;   // [B][K] routed experts in router order
    double* w64;    // [B][K] their softmax weights
    DeviceStatus* status;
};
cudaError_t launch_decode_topk(const DecodeTopkParams& p, cudaStream_t s);

// Decode, bf16 layers: the gate/up half of the expert FFN over the pool. The kernel finishes the routing in its
// prologue (every CTA: pool of Eq. 11 from the routed weights, minimum-loss targets of Eq. 12, remap of Eq. 14,
// rows per group), streams the pool's gate and up weights once against x read in place, and leaves H (compact rows)
// and the execution lists for the grouped down projection (ffn_decode.cu)
struct DecodeFfnParams {
    CUtensorMap tm_x;     // x [B][d], box a_rows x 64
    CUtensorMap tm_xg;    // x, box 1 x 64: rows gathered four at a time (more than 128 tokens)
    CUtensorMap tm_wg;    // W_gate as [(E*I)][d], box 128 x 64
    CUtensorMap tm_wu;    // W_up
    CUtensorMap tm_wg64;  // the same with 64-row boxes (half-width items)
    CUtensorMap tm_wu64;
    CUtensorMap tm_wg_alt;  // and with boxes of alt rows
    CUtensorMap tm_wu_alt;
    int alt;                // 96, 32 or 0: decode_ffn_alt
    const int32_t* ids;   // [B][K] from the top-k kernel
    const double* w64;    // [B][K]
    const float* S;       // tables (dynamic pool)
    const float* L;
    const float* h;
    const int32_t* st_pool;    // static pool (all null for the dynamic pool)
    const int32_t* st_target;
    const float* st_scale;
    int B, N, K, M, n_shared, d, I, a_rows;
    int stages, scratch_off;  // shared-memory plan made by the launcher
    // metadata written by CTA 0 (workspace copies; all null when the caller asks for none)
    int32_t* pool_ids;    // [N] (-1 padded)
    int32_t* pool_size;   // [1]
    uint32_t* pool_mask;  // [8]
    int32_t* out_ids;     // [B][K] remapped
    float* out_w;         // [B][K]
    int32_t* target;      // [N]
    float* scale;         // [N]
    // execution lists: one row per distinct (token, pool expert), grouped by pool rank (shared expert last)
    __nv_bfloat16* H;     // [rows][I]
    int32_t* row_tok;     // [rows]
    float* row_w;         // [rows] merged weight of the row
    int32_t* slot_row;    // [B][K] row of each routed slot, -1 for a slot merged into an earlier one
    int32_t* grp_expert;  // [G]
    int32_t* grp_off;     // [G+1]
    int32_t* grp_tiles;   // [G+1] prefix of 128-row tiles per group
    int32_t* n_groups;    // [3]: groups, rows, first row of the shared expert's group
    DeviceStatus* status;
};
cudaError_t launch_decode_ffn(const DecodeFfnParams& p, int sms, cudaStream_t s);
int decode_ffn_alt(int B, int max_groups, int I, int sms);
size_t decode_ffn_smem_plan(int B, int K, int N, int alt, int* stages, int* scratch_off, int* a_rows);
// Decode of at most kSmallDecodeBatch tokens, bf16 layers: two kernels (decode_small.cu). Prefill calls that short run the
// same two after their own routing.
constexpr int kSmallDecodeBatch = 8;
struct DecodeSmallParams {
    const __nv_bfloat16* x;
    const __nv_bfloat16* wg;
    const __nv_bfloat16* wu;
    const __nv_bfloat16* wd;
    __nv_bfloat16* y;
    const float* logits;  // [B][N], or null: ids and w64 come from the top-k kernel
    const int32_t* ids;
    const double* w64;
    const float* w_in;    // prefill: the routes' final weights [B][K]; ids are then executed as they are, no pool, no remap
    const float* S;
    const float* L;
    const float* h;
    const int32_t* st_pool;    // static pool (all null for the dynamic pool)
    const int32_t* st_target;
    const float* st_scale;
    int B, N, K, M, n_shared, d, I;
    int max_groups, max_rows;  // bounds of the lists below
    int split;                 // set by the launcher
    // metadata (all null when the caller asks for none)
    int32_t* pool_ids;
    int32_t* pool_size;
    uint32_t* pool_mask;
    int32_t* out_ids;
    float* out_w;
    int32_t* target;
    float* scale;
    // one row per distinct (token, pool expert)
    __nv_bfloat16* H;     // [rows][I]
    int32_t* row_tok;
    float* row_w;
    int32_t* row_grp;
    int32_t* grp_expert;
    int32_t* n_groups;    // [2]: groups, rows
    DeviceStatus* status; // cleared here when this is the call's first kernel (else null)
};
bool decode_small_fits(int B, int K, int d, const void* wg, const void* wu, const void* wd);
// route: prefill whose tokens the gate/up kernel routes itself (no metadata; ids and w_in unused), or null
cudaError_t launch_decode_small(DecodeSmallParams p, const PrefillRouteParams* route, int sms, cudaStream_t s);
cudaError_t launch_static_pool(int N, int M, const float* S, const float* L, const float* h, int32_t* pool_ids,
                               int32_t* target, float* scale, cudaStream_t s);

// ---------------------------------------------------------------- fp32 expert FFN (CUDA cores)
struct FfnF32Params {
    const float* x;  // [x_rows][d]
    const float* wg;
    const float* wu;
    const float* wd;
    int d, I, G;                  // G: groups (upper bound when n_groups_dev is given)
    int tile_rows;                // rows per tile
    int fpc, hld;                 // set by the launcher: features per CTA (tall tiles), row pitch of H in shared memory
    int64_t x_rows;               // without row_tok: row r reads token r % x_rows
    const int32_t* offsets;       // [G+1] first sorted row of each group
    const int32_t* tile_start;    // [G+1] prefix of row tiles (tile_rows each)
    const int32_t* grp_expert;    // [G] expert of each group (null: the group itself)
    const int32_t* n_groups_dev;  // groups known only on the device (decode)
    const int32_t* row_tok;       // [rows] token of each sorted row, or null
    const float* row_w;           // [rows]; read when y is set
    float* out;                   // [rows][d] unweighted expert outputs, or
    float* y;                     // [tokens][d]: every token has one row, stored weighted (out unused)
};
int ffn_f32_tile_rows(int64_t rows, int G, int d, int I, int sms);
// Prefill of few tokens: the FFN kernel routes the tokens itself and writes the permutation (p.offsets, tile_start, row_tok,
// row_w unused)
struct FfnF32Route {
    PrefillRouteParams r;  // block_hist, sb_hist unused
    int n_shared;
    int32_t* offsets;      // as PrefillScatterParams
    int32_t* perm;
    int32_t* inv_pos;
    int32_t* row_tok;
    float* row_w;
};
// rows: of all groups, at most; slots: routes per token that the kernel holds; decode: its routing (more state than prefill's)
bool ffn_f32_routes(bool decode, int64_t T, int64_t rows, int G, int N, int slots, int d, int I, int tile_rows, int sms);
cudaError_t launch_ffn_f32_routed(const FfnF32Params& p, const FfnF32Route& rt, int64_t rows, cudaStream_t s);
// Decode of few tokens, likewise (the group tables of rt are not written)
cudaError_t launch_ffn_f32_routed(const FfnF32Params& p, const DecodeRouteParams& rt, int64_t rows, cudaStream_t s);
cudaError_t launch_ffn_f32(const FfnF32Params& p, int64_t rows, int sms, cudaStream_t s);
cudaError_t launch_combine_f32(const float* out, const int32_t* inv_pos, const float* row_w, int64_t T, int Kr, int d,
                               int n_shared, const int32_t* shared0_dev, float* y, cudaStream_t s);

// ---------------------------------------------------------------- router scores, final sums of the bf16 path
// Router scores of more than one row tile of tokens, bf16 (router_gemm.cu)
struct RouterGemmParams {
    CUtensorMap tm_x;   // x [T][d], box 128 x 64
    CUtensorMap tm_wr;  // W_r [N][d], box router_npad(N) x 64 (rows past N are zero-filled)
    float* logits;      // [T][N]
    int T, N, nkb;      // nkb = d / 64
    int clear_status;   // the call's first kernel
    DeviceStatus* status;
    // set by the launcher
    int split, npad, part_ld, stages;
    uint32_t tmem_cols;
};
int router_npad(int N);
cudaError_t launch_router_gemm(RouterGemmParams p, int sms, cudaStream_t s);
cudaError_t launch_router_simt(const void* x, const void* wr, int dtype, int64_t T, int N, int d, float* out,
                               DeviceStatus* status, cudaStream_t s);
// y[i] = sum_j O[inv_pos[i*Kr+j]] (entries < 0 skipped) (+ O[shared0 + i] for the shared expert), fp32 sum in slot
// order, bf16 out. shared0 = T*Kr, or *shared0_dev when that is given (decode: known only on the device). A row may
// be stored as `parts` partial rows (decode's K split), part k at row k * part_rows + row: summed in that order.
cudaError_t launch_combine_rows(const __nv_bfloat16* O, const int32_t* inv_pos, int64_t T, int Kr, int d,
                                int n_shared, const int32_t* shared0_dev, int parts, int64_t part_rows,
                                __nv_bfloat16* y, cudaStream_t s);
constexpr int kMaxDecodeKsplit = 2;

// ---------------------------------------------------------------- calibration
struct CalibStatsParams {
    const float* out;    // expert outputs, one row of d floats per (token, slot)
    // row of (token i, slot a): inv_pos[i*Ke + a] if inv_pos is set, else i*tok_stride + a*slot_stride
    const int32_t* inv_pos;
    int64_t tok_stride, slot_stride;
    const int32_t* ids;  // [m][Ke]
    int64_t m;
    int Ke, d, N;
    double* A;  // [N][N]
    double* Bv;
    double* C;
    int32_t* cnt;  // [N][N]
    double* H;     // [N]
    int32_t* hc;   // [N]
    DeviceStatus* status;
};
cudaError_t launch_calib_stats(const CalibStatsParams& p, int sms, cudaStream_t s);
// Common-input mode with identity slots (slot a = expert a, inv_pos unused): same sums via per-token Gram
// products held in registers; nrm is scratch for m*Ke doubles
cudaError_t launch_calib_stats_common(const CalibStatsParams& p, double* nrm, int sms, cudaStream_t s);
cudaError_t launch_calib_finalize(const CalibStatsParams& p, const exfold_calib_opts& o, float* S, float* L,
                                  float* h, float* lnh, int32_t* n_obs, int32_t* unobserved, cudaStream_t s);
cudaError_t launch_iota_ids(int32_t* ids, int64_t m, int N, cudaStream_t s);
// Common-input calibration: every expert e owns rows [e*m, (e+1)*m) = all tokens in order
cudaError_t launch_calib_common_rows(int32_t* offsets, int32_t* work_start, int64_t m, int N, int tile_rows, cudaStream_t s);

// ---------------------------------------------------------------- tcgen05 grouped GEMMs (bf16)
// SM pairs, of n_clusters, that the CTA-pair passes keep when the odd-tile passes run beside them on the other
// 2 * (n_clusters - P) SMs. Every kernel of a call (both passes of both GEMMs) evaluates this on the device from the
// same group offsets, so they agree, and the split is the same for GEMM-1 and GEMM-2: `pairs` whole pairs of row tiles
// and `odd` odd tiles, each times the column tiles (nt) and k-blocks per item (nkb) of the two GEMMs. Side by side,
// a pair item takes a cluster ~0.73 of the time an odd item takes one SM (measured on the Mixtral shape: 25.9 against
// 35.7 us per 64-k-block item; the one-CTA kernel is the hungrier of the two for L2 bandwidth and slows down more
// beside the other). The choice minimises the longer of the two chains (GEMM-1 pass, then GEMM-2 pass), each pass
// counted in rounds of items. The odd-tile pass cannot get more than the odd_ctas CTAs it was launched with.
struct SideBySide {
    int nt1, nkb1, nt2, nkb2;  // column tiles and k-blocks per work item of GEMM-1 and GEMM-2
    int n_sm_pairs;            // SM pairs the pair passes are launched over
    int odd_ctas;              // CTAs the odd-tile passes are launched with (even); 0: the passes do not run side by side
    int shared_pairs1;         // whole row-tile pairs of the shared expert that GEMM-1's pair pass does not run (they
                               // ran beside the routing kernels, GroupedGemmParams::shared_split), else 0
};
__host__ __device__ inline int pair_pass_clusters(int pairs, int odd, const SideBySide& sb) {
    const int n = sb.n_sm_pairs;
    if (odd <= 0) return n;
    const int p_min = n - sb.odd_ctas / 2 > 0 ? n - sb.odd_ctas / 2 : 0;
    if (pairs <= 0) return p_min;
    int best = p_min > 1 ? p_min : 1;
    float best_t = 3.0e38f;
    for (int P = best; P < n; ++P) {
        const int Q = 2 * (n - P);
        const int pairs1 = pairs - sb.shared_pairs1;
        const float tp = 0.73f * (float)(((pairs1 * sb.nt1 + P - 1) / P) * sb.nkb1 + ((pairs * sb.nt2 + P - 1) / P) * sb.nkb2);
        const float to = (float)(((odd * sb.nt1 + Q - 1) / Q) * sb.nkb1 + ((odd * sb.nt2 + Q - 1) / Q) * sb.nkb2);
        const float t = tp > to ? tp : to;
        if (t < best_t) {
            best_t = t;
            best = P;
        }
    }
    return best;
}
struct GroupedGemmParams {
    CUtensorMap tm_a;    // GEMM-1: gathered rows Xs [R][d]; GEMM-2: H [Rtot][I]
    CUtensorMap tm_a2;   // GEMM-1: x [T][d] for the shared expert's rows
    CUtensorMap tm_b0;   // GEMM-1: W_gate as [(E*I)][d]; GEMM-2: W_down as [(E*d)][I]
    CUtensorMap tm_b1;   // GEMM-1: W_up; GEMM-2 on CTA pairs: W_down with 128-row boxes (each CTA stages half a tile)
    const int32_t* offsets;     // [G+1]
    const int32_t* work_start;  // [G+1] prefix of row tiles
    int G;                      // groups (N + n_shared)
    int n_routed;               // N
    int R;                      // routed rows (shared rows start here)
    int d, I;
    int n_ntiles;               // column tiles
    int n_cols;                 // decode: columns per tile, 256, 128 or 64 (tm_b0's box)
    int ksplit;                 // GEMM-2, decode: K parts per tile; part k of a row goes to plane k of the row buffer
    int a_rows;                 // decode: rows of the A (token) box, a multiple of 32 <= 128; prefill: 128
    const int32_t* grp_expert;  // [G] expert whose weights group g uses (null: g itself)
    const int32_t* n_groups_dev;  // device-side group count (null: G)
    // epilogues
    __nv_bfloat16* H;           // GEMM-1 out [Rtot][I]
    const int32_t* row_tok;     // GEMM-2
    const float* row_w;         // GEMM-2
    __nv_bfloat16* y;           // GEMM-2 bf16 target: row = token (store_rows == 0) or the sorted row itself
    int store_rows;             // 1: y is the per-route buffer O[row][d] that the combine kernel sums
    float* o32;                 // GEMM-2, calibration: unweighted fp32 outputs O32[row][d] (null: the epilogues above)
    int x_rows;                 // GEMM-1: rows of x; a group that reads x directly starts at row (row0 - R) % x_rows
    int shared_split;           // CTA-pair GEMM-1. 1: this launch runs only the whole row-tile pairs of the shared expert
                                //    (rows [R, R + x_rows) of expert n_routed, read from x: nothing the routing kernels
                                //    write is touched, so it runs beside them); 2: those pairs ran that way, skip them
    int odd_only;               // 1: only each group's last row tile, and only if its tile count is odd (the rest ran on CTA pairs)
    SideBySide sbs;             // odd_ctas > 0: the CTA-pair pass and the odd-tile pass run at the same time (two
                                //    streams); each keeps its share of the SM pairs (pair_pass_clusters) and the CTAs
                                //    beyond it leave at once
    DeviceStatus* status;
};
cudaError_t launch_grouped_gemm1(const GroupedGemmParams& p, int grid, cudaStream_t s);
cudaError_t launch_grouped_gemm2(const GroupedGemmParams& p, int grid, cudaStream_t s);
// Prefill on CTA pairs: every group's row tiles two at a time (a last odd tile is left to the kernels above with
// odd_only = 1). GEMM-2 needs tm_b1 = W_down with 128-row boxes. No grp_expert, no K split.
cudaError_t launch_grouped_gemm1_pair(const GroupedGemmParams& p, int grid, cudaStream_t s);
cudaError_t launch_grouped_gemm2_pair(const GroupedGemmParams& p, int grid, cudaStream_t s);
// The odd-tile pass beside them (p.odd_only = 1; prefill instantiation), launched two CTAs at a time so that the two
// grids share the GPU by whole SM pairs
cudaError_t launch_grouped_gemm1_odd(const GroupedGemmParams& p, int grid, cudaStream_t s);
cudaError_t launch_grouped_gemm2_odd(const GroupedGemmParams& p, int grid, cudaStream_t s);

// Whole 256-row tiles and ragged remainders of every group in one dynamically scheduled pass over CTA pairs (gemm_mixed.cu)
struct MixedGemmParams {
    GroupedGemmParams g;       // work_start counts kMixedTiles; tm_b1: W_down with 128-row boxes (GEMM-2)
    CUtensorMap tm_a_part[3];  // tm_a's matrix with boxes of 64, 32 and 16 rows
    CUtensorMap tm_x_part[3];  // tm_a2's (GEMM-1)
    CUtensorMap tm_b0_half;    // W_gate and W_up with 64-row boxes (GEMM-1)
    CUtensorMap tm_b1_half;
    int* queue;                // work counter, zero at the start
};
cudaError_t launch_grouped_gemm1_mixed(const MixedGemmParams& p, int grid, cudaStream_t s);
cudaError_t launch_grouped_gemm2_mixed(const MixedGemmParams& p, int grid, cudaStream_t s);

}  // namespace exfold
