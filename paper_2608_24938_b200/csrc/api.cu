// C ABI of the folded-MoE library: argument validation, workspace planning, TMA tensor maps
// and the launch sequences of the three calls. No device memory is allocated here.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "ptx.cuh"


namespace exfold {

static std::atomic<int64_t> g_launches{0};
void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
static thread_local bool t_pdl = false;
static thread_local bool t_keep_status = false;  // set while a host-buffer call runs its second and later chunks
void set_pdl(bool on) { t_pdl = on; }
bool pdl_enabled() { return t_pdl; }

namespace {

// ------------------------------------------------------------------ optional per-kernel event timing
struct Profiler {
    bool on = false;
    cudaEvent_t beg[EXFOLD_PROFILE_SLOTS];
    cudaEvent_t end[EXFOLD_PROFILE_SLOTS];
    bool used[EXFOLD_PROFILE_SLOTS];
} g_prof;

struct ProfScope {  // records an event pair around one launch when profiling is enabled
    int slot;
    cudaStream_t s;
    ProfScope(int slot_, cudaStream_t s_) : slot(slot_), s(s_) {
        if (g_prof.on) cudaEventRecord(g_prof.beg[slot], s);
    }
    ~ProfScope() {
        if (g_prof.on) {
            cudaEventRecord(g_prof.end[slot], s);
            g_prof.used[slot] = true;
        }
    }
};
void prof_reset() {
    for (int i = 0; i < EXFOLD_PROFILE_SLOTS; ++i) g_prof.used[i] = false;
}

// ------------------------------------------------------------------ workspace plan
struct Plan {
    size_t status, ids, w, omit_src, omit_tgt, block_hist, sb_hist, offsets, work_start, totals, perm, row_tok, row_w,
        row_grp, pool_ids, pool_size, pool_mask, target, scale, grp_expert, grp_off, n_groups, calib, big,
        xs, H, out, grp_tiles, obuf, inv_pos, calib_nrm, w64, total;
};

bool valid_layer(const exfold_layer* l) {
    if (!l) return false;
    if (l->n_experts < 2 || l->n_experts > kMaxExperts) return false;
    if (l->n_shared < 0 || l->n_shared > 1) return false;
    if (l->top_k < 1 || l->top_k > kMaxTopK || l->top_k > l->n_experts) return false;
    if (l->hidden < 1 || l->inter < 1) return false;
    if (l->dtype != EXFOLD_F32 && l->dtype != EXFOLD_BF16) return false;
    if (l->dtype == EXFOLD_BF16 && (l->hidden % 64 != 0 || l->inter % 64 != 0)) return false;
    if (l->dtype == EXFOLD_F32 && (l->hidden % 4 != 0)) return false;
    return true;
}

Plan make_plan(const exfold_layer& l, int64_t Tm, int Kr) {
    Plan p{};
    const int N = l.n_experts, G = N + l.n_shared;
    const size_t Rm = (size_t)Tm * Kr, Rtot = Rm + (size_t)Tm * l.n_shared;
    const size_t nblk = (size_t)(Tm + kRouteTokensPerBlock - 1) / kRouteTokensPerBlock;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    p.status = take(sizeof(DeviceStatus));
    p.ids = take(Rm * 4);
    p.w = take(Rm * 4);
    p.omit_src = take((size_t)Tm * l.top_k * 4);
    p.omit_tgt = take((size_t)Tm * l.top_k * 4);
    p.block_hist = take(nblk * N * 4);
    p.sb_hist = take((nblk + kRouteSuperBlock - 1) / kRouteSuperBlock * N * 4);
    p.offsets = take((G + 2) * 4);
    p.work_start = take((G + 2) * 4);
    p.totals = take(16);
    p.perm = take(Rm * 4);
    p.inv_pos = take(Rm * 4);
    p.row_tok = take(Rtot * 4);
    p.row_w = take(Rtot * 4);
    p.row_grp = take(Rtot * 4);  // small batches: group of each row
    p.w64 = take((size_t)std::min<int64_t>(Tm, kMaxDecodeBatch) * l.top_k * 8);  // decode: routed weights in double
    p.pool_ids = take((size_t)N * 4);
    p.pool_size = take(16);
    p.pool_mask = take(32);
    p.target = take((size_t)N * 4);
    p.scale = take((size_t)N * 4);
    p.grp_expert = take((G + 2) * 4);
    p.grp_off = take((G + 2) * 4);
    p.grp_tiles = take((G + 2) * 4);
    p.n_groups = take(16);
    p.calib = take((size_t)N * N * (3 * 8 + 4) + (size_t)N * (8 + 4) + 256);
    p.calib_nrm = take(Rm * 8);  // calibration, common-input mode: squared output norms per (token, expert)
    // large buffers: the bf16 pipeline (sorted rows, H, fp32 accumulator) and the fp32 path's
    // per-route outputs are never live at the same time and share one region
    p.big = off;
    size_t a = 0;
    if (l.dtype == EXFOLD_BF16) {
        // xs and obuf are adjacent: calibration reuses the two together (>= Rtot*d*4 bytes) for the
        // fp32 per-row expert outputs once GEMM-1 has consumed the gathered rows
        p.xs = p.big;
        a = align_up(Rtot * (size_t)l.hidden * 2, 1024);
        p.obuf = p.big + a;  // per-row bf16 outputs O [Rtot][d] (decode: one plane per K part)
        a += align_up(std::max((size_t)Tm * l.hidden * 4, Rtot * (size_t)l.hidden * 2), 1024);
        p.H = p.big + a;
        a += align_up(Rtot * (size_t)l.inter * 2, 1024);
    }
    p.out = p.big;
    size_t b = align_up(Rtot * (size_t)l.hidden * 4, 1024);
    p.total = p.big + (a > b ? a : b);
    return p;
}

template <typename T>
T* at(void* ws, size_t off) {
    return reinterpret_cast<T*>(reinterpret_cast<char*>(ws) + off);
}

// ------------------------------------------------------------------ tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

constexpr int kMaxHostChunks = 4;  // host-buffer prefill: chunks of >= 2048 tokens in flight

// bf16 matrix [rows][cols] row-major; box = box_rows x kGemmBK columns, 128-byte swizzle (a box row)
bool make_tmap(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {(cuuint32_t)kGemmBK, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Host-side CUDA objects the library keeps per (host thread, device), created on first use and kept until
// exfold_thread_release() or the end of the process:
//   side stream + fork / join / mid events: the odd-tile passes of a prefill call run beside the CTA-pair passes;
//   in / out streams + events: the chunked host-buffer prefill copies the next chunk in and the previous one out
//   while the caller's stream computes.
// Nothing else survives a call. Two caller streams used from one host thread share these objects, so the parts of
// their calls that run on them are ordered one after the other (results are unaffected).
constexpr int kMaxDevices = 64;
struct ThreadDeviceState {
    cudaStream_t side = nullptr, in = nullptr, out = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr, mid = nullptr;
    cudaEvent_t start = nullptr, done = nullptr, copied[kMaxHostChunks] = {}, computed[kMaxHostChunks] = {};
    bool side_ok = false, host_ok = false;
    int* result = nullptr;  // pinned host words that a calibration's last kernels write their counts to
    int sms = 0;
    void release() {
        auto ev = [](cudaEvent_t& e) { if (e) cudaEventDestroy(e); e = nullptr; };
        auto st = [](cudaStream_t& s) { if (s) cudaStreamDestroy(s); s = nullptr; };
        ev(fork); ev(join); ev(mid); ev(start); ev(done);
        for (int c = 0; c < kMaxHostChunks; ++c) { ev(copied[c]); ev(computed[c]); }
        st(side); st(in); st(out);
        if (result) cudaFreeHost(result);
        result = nullptr;
        side_ok = host_ok = false;
    }
};
thread_local ThreadDeviceState t_state[kMaxDevices];

ThreadDeviceState* thread_state() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    return &t_state[dev];
}
}  // namespace

cudaError_t ensure_smem_bytes(const void* kernel, size_t bytes) {
    struct Entry {
        const void* kernel;
        int dev;
        size_t limit;
    };
    static thread_local Entry cache[256] = {};  // by kernel address; a collision only asks the driver again
    int dev = 0, optin = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    Entry& e = cache[(reinterpret_cast<uintptr_t>(kernel) >> 4) & 255];
    if (e.kernel != kernel || e.dev != dev) {
        // every thread sets the same value, the most a block may have, so none can lower what another relies on
        cudaFuncAttributes fa;
        if ((err = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return err;
        if ((err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return err;
        const size_t limit = (size_t)optin - fa.sharedSizeBytes;
        if ((err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit)) != cudaSuccess) return err;
        e = Entry{kernel, dev, limit};
    }
    return bytes <= e.limit ? cudaSuccess : cudaErrorInvalidValue;
}

namespace {
bool new_event(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess; }
// second stream (and fork / join events) for the odd-tile passes of a prefill call
ThreadDeviceState* side_stream() {
    ThreadDeviceState* h = thread_state();
    if (h && !h->side_ok) {
        // highest priority: what runs here beside a bandwidth-bound kernel of the caller's stream (the shared
        // expert's GEMM-1 beside the scatter kernel) gets its SMs first and the other kernel fills the rest
        int lo = 0, hi = 0;
        if (cudaDeviceGetStreamPriorityRange(&lo, &hi) != cudaSuccess) hi = 0;
        h->side_ok = cudaStreamCreateWithPriority(&h->side, cudaStreamNonBlocking, hi) == cudaSuccess &&
                     new_event(&h->fork) && new_event(&h->join) && new_event(&h->mid);
    }
    return h && h->side_ok ? h : nullptr;
}
// copy-in / copy-out streams and events of the chunked host-buffer prefill
ThreadDeviceState* host_helpers() {
    ThreadDeviceState* h = thread_state();
    if (h && !h->host_ok) {
        bool ok = cudaStreamCreateWithFlags(&h->in, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&h->out, cudaStreamNonBlocking) == cudaSuccess && new_event(&h->start) &&
                  new_event(&h->done);
        for (int c = 0; ok && c < kMaxHostChunks; ++c) ok = new_event(&h->copied[c]) && new_event(&h->computed[c]);
        h->host_ok = ok;
    }
    return h && h->host_ok ? h : nullptr;
}
// One pinned word per calibration job: read after the stream has drained, without a copy
int* result_words() {
    ThreadDeviceState* h = thread_state();
    if (h && !h->result && cudaHostAlloc(reinterpret_cast<void**>(&h->result), EXFOLD_MAX_CALIB_JOBS * sizeof(int), cudaHostAllocDefault) != cudaSuccess)
        h->result = nullptr;
    return h ? h->result : nullptr;
}
// Once the side stream has been forked off the caller's stream it is joined again on every way out of the call
// (also the error returns): later work on the caller's stream, or the end of a stream capture, must not overtake it.
struct SideJoin {
    ThreadDeviceState* side;
    cudaStream_t s;
    bool armed = true;
    cudaError_t join() {
        armed = false;
        cudaError_t e = cudaEventRecord(side->join, side->side);
        return e != cudaSuccess ? e : cudaStreamWaitEvent(s, side->join, 0);
    }
    ~SideJoin() {
        if (armed) join();
    }
};

int sm_count() {  // of the current device
    ThreadDeviceState* h = thread_state();
    int n = h ? h->sms : 0;
    if (n <= 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
        if (h) h->sms = n;
    }
    return n;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

#define EXFOLD_CUDA(call)                                 \
    do {                                                  \
        cudaError_t e__ = (call);                         \
        if (e__ != cudaSuccess) return EXFOLD_ERR_CUDA;   \
    } while (0)

// Row tiles of a grouped GEMM over `rows` sorted rows of G groups: on average half a tile per group is a ragged last one
int64_t expected_tiles(int64_t rows, int G) { return rows / kTileM + G / 2; }

// For the calls that use_mixed (below) leaves to row tiles of 128 rows, and with a shared expert for its early pairs:
// whether the two GEMMs run their whole pairs of row tiles on CTA pairs (gemm_pair.cu: a third less operand traffic per
// SM, a deeper ring) with the groups' odd last tiles beside them, or every tile on the one-CTA kernel. The pairs pay once
// a group owns a tile or more on average (before, most tiles are odd ones, and the weights of a group with three tiles
// are read by both passes) and the GEMMs are long enough for the second stream's fork and join: from ~400 k-blocks per
// SM. Measured, pair / one-CTA time of the call: Qwen3 shape (K' = 4) 1024 tokens 206 / 168 us, 4096 328 / 300, 6144
// 408 / 409, 8192 467 / 502; GLM shape 2048 tokens 1025 / 899 us, 4096 1229 / 1289; Mixtral shape (K' = 1) 512 tokens
// 511 / 496 us, 1024 630 / 695, 4096 1277 / 1852; 64 experts of 1024 x 512, 8192 tokens 160 / 157 us. With few tiles in
// all, the sizes of the last tiles decide (Mixtral shape, 17 tiles: 1179 / 1078 us): one-CTA below 24.
bool use_pairs(int64_t rows, int G, int d, int I) {
    const int64_t tiles = rows / kTileM;
    const int64_t kblocks = (int64_t)((I + 127) / 128) * (d / kGemmBK) + (int64_t)((d + 255) / 256) * (I / kGemmBK);
    return tiles >= G && expected_tiles(rows, G) >= 24 && tiles * kblocks >= (int64_t)400 * sm_count();
}

// The two grouped GEMMs of bf16 expert rows (prefill, calibration): g = GEMM-1, g2 = GEMM-2 on `rows` sorted rows.
// Without `pairs` every row tile runs on the one-CTA kernel. With it, whole pairs of row tiles run on CTA pairs on the
// caller's stream and the groups' odd last tiles beside them on a second stream.
int enqueue_expert_gemms(GroupedGemmParams& g, GroupedGemmParams& g2, int64_t rows, bool pairs, int shared_pairs,
                         cudaStream_t s) {
    const int G = g.G, nt1 = g.n_ntiles, nt2 = g2.n_ntiles, d = g.d, I = g.I;
    if (!pairs) {
        const int64_t max_tiles = rows / kTileM + G;
        { ProfScope ps(3, s); EXFOLD_CUDA(launch_grouped_gemm1(g, (int)std::min<int64_t>(sm_count(), max_tiles * nt1), s)); }
        { ProfScope ps(4, s); EXFOLD_CUDA(launch_grouped_gemm2(g2, (int)std::min<int64_t>(sm_count(), max_tiles * nt2), s)); }
        return EXFOLD_OK;
    }
    // Both passes are launched over all SMs, the pair pass on the caller's stream and the odd-tile pass on a
    // second one; on the device each keeps its share of the SM pairs (pair_pass_clusters of the actual tile
    // counts) and its other CTAs leave at once, so the two grids settle side by side whatever the routing.
    // Rows of whole tile pairs and rows of odd last tiles never meet before the combine step, so each pass
    // of GEMM-2 follows the same pass of GEMM-1 on its own stream: caller's stream: GEMM-1 pairs -> GEMM-2
    // pairs; side stream: GEMM-1 odd tiles -> GEMM-2 odd tiles; joined before the combine kernel (or the
    // end of the call). With per-kernel timing on, and in calibration, whose fp32 outputs overwrite the rows that
    // GEMM-1 reads, the streams also join between the two GEMMs.
    const bool join_mid = g_prof.on || g2.o32 != nullptr;
    const int sms = sm_count() & ~1;
    ThreadDeviceState* sidep = side_stream();
    if (!sidep) return EXFOLD_ERR_CUDA;
    ThreadDeviceState& side = *sidep;
    GroupedGemmParams go1 = g, go2 = g2;
    go1.odd_only = go2.odd_only = 1;
    // The odd-tile pass is launched with about twice the CTAs its expected share of the work needs (its share
    // is decided on the device, where the tile counts are known): CTAs without work leave at once, but every
    // one of them has to pass through one of the pass's few SMs first.
    const double odd_est = std::max<double>(1.0, G / 2.0),
                 pair_est = std::max<double>(1.0, (expected_tiles(rows, G) - G / 2.0) / 2.0);
    const double q_est = sms * odd_est / (odd_est + 2 * 0.73 * pair_est);
    const int odd_grid = std::min(sms, 2 * (int)std::ceil(q_est) + 8) & ~1;
    const SideBySide sbs{nt1, d / kGemmBK, nt2, I / kGemmBK, sms / 2, odd_grid, shared_pairs};
    g.sbs = g2.sbs = go1.sbs = go2.sbs = sbs;
    SideJoin joiner{sidep, s};
    EXFOLD_CUDA(cudaEventRecord(side.fork, s));
    EXFOLD_CUDA(cudaStreamWaitEvent(side.side, side.fork, 0));
    {
        ProfScope ps(3, s);
        { ProfScope pp(12, s); EXFOLD_CUDA(launch_grouped_gemm1_pair(g, sms, s)); }
        EXFOLD_CUDA(launch_grouped_gemm1_odd(go1, odd_grid, side.side));
        if (join_mid) {
            EXFOLD_CUDA(cudaEventRecord(side.mid, side.side));
            EXFOLD_CUDA(cudaEventRecord(side.fork, s));
            EXFOLD_CUDA(cudaStreamWaitEvent(s, side.mid, 0));
            EXFOLD_CUDA(cudaStreamWaitEvent(side.side, side.fork, 0));
        }
    }
    ProfScope ps(4, s);
    { ProfScope pp(13, s); EXFOLD_CUDA(launch_grouped_gemm2_pair(g2, sms, s)); }
    EXFOLD_CUDA(launch_grouped_gemm2_odd(go2, odd_grid, side.side));
    EXFOLD_CUDA(joiner.join());
    return EXFOLD_OK;
}

// The same GEMMs on the mixed kernel (gemm_mixed.cu): one launch each on the caller's stream. x, w_gate, w_up: the matrices
// behind g.tm_a2, tm_b0 and tm_b1; `experts` of them.
int enqueue_mixed_gemms(const GroupedGemmParams& g, const GroupedGemmParams& g2, const void* xs, int64_t R, int64_t rows,
                        const void* x, const void* w_gate, const void* w_up, int experts, cudaStream_t s) {
    MixedGemmParams m1{}, m2{};
    m1.g = g;
    m2.g = g2;
    const uint64_t wrows = (uint64_t)experts * g.I;
    if (!make_tmap(&m1.tm_b0_half, w_gate, wrows, g.d, 64) || !make_tmap(&m1.tm_b1_half, w_up, wrows, g.d, 64)) return EXFOLD_ERR_CUDA;
    for (int i = 0; i < 3; ++i)
        if (!make_tmap(&m1.tm_a_part[i], xs, (uint64_t)R, g.d, 64 >> i) || !make_tmap(&m1.tm_x_part[i], x, (uint64_t)g.x_rows, g.d, 64 >> i) ||
            !make_tmap(&m2.tm_a_part[i], g.H, (uint64_t)rows, g.I, 64 >> i))
            return EXFOLD_ERR_CUDA;
    m1.queue = &g.status->queue[0];
    m2.queue = &g.status->queue[1];
    { ProfScope ps(3, s); EXFOLD_CUDA(launch_grouped_gemm1_mixed(m1, sm_count(), s)); }
    { ProfScope ps(4, s); EXFOLD_CUDA(launch_grouped_gemm2_mixed(m2, sm_count(), s)); }
    return EXFOLD_OK;
}

// Whether they do. The mixed kernel computes and loads what a group's rows need, where row tiles of 128 rows waste half a tile
// per group, and reads a weight tile once; but it has half as many workers (CTA pairs), and an item costs a pair more to hand over.
// So it wants a few rounds of items, and the more rows per group the shorter the items are (k-blocks of an item, the mean over both
// GEMMs' work: a hand-over against that). Whole prefill call on row tiles / mixed, even and skewed scores, three layers in turn:
//   12 k-blocks and more: 24 rows per group, any number from 48 k-blocks of GEMM-1 on. GLM shape (K' = 4) 59 tokens 552 / 518 us, 192 /
//   187, 400 746 / 705, 349 / 336, 1200 802 / 757, 547 / 503; Qwen3 shape (K' = 6) 777 tokens 234 / 228, 185 / 180, 2200 285 / 276, 284 /
//   268; Mixtral shape (K' = 2) 200 tokens 484 / 464, 489 / 476; 160 experts of 1024 x 1024 (K' = 4) 1300 tokens 216 / 205, 127 / 126,
//   4000 265 / 248, 225 / 212; 128 of 768 x 1536 (K' = 4) 1500 tokens 192 / 190, 140 / 139; the line itself: 64 + 1 of 2048 x 1408 (K' = 2)
//   800 tokens 218 / 216, 151 / 154, 96 + 1 of 1536 x 768 (K' = 3) 1500 tokens 165 / 169, 135 / 134.
//   9: 144 rows. 160 of 1024 x 320 (K' = 4) 1800 tokens (45 rows) 102 / 105, 78 / 87, 8000 (200) 183 / 176, 173 / 165.
//   8: 320 rows. 139 + 1 of 576 x 448 (K' = 3) 2102 tokens (60) 85 / 97, 71 / 79, 5000 (143) 115 / 125, 107 / 113, (K' = 2) 14000 (300)
//   181 / 181, 169 / 166; 256 of 512 x 512 (K' = 3) 12600 tokens (148) 192 / 198, 162 / 169.
//   Fewer: never. 200 of 320 x 1280 (K' = 4) 10000 tokens (200) 244 / 257, 234 / 231; 114 + 1 of 192 x 448 (K' = 5) 13328 tokens (695) skewed
//   161 / 174; 64 of 128 x 1024 (K' = 3) 9000 tokens (422) 94 / 104, 94 / 105.
// Where use_pairs would run pairs of row tiles beside odd ones, those / mixed: GLM shape 16384 tokens 2576 / 2423, Mixtral shape 2000
// tokens 748 / 689, 4096 1271 / 1187 (8 experts of it, skewed, 3376 tokens 1123 / 1087), Qwen3 shape 8192 tokens 400 / 381; under the power
// cap alike (2939 / 2757, 1455 / 1358). With eight row tiles per group and more there is little left to waste: 128 of 2048 x 768 (K' = 8)
// 16384 tokens 1396 / 1375, 1408 / 1402, 64 of 2048 x 1408 (K' = 6) 12000 tokens 1245 / 1258, 1255 / 1250, GLM shape (K' = 8) 16000 tokens 4904 /
// 4841, 4782 / 4873. Few items: 64 of 1024 x 512 (K' = 4) 768 tokens 64 / 71; 11 of 2688 x 512 (K' = 3) 58 / 65.
bool use_mixed(int64_t rows, int G, int d, int I) {
    const int64_t items = (int64_t)G * ((I + 127) / 128) * std::max<int64_t>(1, rows / (256 * (int64_t)G));
    if (rows / kTileM >= (int64_t)8 * G || items < (int64_t)3 * sm_count()) return false;
    const int64_t kblocks = (int64_t)3 * d * I / ((2 * (int64_t)I + d) * kGemmBK);  // GEMM-1 is two thirds of the work
    if (kblocks >= 12) return d >= 48 * kGemmBK || rows >= (int64_t)24 * G;
    return kblocks >= 8 && rows >= (int64_t)(kblocks >= 9 ? 144 : 320) * G;
}

struct PdlScope {  // programmatic dependent launch for the launches of this scope
    explicit PdlScope(bool on) { set_pdl(on); }
    ~PdlScope() { set_pdl(false); }
};

FfnF32Params f32_params(const void* x, const void* wg, const void* wu, const void* wd, int d, int I, int G, int tile_rows) {
    FfnF32Params p{};
    p.x = reinterpret_cast<const float*>(x); p.wg = reinterpret_cast<const float*>(wg);
    p.wu = reinterpret_cast<const float*>(wu); p.wd = reinterpret_cast<const float*>(wd);
    p.d = d; p.I = I; p.G = G; p.tile_rows = tile_rows; p.x_rows = 1;
    return p;
}

int copy_meta(void* dst, const void* src, size_t bytes, cudaStream_t s) {
    if (dst == nullptr || bytes == 0) return EXFOLD_OK;
    EXFOLD_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, s));
    return EXFOLD_OK;
}

int check_common(const exfold_layer* layer, const void* x, const float* logits, int64_t T, const void* wg,
                 const void* wu, const void* wd, const exfold_tables* t, void* y, void* ws) {
    if (!valid_layer(layer)) return EXFOLD_ERR_INVALID_ARG;
    if (!x || !logits || !wg || !wu || !wd || !y || !ws) return EXFOLD_ERR_INVALID_ARG;
    if (!t || !t->S || !t->L || !t->h || !t->lnh) return EXFOLD_ERR_INVALID_ARG;
    if (T < 1 || T > (int64_t)1 << 24) return EXFOLD_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(y) || !aligned16(wg) || !aligned16(wu) || !aligned16(wd) ||
        (reinterpret_cast<uintptr_t>(ws) & 255) != 0)
        return EXFOLD_ERR_INVALID_ARG;
    return EXFOLD_OK;
}

}  // namespace

// Synchronises the stream, decodes and clears the status record at `rec` (device memory)
int read_status_record(void* rec, cudaStream_t s) {
    if (cudaStreamSynchronize(s) != cudaSuccess) return EXFOLD_ERR_CUDA;
    int code = 0;
    if (cudaMemcpy(&code, rec, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return EXFOLD_ERR_CUDA;
    if (cudaMemset(rec, 0, sizeof(DeviceStatus)) != cudaSuccess) return EXFOLD_ERR_CUDA;
    if (code == 0) return EXFOLD_OK;
    return code == EXFOLD_ERR_DEVICE_TIMEOUT ? EXFOLD_ERR_DEVICE_TIMEOUT : EXFOLD_ERR_CUDA;
}
}  // namespace exfold

using namespace exfold;

extern "C" {

size_t exfold_workspace_bytes(const exfold_layer* layer, int64_t max_tokens, int32_t routes_per_token) {
    if (!valid_layer(layer) || max_tokens < 1 || routes_per_token < 1 || routes_per_token > kMaxExperts) return 0;
    return make_plan(*layer, max_tokens, routes_per_token).total;
}

size_t exfold_host_staging_bytes(const exfold_layer* layer, int64_t max_tokens) {
    if (!valid_layer(layer) || max_tokens < 1) return 0;
    const size_t el = layer->dtype == EXFOLD_BF16 ? 2 : 4;
    return 2 * align_up((size_t)max_tokens * layer->hidden * el, 256) +
           align_up((size_t)max_tokens * layer->n_experts * 4, 256);
}

int64_t exfold_launch_count(void) { return g_launches.load(); }

int exfold_profile_enable(int enable) {
    if (enable && !g_prof.on) {
        for (int i = 0; i < EXFOLD_PROFILE_SLOTS; ++i) {
            if (cudaEventCreate(&g_prof.beg[i]) != cudaSuccess) return EXFOLD_ERR_CUDA;
            if (cudaEventCreate(&g_prof.end[i]) != cudaSuccess) return EXFOLD_ERR_CUDA;
        }
        prof_reset();
        g_prof.on = true;
    } else if (!enable && g_prof.on) {
        g_prof.on = false;
        for (int i = 0; i < EXFOLD_PROFILE_SLOTS; ++i) {
            cudaEventDestroy(g_prof.beg[i]);
            cudaEventDestroy(g_prof.end[i]);
        }
    }
    return EXFOLD_OK;
}

int exfold_profile_read(float* ms, int32_t n_slots) {
    if (!ms || n_slots < 0) return EXFOLD_ERR_INVALID_ARG;
    for (int i = 0; i < n_slots; ++i) {
        ms[i] = -1.0f;
        if (!g_prof.on || i >= EXFOLD_PROFILE_SLOTS || !g_prof.used[i]) continue;
        if (cudaEventSynchronize(g_prof.end[i]) != cudaSuccess) return EXFOLD_ERR_CUDA;
        if (cudaEventElapsedTime(&ms[i], g_prof.beg[i], g_prof.end[i]) != cudaSuccess) return EXFOLD_ERR_CUDA;
    }
    return EXFOLD_OK;
}

const char* exfold_status_string(int status) {
    switch (status) {
        case EXFOLD_OK: return "ok";
        case EXFOLD_ERR_INVALID_ARG: return "invalid argument";
        case EXFOLD_ERR_UNSUPPORTED: return "unsupported configuration";
        case EXFOLD_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case EXFOLD_ERR_CUDA: return "CUDA error";
        case EXFOLD_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait ran out";
        case EXFOLD_ERR_EXCEEDS_STATIC_SCRATCH:
            return "layer and batch need more scratch than the built-in EXFOLD_STATIC_SCRATCH_BYTES array holds";
        case EXFOLD_WARN_UNOBSERVED_EXPERT: return "warning: an expert was never observed during calibration";
        default: return "unknown status";
    }
}

int exfold_device_status(void* ws, void* cuda_stream) {
    if (!ws) return EXFOLD_ERR_INVALID_ARG;
    return read_status_record(ws, reinterpret_cast<cudaStream_t>(cuda_stream));
}

int exfold_thread_release(void) {
    ThreadDeviceState* h = thread_state();
    if (!h) return EXFOLD_ERR_CUDA;
    h->release();
    return EXFOLD_OK;
}

int exfold_moe_prefill(const exfold_layer* layer, const void* x, const float* logits, int64_t T, const void* w_gate,
                       const void* w_up, const void* w_down, const exfold_tables* tables, int32_t k_pre, void* y,
                       const exfold_prefill_meta* meta, void* ws, size_t ws_bytes, void* cuda_stream) {
    return exfold_moe_prefill_ex(layer, x, logits, T, w_gate, w_up, w_down, tables, k_pre, nullptr, y, meta, ws,
                                 ws_bytes, cuda_stream);
}

int exfold_moe_prefill_ex(const exfold_layer* layer, const void* x, const float* logits, int64_t T,
                          const void* w_gate, const void* w_up, const void* w_down, const exfold_tables* tables,
                          int32_t k_pre, const exfold_fold_opts* opts, void* y, const exfold_prefill_meta* meta,
                          void* ws, size_t ws_bytes, void* cuda_stream) {
    int rc = check_common(layer, x, logits, T, w_gate, w_up, w_down, tables, y, ws);
    if (rc != EXFOLD_OK) return rc;
    const exfold_layer& l = *layer;
    if (k_pre < 1 || k_pre > l.top_k) return EXFOLD_ERR_INVALID_ARG;
    const int N = l.n_experts, K = l.top_k, Kp = k_pre, d = l.hidden, I = l.inter, G = N + l.n_shared;
    const int64_t R = T * Kp, Rtot = R + T * l.n_shared;
    // A few tokens: the two kernels of a small decode batch on the routes (whatever gemm_path says: same results for all)
    const bool small = l.dtype == EXFOLD_BF16 && T <= kSmallDecodeBatch && decode_small_fits((int)T, Kp, d, w_gate, w_up, w_down);
    if (Rtot > (int64_t)1 << 30) return EXFOLD_ERR_UNSUPPORTED;
    const Plan pl = make_plan(l, T, Kp);
    if (ws_bytes < pl.total) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    const bool bf16 = l.dtype == EXFOLD_BF16;
    const bool direct = Kp == 1 && l.n_shared == 0;  // every token is written exactly once

    CUtensorMap tm_xs, tm_x, tm_wg, tm_wu, tm_h, tm_wd, tm_wd_half;
    const int mode = opts == nullptr || opts->gemm_path < 0 || opts->gemm_path > 3 ? 0 : opts->gemm_path;
    const bool pairs = bf16 && !small && (mode == 2 ? Rtot >= 2 * kTileM : mode != 1 && use_pairs(Rtot, G, d, I));
    const bool mixed = bf16 && !small && (mode == 3 || (mode == 0 && use_mixed(Rtot, G, d, I)));
    const int sms = sm_count() & ~1;
    if (bf16 && !small) {
        const uint64_t E = (uint64_t)G;
        bool ok = make_tmap(&tm_xs, at<char>(ws, pl.xs), (uint64_t)R, d, 128) && make_tmap(&tm_x, x, (uint64_t)T, d, 128) &&
                  make_tmap(&tm_wg, w_gate, E * I, d, 128) && make_tmap(&tm_wu, w_up, E * I, d, 128) &&
                  make_tmap(&tm_h, at<char>(ws, pl.H), (uint64_t)Rtot, I, 128) &&
                  make_tmap(&tm_wd, w_down, E * d, I, 256) && make_tmap(&tm_wd_half, w_down, E * d, I, 128);
        if (!ok) return EXFOLD_ERR_CUDA;
    }

    prof_reset();
    // Calls without the CTA-pair passes (fp32 layers, shorter bf16 prompts) are a chain of short kernels on one stream:
    // programmatic dependent launch hides their launches and set-up (Qwen3 shape 20 tokens 66.8 -> 56.5 us, 777 tokens 279
    // -> 270; Mixtral shape 200 tokens 532 -> 514). So are the mixed kernel's calls (0.5-1 % of the call). The CTA-pair passes
    // beside odd-tile passes launch plainly: early-resident successors compete with the running kernels (19-32 us slower).
    PdlScope pdl_scope(!pairs || mixed);

    PrefillRouteParams rp{};
    rp.logits = logits; rp.S = tables->S; rp.L = tables->L; rp.lnh = tables->lnh;
    rp.T = T; rp.N = N; rp.K = K; rp.Kp = Kp;
    rp.loss_thr = opts ? opts->loss_threshold : INFINITY;
    rp.rescale = opts ? opts->rescale : 0;
    rp.confidence = opts ? opts->confidence_split : 0;
    rp.ids = at<int32_t>(ws, pl.ids); rp.w = at<float>(ws, pl.w);
    rp.omit_src = at<int32_t>(ws, pl.omit_src); rp.omit_tgt = at<int32_t>(ws, pl.omit_tgt);
    rp.block_hist = at<int32_t>(ws, pl.block_hist);
    rp.sb_hist = at<int32_t>(ws, pl.sb_hist);
    // the first kernel of the call clears the status record (not for the later chunks of a chunked host call)
    rp.status = t_keep_status ? nullptr : at<DeviceStatus>(ws, pl.status);
    rp.queue = mixed ? at<DeviceStatus>(ws, pl.status)->queue : nullptr;
    // few tokens of an fp32 layer: its FFN kernel routes them itself
    const int tile_rows = mixed ? kMixedTiles : bf16 ? kTileM : ffn_f32_tile_rows(Rtot, G, d, I, sm_count());
    const bool routed = !bf16 && ffn_f32_routes(false, T, Rtot, G, N, Kp, d, I, tile_rows, sm_count());
    // (so do the small-batch kernels, unless the caller asks for the metadata, of which the scatter kernel writes a part)
    const bool small_routed = small && meta == nullptr;
    if (!routed && !small_routed) { ProfScope ps(0, s); EXFOLD_CUDA(launch_prefill_route(rp, s)); }

    // The shared expert's gate/up projection needs nothing the routing kernels produce (its rows are x itself, its
    // rows of H lie behind the routed ones): its whole row-tile pairs run on the second stream beside the scatter
    // kernel, which moves bytes while the tensor pipes would idle. (After the routing kernel, which clears the status
    // record every kernel's waits look at.) The CTA-pair GEMM-1 that follows the scatter kernel skips those pairs.
    // Not with per-kernel timing on: the timed kernels are then the plain sequence, GEMM-1 with all its pairs.
    const int shared_pairs = pairs && l.n_shared && !g_prof.on ? (int)(((T + kTileM - 1) / kTileM) / 2) : 0;
    ThreadDeviceState* early_side = nullptr;
    if (shared_pairs > 0) {
        early_side = side_stream();
        if (!early_side) return EXFOLD_ERR_CUDA;
        GroupedGemmParams gs{};
        gs.tm_a = tm_xs; gs.tm_a2 = tm_x; gs.tm_b0 = tm_wg; gs.tm_b1 = tm_wu; gs.x_rows = (int)T;
        gs.G = G; gs.n_routed = N; gs.R = (int)R; gs.d = d; gs.I = I; gs.n_ntiles = (I + 127) / 128; gs.ksplit = 1;
        gs.a_rows = kTileM; gs.H = at<__nv_bfloat16>(ws, pl.H); gs.status = at<DeviceStatus>(ws, pl.status);
        gs.shared_split = 1;
        gs.sbs = SideBySide{(I + 127) / 128, d / kGemmBK, (d + 255) / 256, I / kGemmBK, sms / 2, 0, 0};
        EXFOLD_CUDA(cudaEventRecord(early_side->fork, s));
        EXFOLD_CUDA(cudaStreamWaitEvent(early_side->side, early_side->fork, 0));
        EXFOLD_CUDA(launch_grouped_gemm1_pair(gs, sms, early_side->side));
        EXFOLD_CUDA(cudaEventRecord(early_side->mid, early_side->side));
    }
    SideJoin early_join{early_side, s};  // joins the second stream on the error returns before the passes below take over
    early_join.armed = early_side != nullptr;

    PrefillScatterParams cp{};
    cp.T = T; cp.N = N; cp.n_shared = l.n_shared; cp.Kp = Kp; cp.d_bytes = bf16 ? d * 2 : 0;
    cp.tile_rows = tile_rows;
    cp.nblk = (int)((T + kRouteTokensPerBlock - 1) / kRouteTokensPerBlock);
    cp.ids = rp.ids; cp.w = rp.w; cp.block_hist = rp.block_hist; cp.sb_hist = rp.sb_hist;
    cp.offsets = at<int32_t>(ws, pl.offsets); cp.work_start = at<int32_t>(ws, pl.work_start);
    cp.x = x; cp.xs = bf16 ? at<char>(ws, pl.xs) : nullptr;
    cp.perm = at<int32_t>(ws, pl.perm); cp.row_tok = at<int32_t>(ws, pl.row_tok);
    cp.row_w = at<float>(ws, pl.row_w);
    cp.inv_pos = at<int32_t>(ws, pl.inv_pos);
    if (small) cp.xs = nullptr;  // the tokens are read in place; only the metadata needs the permutation
    if (!routed && (!small || meta)) { ProfScope ps(2, s); EXFOLD_CUDA(launch_prefill_scatter(cp, s)); }

    if (small) {
        DecodeSmallParams sp{};
        sp.x = reinterpret_cast<const __nv_bfloat16*>(x); sp.wg = reinterpret_cast<const __nv_bfloat16*>(w_gate);
        sp.wu = reinterpret_cast<const __nv_bfloat16*>(w_up); sp.wd = reinterpret_cast<const __nv_bfloat16*>(w_down);
        sp.y = reinterpret_cast<__nv_bfloat16*>(y); sp.ids = rp.ids; sp.w_in = rp.w;
        if (small_routed) sp.status = rp.status;
        sp.B = (int)T; sp.N = N; sp.K = Kp; sp.M = N; sp.n_shared = l.n_shared; sp.d = d; sp.I = I;
        sp.max_groups = (int)std::min<int64_t>(N, R) + l.n_shared; sp.max_rows = (int)Rtot;
        sp.H = at<__nv_bfloat16>(ws, pl.H); sp.row_tok = cp.row_tok; sp.row_w = cp.row_w; sp.row_grp = at<int32_t>(ws, pl.row_grp);
        sp.grp_expert = at<int32_t>(ws, pl.grp_expert); sp.n_groups = at<int32_t>(ws, pl.n_groups);
        ProfScope ps(3, s);
        EXFOLD_CUDA(launch_decode_small(sp, small_routed ? &rp : nullptr, sm_count(), s));
    } else if (bf16) {
        GroupedGemmParams g{};
        g.tm_a = tm_xs; g.tm_a2 = tm_x; g.tm_b0 = tm_wg; g.tm_b1 = tm_wu; g.x_rows = (int)T; g.o32 = nullptr;
        g.offsets = cp.offsets; g.work_start = cp.work_start; g.G = G; g.n_routed = N; g.R = (int)R;
        g.d = d; g.I = I; g.n_ntiles = (I + 127) / 128; g.ksplit = 1; g.a_rows = kTileM;
        g.grp_expert = nullptr; g.n_groups_dev = nullptr;
        g.H = at<__nv_bfloat16>(ws, pl.H); g.row_tok = cp.row_tok; g.row_w = cp.row_w;
        g.y = nullptr; g.status = at<DeviceStatus>(ws, pl.status);
        GroupedGemmParams g2 = g;  // GEMM-2: H x W_down -> y (or the per-route buffer O)
        g2.tm_a = tm_h; g2.tm_b0 = tm_wd; g2.tm_b1 = tm_wd_half; g2.n_ntiles = (d + 255) / 256;
        // K' = 1 without a shared expert: every token is written once, straight into y. Otherwise each
        // route's weighted output goes to O (bf16, sorted rows) and the combine kernel sums per token.
        g2.y = direct ? reinterpret_cast<__nv_bfloat16*>(y) : at<__nv_bfloat16>(ws, pl.obuf);
        g2.store_rows = direct ? 0 : 1;
        if (shared_pairs > 0) {  // the shared expert's pairs of GEMM-1 are done (or running) on the second stream
            g.shared_split = 2;
            EXFOLD_CUDA(cudaStreamWaitEvent(s, early_side->mid, 0));
        }
        rc = mixed ? enqueue_mixed_gemms(g, g2, at<char>(ws, pl.xs), R, Rtot, x, w_gate, w_up, G, s)
                   : enqueue_expert_gemms(g, g2, Rtot, pairs, shared_pairs, s);
        if (rc != EXFOLD_OK) return rc;
        early_join.armed = false;  // the passes above have joined the second stream
        if (!direct) {
            ProfScope ps(5, s);
            EXFOLD_CUDA(launch_combine_rows(at<__nv_bfloat16>(ws, pl.obuf), cp.inv_pos, T, Kp, d, l.n_shared, nullptr, 1, 0,
                                            reinterpret_cast<__nv_bfloat16*>(y), s));
        }
    } else {
        FfnF32Params fp = f32_params(x, w_gate, w_up, w_down, d, I, G, cp.tile_rows);
        fp.offsets = cp.offsets; fp.tile_start = cp.work_start; fp.row_tok = cp.row_tok; fp.row_w = cp.row_w;
        if (direct) fp.y = reinterpret_cast<float*>(y);
        else fp.out = at<float>(ws, pl.out);
        if (routed) {
            const FfnF32Route rt{rp, l.n_shared, cp.offsets, cp.perm, cp.inv_pos, cp.row_tok, cp.row_w};
            ProfScope ps(10, s);
            EXFOLD_CUDA(launch_ffn_f32_routed(fp, rt, Rtot, s));
        } else {
            ProfScope ps(10, s);
            EXFOLD_CUDA(launch_ffn_f32(fp, Rtot, sm_count(), s));
        }
        if (!direct) {
            ProfScope ps(11, s);
            EXFOLD_CUDA(launch_combine_f32(fp.out, cp.inv_pos, cp.row_w, T, Kp, d, l.n_shared, nullptr,
                                           reinterpret_cast<float*>(y), s));
        }
    }
    if (meta) {
        if ((rc = copy_meta(meta->ids, rp.ids, (size_t)R * 4, s))) return rc;
        if ((rc = copy_meta(meta->w, rp.w, (size_t)R * 4, s))) return rc;
        if ((rc = copy_meta(meta->omit_src, rp.omit_src, (size_t)T * (K - Kp) * 4, s))) return rc;
        if ((rc = copy_meta(meta->omit_tgt, rp.omit_tgt, (size_t)T * (K - Kp) * 4, s))) return rc;
        if ((rc = copy_meta(meta->perm, cp.perm, (size_t)R * 4, s))) return rc;
        if ((rc = copy_meta(meta->offsets, cp.offsets, (size_t)(N + 1) * 4, s))) return rc;
    }
    return EXFOLD_OK;
}

static int router_enqueue(const exfold_layer* layer, const void* x, const void* w_router, int64_t T, float* logits,
                          void* ws, size_t ws_bytes, cudaStream_t s, bool clear_status);

// Dynamic (tables != null) or static (spool != null) decode step.
// w_router != null: the router scores are computed first (into `logits`, which is then an output).
static int decode_impl(const exfold_layer* layer, const void* x, const float* logits, int64_t B, const void* w_gate,
                       const void* w_up, const void* w_down, const exfold_tables* tables,
                       const exfold_static_pool* spool, int32_t pool_m, void* y, const exfold_decode_meta* meta,
                       void* ws, size_t ws_bytes, void* cuda_stream, const void* w_router = nullptr) {
    exfold_tables dummy{};  // the static path needs no tables: satisfy the common pointer checks
    if (spool != nullptr) {
        if (!spool->pool_ids || !spool->target || !spool->scale) return EXFOLD_ERR_INVALID_ARG;
        dummy.S = dummy.L = dummy.h = dummy.lnh = spool->scale;
        tables = &dummy;
        pool_m = spool->pool_m;
    }
    int rc = check_common(layer, x, logits, B, w_gate, w_up, w_down, tables, y, ws);
    if (rc != EXFOLD_OK) return rc;
    const exfold_layer& l = *layer;
    if (pool_m < 1 || pool_m > l.n_experts) return EXFOLD_ERR_INVALID_ARG;
    if (B > kMaxDecodeBatch || B * l.top_k > 4096) return EXFOLD_ERR_UNSUPPORTED;
    const int N = l.n_experts, K = l.top_k, d = l.hidden, I = l.inter, G = N + l.n_shared;
    const Plan pl = make_plan(l, B, K);
    if (ws_bytes < pl.total) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    const bool bf16 = l.dtype == EXFOLD_BF16;
    const int max_rows = (int)(B * K + B * l.n_shared);
    // a group has at most B rows: the token box of the GEMMs needs only that many (multiple of 32, <= 128)
    const int a_rows = (int)std::min<int64_t>(kTileM, (B + 31) / 32 * 32);

    CUtensorMap tm_wg, tm_wu, tm_h;
    if (bf16) {
        const uint64_t E = (uint64_t)G;
        bool ok = make_tmap(&tm_wg, w_gate, E * I, d, 128) && make_tmap(&tm_wu, w_up, E * I, d, 128) &&
                  make_tmap(&tm_h, at<char>(ws, pl.H), (uint64_t)max_rows, I, a_rows);
        if (!ok) return EXFOLD_ERR_CUDA;
    }
    prof_reset();
    PdlScope pdl_scope(true);

    DecodeRouteParams rp{};
    rp.logits = logits; rp.S = tables->S; rp.L = tables->L; rp.h = tables->h;
    rp.B = (int)B; rp.N = N; rp.K = K; rp.M = pool_m; rp.n_shared = l.n_shared;
    if (spool != nullptr) {
        rp.st_pool = spool->pool_ids; rp.st_target = spool->target; rp.st_scale = spool->scale;
    }
    rp.pool_ids = at<int32_t>(ws, pl.pool_ids); rp.pool_size = at<int32_t>(ws, pl.pool_size);
    rp.pool_mask = at<uint32_t>(ws, pl.pool_mask); rp.ids = at<int32_t>(ws, pl.ids); rp.w = at<float>(ws, pl.w);
    rp.target = at<int32_t>(ws, pl.target); rp.scale = at<float>(ws, pl.scale);
    rp.row_tok = at<int32_t>(ws, pl.row_tok); rp.row_w = at<float>(ws, pl.row_w);
    rp.grp_expert = at<int32_t>(ws, pl.grp_expert); rp.grp_off = at<int32_t>(ws, pl.grp_off);
    rp.grp_tiles = at<int32_t>(ws, pl.grp_tiles); rp.n_groups = at<int32_t>(ws, pl.n_groups);
    rp.slot_row = at<int32_t>(ws, pl.inv_pos);
    rp.status = at<DeviceStatus>(ws, pl.status);
    if (bf16) {
        DecodeTopkParams tp{};
        tp.logits = logits; tp.x = reinterpret_cast<const __nv_bfloat16*>(x);
        tp.w_router = reinterpret_cast<const __nv_bfloat16*>(w_router); tp.logits_out = const_cast<float*>(logits);
        tp.B = (int)B; tp.N = N; tp.K = K; tp.d = d;
        tp.ids = rp.ids; tp.w64 = at<double>(ws, pl.w64); tp.status = rp.status;
        // the remapped slots go to a second array: the Top-K ids are read by every CTA while one of them writes
        int32_t* const out_ids = at<int32_t>(ws, pl.perm);
        if (decode_small_fits((int)B, K, d, w_gate, w_up, w_down)) {
            if (w_router != nullptr) { ProfScope ps(6, s); EXFOLD_CUDA(launch_decode_topk(tp, s)); }
            DecodeSmallParams sp{};
            sp.x = tp.x; sp.wg = reinterpret_cast<const __nv_bfloat16*>(w_gate); sp.wu = reinterpret_cast<const __nv_bfloat16*>(w_up);
            sp.wd = reinterpret_cast<const __nv_bfloat16*>(w_down); sp.y = reinterpret_cast<__nv_bfloat16*>(y);
            sp.logits = w_router == nullptr ? logits : nullptr; sp.ids = tp.ids; sp.w64 = tp.w64;
            sp.S = tables->S; sp.L = tables->L; sp.h = tables->h;
            sp.st_pool = rp.st_pool; sp.st_target = rp.st_target; sp.st_scale = rp.st_scale;
            sp.B = (int)B; sp.N = N; sp.K = K; sp.M = pool_m; sp.n_shared = l.n_shared; sp.d = d; sp.I = I;
            sp.max_groups = (int)std::min<int64_t>(std::min(pool_m, N), B * K) + l.n_shared; sp.max_rows = max_rows;
            if (meta) {
                sp.pool_ids = rp.pool_ids; sp.pool_size = rp.pool_size; sp.pool_mask = rp.pool_mask;
                sp.out_ids = out_ids; sp.out_w = rp.w; sp.target = rp.target; sp.scale = rp.scale;
            }
            sp.H = at<__nv_bfloat16>(ws, pl.H); sp.row_tok = rp.row_tok; sp.row_w = rp.row_w;
            sp.row_grp = at<int32_t>(ws, pl.row_grp); sp.grp_expert = rp.grp_expert; sp.n_groups = rp.n_groups;
            sp.status = w_router == nullptr ? rp.status : nullptr;
            { ProfScope ps(14, s); EXFOLD_CUDA(launch_decode_small(sp, nullptr, sm_count(), s)); }
        } else {
            // Token-parallel Top-K (with the router scores when w_router is given) -> gate/up kernel that finishes the
            // routing in its prologue and streams the pool's gate and up weights against x in place -> grouped down
            // projection over the compact rows -> per-token sum of the rows.
            int stages = 0, scratch_off = 0, ar = 0;
            const int max_groups = std::min(pool_m, N) + l.n_shared, sms = std::min(sm_count(), kMaxCtas);
            const int alt = decode_ffn_alt((int)B, max_groups, I, sms);
            decode_ffn_smem_plan((int)B, K, N, alt, &stages, &scratch_off, &ar);
            if (stages < 2) return EXFOLD_ERR_UNSUPPORTED;
            // Fewer (expert, column tile) items than half the SMs (few experts, large I): K is split in two so that
            // enough SMs stream W_down; each part's rows go to a plane of their own (the two planes are the row buffer
            // and the unused gathered-rows region before it) and are summed, in order, by the kernel after.
            const int64_t row_tiles = (int64_t)max_groups * ((B + kTileM - 1) / kTileM), base_items = row_tiles * ((d + 255) / 256);
            const int ksplit = (2 * base_items < sms && I / 64 >= 8) ? kMaxDecodeKsplit : 1;
            // Still few: narrower column tiles, as long as each has an SM to itself. (Fewer columns take the tensor pipe less time,
            // but a k-block's copies and hand-over stay what they were: more rounds of narrower tiles lose.) Whole call, 256
            // columns / these: Qwen3 shape 128 tokens, pool 2 29.2 / 27.2 us; GLM shape 100 tokens, pool 1 47.1 / 45.1; Mixtral
            // shape 200 tokens, pool 1 152.8 / 144.3; 64 columns in three rounds: GLM shape 16 tokens, pool 4 50.4 / 60.0.
            int n_cols = 256;
            while (n_cols > 64 && base_items * (512 / n_cols) * ksplit <= sms) n_cols >>= 1;
            CUtensorMap tm_wd;
            const uint64_t E = (uint64_t)G;
            DecodeFfnParams fp{};
            fp.alt = alt; fp.tm_wg = tm_wg; fp.tm_wu = tm_wu;
            if (!make_tmap(&tm_wd, w_down, E * d, I, n_cols) || !make_tmap(&fp.tm_x, x, (uint64_t)B, d, ar) ||
                (B > 128 && !make_tmap(&fp.tm_xg, x, (uint64_t)B, d, 1)) ||
                !make_tmap(&fp.tm_wg64, w_gate, E * I, d, 64) || !make_tmap(&fp.tm_wu64, w_up, E * I, d, 64) ||
                (alt && (!make_tmap(&fp.tm_wg_alt, w_gate, E * I, d, alt) || !make_tmap(&fp.tm_wu_alt, w_up, E * I, d, alt))))
                return EXFOLD_ERR_CUDA;
            { ProfScope ps(6, s); EXFOLD_CUDA(launch_decode_topk(tp, s)); }
            fp.ids = rp.ids; fp.w64 = tp.w64; fp.S = tables->S; fp.L = tables->L; fp.h = tables->h;
            fp.st_pool = rp.st_pool; fp.st_target = rp.st_target; fp.st_scale = rp.st_scale;
            fp.B = (int)B; fp.N = N; fp.K = K; fp.M = pool_m; fp.n_shared = l.n_shared; fp.d = d; fp.I = I; fp.a_rows = ar;
            fp.stages = stages; fp.scratch_off = scratch_off;
            if (meta) {
                fp.pool_ids = rp.pool_ids; fp.pool_size = rp.pool_size; fp.pool_mask = rp.pool_mask;
                fp.out_ids = out_ids; fp.out_w = rp.w; fp.target = rp.target; fp.scale = rp.scale;
            }
            fp.H = at<__nv_bfloat16>(ws, pl.H); fp.row_tok = rp.row_tok; fp.row_w = rp.row_w;
            fp.slot_row = rp.slot_row;
            fp.grp_expert = rp.grp_expert; fp.grp_off = rp.grp_off; fp.grp_tiles = rp.grp_tiles; fp.n_groups = rp.n_groups;
            fp.status = rp.status;
            { ProfScope ps(14, s); EXFOLD_CUDA(launch_decode_ffn(fp, sm_count(), s)); }
            // Down projection on the grouped GEMM-2 kernel over the compact rows (the whole intermediate dimension is
            // its K, so no partial outputs meet in memory); each row's weighted output is stored once, in bf16, and a
            // token's rows are then summed in slot order: no atomics, so a decode step is reproducible bit for bit.
            GroupedGemmParams g{};
            g.tm_a = tm_h; g.tm_a2 = tm_h; g.x_rows = 1; g.o32 = nullptr;
            g.offsets = rp.grp_off; g.work_start = rp.grp_tiles; g.G = max_groups; g.n_routed = 0x7fffffff;
            g.R = max_rows; g.d = d; g.I = I; g.a_rows = a_rows;
            g.grp_expert = rp.grp_expert; g.n_groups_dev = rp.n_groups;
            g.H = fp.H; g.row_tok = rp.row_tok; g.row_w = rp.row_w;
            g.y = at<__nv_bfloat16>(ws, pl.obuf); g.store_rows = 1; g.status = rp.status;
            g.ksplit = ksplit; g.n_cols = n_cols; g.n_ntiles = (d + n_cols - 1) / n_cols; g.tm_b0 = tm_wd; g.tm_b1 = tm_wd;
            const int64_t items = row_tiles * g.n_ntiles * ksplit;
            g.y = g.ksplit > 1 ? at<__nv_bfloat16>(ws, pl.obuf) - (size_t)max_rows * d : at<__nv_bfloat16>(ws, pl.obuf);
            { ProfScope ps(9, s); EXFOLD_CUDA(launch_grouped_gemm2(g, (int)std::min<int64_t>(sms, items), s)); }
            { ProfScope ps(5, s); EXFOLD_CUDA(launch_combine_rows(g.y, fp.slot_row, B, K, d, l.n_shared, rp.n_groups + 2, g.ksplit,
                                                           max_rows, reinterpret_cast<__nv_bfloat16*>(y), s)); }
        }
        rp.ids = out_ids;  // for the metadata copies below
    } else {
        if (w_router != nullptr) {
            rc = router_enqueue(layer, x, w_router, B, const_cast<float*>(logits), ws, ws_bytes, s, false);
            if (rc != EXFOLD_OK) return rc;
        }
        const int max_groups = std::min(pool_m, N) + l.n_shared;
        // a token has at most as many rows as the pool has experts
        const int64_t rows = B * std::min(K, (int)pool_m) + B * l.n_shared;
        rp.tile_rows = ffn_f32_tile_rows(rows, max_groups, d, I, sm_count());
        const bool routed = ffn_f32_routes(true, B, rows, max_groups, N, K, d, I, rp.tile_rows, sm_count());
        if (!routed) { ProfScope ps(6, s); EXFOLD_CUDA(launch_decode_route(rp, s)); }
        FfnF32Params fp = f32_params(x, w_gate, w_up, w_down, d, I, max_groups, rp.tile_rows);
        fp.offsets = rp.grp_off; fp.tile_start = rp.grp_tiles; fp.grp_expert = rp.grp_expert; fp.n_groups_dev = rp.n_groups;
        fp.row_tok = rp.row_tok; fp.row_w = rp.row_w; fp.out = at<float>(ws, pl.out);
        { ProfScope ps(10, s); EXFOLD_CUDA(routed ? launch_ffn_f32_routed(fp, rp, rows, s) : launch_ffn_f32(fp, rows, sm_count(), s)); }
        { ProfScope ps(11, s); EXFOLD_CUDA(launch_combine_f32(fp.out, rp.slot_row, rp.row_w, B, K, d, l.n_shared, rp.n_groups + 2,
                                                              reinterpret_cast<float*>(y), s)); }
    }
    if (meta) {
        if ((rc = copy_meta(meta->pool_ids, rp.pool_ids, (size_t)pool_m * 4, s))) return rc;
        if ((rc = copy_meta(meta->pool_size, rp.pool_size, 4, s))) return rc;
        if ((rc = copy_meta(meta->pool_mask, rp.pool_mask, (size_t)((N + 31) / 32) * 4, s))) return rc;
        if ((rc = copy_meta(meta->ids, rp.ids, (size_t)B * K * 4, s))) return rc;
        if ((rc = copy_meta(meta->w, rp.w, (size_t)B * K * 4, s))) return rc;
        if ((rc = copy_meta(meta->target, rp.target, (size_t)N * 4, s))) return rc;
        if ((rc = copy_meta(meta->scale, rp.scale, (size_t)N * 4, s))) return rc;
    }
    return EXFOLD_OK;
}

int exfold_moe_decode(const exfold_layer* layer, const void* x, const float* logits, int64_t B, const void* w_gate,
                      const void* w_up, const void* w_down, const exfold_tables* tables, int32_t pool_m, void* y,
                      const exfold_decode_meta* meta, void* ws, size_t ws_bytes, void* cuda_stream) {
    return decode_impl(layer, x, logits, B, w_gate, w_up, w_down, tables, nullptr, pool_m, y, meta, ws, ws_bytes,
                       cuda_stream);
}

int exfold_moe_decode_static(const exfold_layer* layer, const void* x, const float* logits, int64_t B,
                             const void* w_gate, const void* w_up, const void* w_down, const exfold_static_pool* pool,
                             void* y, const exfold_decode_meta* meta, void* ws, size_t ws_bytes, void* cuda_stream) {
    if (pool == nullptr) return EXFOLD_ERR_INVALID_ARG;
    return decode_impl(layer, x, logits, B, w_gate, w_up, w_down, nullptr, pool, pool->pool_m, y, meta, ws, ws_bytes,
                       cuda_stream);
}

int exfold_static_pool_build(const exfold_layer* layer, const exfold_tables* tables, int32_t pool_m,
                             exfold_static_pool* out, void* cuda_stream) {
    if (!valid_layer(layer) || !tables || !tables->S || !tables->L || !tables->h || !out) return EXFOLD_ERR_INVALID_ARG;
    if (!out->pool_ids || !out->target || !out->scale) return EXFOLD_ERR_INVALID_ARG;
    if (pool_m < 1 || pool_m > layer->n_experts) return EXFOLD_ERR_INVALID_ARG;
    out->pool_m = pool_m;
    EXFOLD_CUDA(launch_static_pool(layer->n_experts, pool_m, tables->S, tables->L, tables->h, out->pool_ids,
                                   out->target, out->scale, reinterpret_cast<cudaStream_t>(cuda_stream)));
    return EXFOLD_OK;
}

// The arguments of one calibration, before anything is launched. m * Ke <= 2^30 rows follow from m <= 2^22, Ke <= 256.
static int calibrate_check(const exfold_layer* layer, const void* x_cal, const float* logits_cal, int64_t m,
                           const void* w_gate, const void* w_up, const void* w_down, const exfold_calib_opts* opts,
                           const exfold_tables* out, const void* ws, size_t ws_bytes) {
    if (!valid_layer(layer) || !x_cal || !w_gate || !w_up || !w_down || !opts || !out || !ws)
        return EXFOLD_ERR_INVALID_ARG;
    if (!out->S || !out->L || !out->h || !out->lnh) return EXFOLD_ERR_INVALID_ARG;
    if (m < 1 || m > (int64_t)1 << 22) return EXFOLD_ERR_INVALID_ARG;
    if (opts->mode != 0 && opts->mode != 1) return EXFOLD_ERR_INVALID_ARG;
    if (opts->mode == 0 && !logits_cal) return EXFOLD_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(ws) & 255) != 0) return EXFOLD_ERR_INVALID_ARG;
    exfold_layer lc = *layer;
    lc.n_shared = 0;  // the shared expert is never folded, so it is not calibrated
    if (ws_bytes < make_plan(lc, m, opts->mode == 1 ? lc.n_experts : lc.top_k).total) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    if (layer->dtype == EXFOLD_BF16 && (!aligned16(x_cal) || !aligned16(w_gate) || !aligned16(w_up) || !aligned16(w_down)))
        return EXFOLD_ERR_INVALID_ARG;
    return EXFOLD_OK;
}

// Enqueues one calibration of checked arguments on the stream (no synchronisation); the number of unobserved experts lands in
// result_words()[job] when the stream gets there.
static int calibrate_enqueue(const exfold_layer* layer, const void* x_cal, const float* logits_cal, int64_t m,
                             const void* w_gate, const void* w_up, const void* w_down, const exfold_calib_opts* opts,
                             exfold_tables* out, void* ws, void* cuda_stream, int job) {
    const exfold_layer& l = *layer;
    const int N = l.n_experts, K = l.top_k, d = l.hidden, I = l.inter;
    const int Ke = opts->mode == 1 ? N : K;
    exfold_layer lc = l;
    lc.n_shared = 0;
    const Plan pl = make_plan(lc, m, Ke);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);

    int* counts = result_words();
    if (!counts) return EXFOLD_ERR_CUDA;
    const bool tensor_path = l.dtype == EXFOLD_BF16;
    const bool pairs = tensor_path && use_pairs(m * Ke, N, d, I);
    const bool mixed = tensor_path && use_mixed(m * Ke, N, d, I);
    PdlScope pdl_scope(!pairs || mixed);  // as in prefill: a chain of kernels of which most are short
    DeviceStatus* status = at<DeviceStatus>(ws, pl.status);
    int32_t* ids = at<int32_t>(ws, pl.ids);
    if (opts->mode == 0) {
        // Top-K in router order: the prefill route kernel with K' = K and no ln(h) term
        PrefillRouteParams rp{};
        rp.logits = logits_cal; rp.S = out->S; rp.L = out->L; rp.lnh = nullptr;
        rp.T = m; rp.N = N; rp.K = K; rp.Kp = K; rp.ids = ids; rp.w = at<float>(ws, pl.w);
        rp.loss_thr = INFINITY;
        rp.omit_src = nullptr; rp.omit_tgt = nullptr; rp.block_hist = at<int32_t>(ws, pl.block_hist);
        rp.sb_hist = at<int32_t>(ws, pl.sb_hist);
        rp.status = status;
        rp.queue = mixed ? status->queue : nullptr;
        EXFOLD_CUDA(launch_prefill_route(rp, s));
    } else {
        EXFOLD_CUDA(cudaMemsetAsync(status, 0, sizeof(DeviceStatus), s));
        EXFOLD_CUDA(launch_iota_ids(ids, m, N, s));
    }
    const int64_t Rc = m * Ke;
    CalibStatsParams cs{};
    const size_t NN = (size_t)N * N, calib_bytes = NN * (3 * 8 + 4) + (size_t)N * (8 + 4);
    // Expert outputs, one fp32 row per (token, expert), sorted by expert. Mode 0 sorts the routed rows like prefill; in
    // mode 1 every expert's rows are the tokens themselves, read from x_cal without a copy.
    int32_t* offsets = at<int32_t>(ws, pl.offsets);
    int32_t* work_start = at<int32_t>(ws, pl.work_start);
    int32_t* row_tok = at<int32_t>(ws, pl.row_tok);
    const int tile_rows = mixed ? kMixedTiles : tensor_path ? kTileM : ffn_f32_tile_rows(Rc, N, d, I, sm_count());
    if (opts->mode == 0) {
        PrefillScatterParams cp{};
        cp.T = m; cp.N = N; cp.n_shared = 0; cp.Kp = K; cp.d_bytes = tensor_path ? d * 2 : 0; cp.tile_rows = tile_rows;
        cp.nblk = (int)((m + kRouteTokensPerBlock - 1) / kRouteTokensPerBlock);
        cp.ids = ids; cp.w = at<float>(ws, pl.w); cp.block_hist = at<int32_t>(ws, pl.block_hist);
        cp.sb_hist = at<int32_t>(ws, pl.sb_hist);
        cp.offsets = offsets; cp.work_start = work_start;
        cp.x = x_cal; cp.xs = tensor_path ? at<char>(ws, pl.xs) : nullptr;
        cp.perm = at<int32_t>(ws, pl.perm); cp.row_tok = row_tok;
        cp.row_w = at<float>(ws, pl.row_w);
        cp.inv_pos = at<int32_t>(ws, pl.inv_pos);
        cp.zero = at<int32_t>(ws, pl.calib); cp.zero_words = (int)(calib_bytes / 4);  // the pair sums
        EXFOLD_CUDA(launch_prefill_scatter(cp, s));
        cs.inv_pos = cp.inv_pos;
    } else {
        EXFOLD_CUDA(cudaMemsetAsync(at<char>(ws, pl.calib), 0, calib_bytes, s));
        EXFOLD_CUDA(launch_calib_common_rows(offsets, work_start, m, N, tile_rows, s));
        cs.inv_pos = nullptr; cs.tok_stride = 1; cs.slot_stride = m;
    }
    if (tensor_path) {
        // GEMM-1 (SwiGLU, H in bf16) -> GEMM-2 with the raw fp32 accumulators stored per sorted row
        CUtensorMap tm_xs, tm_x, tm_wg, tm_wu, tm_h, tm_wd, tm_wd_half;
        const uint64_t E = (uint64_t)N;
        bool ok = make_tmap(&tm_xs, at<char>(ws, pl.xs), (uint64_t)Rc, d, 128) &&
                  make_tmap(&tm_x, x_cal, (uint64_t)m, d, 128) && make_tmap(&tm_wg, w_gate, E * I, d, 128) &&
                  make_tmap(&tm_wu, w_up, E * I, d, 128) && make_tmap(&tm_h, at<char>(ws, pl.H), (uint64_t)Rc, I, 128) &&
                  make_tmap(&tm_wd, w_down, E * d, I, 256) && make_tmap(&tm_wd_half, w_down, E * d, I, 128);
        if (!ok) return EXFOLD_ERR_CUDA;
        GroupedGemmParams g{};
        g.tm_a = tm_xs; g.tm_a2 = tm_x; g.tm_b0 = tm_wg; g.tm_b1 = tm_wu;
        g.offsets = offsets; g.work_start = work_start; g.G = N;
        g.n_routed = opts->mode == 0 ? N : 0;  // mode 1: every group reads x_cal directly
        g.R = 0; g.x_rows = (int)m;
        g.d = d; g.I = I; g.n_ntiles = (I + 127) / 128; g.ksplit = 1; g.a_rows = kTileM;
        g.H = at<__nv_bfloat16>(ws, pl.H); g.row_tok = row_tok; g.row_w = at<float>(ws, pl.row_w);
        g.status = at<DeviceStatus>(ws, pl.status);
        GroupedGemmParams g2 = g;
        g2.tm_a = tm_h; g2.tm_b0 = tm_wd; g2.tm_b1 = tm_wd_half; g2.n_ntiles = (d + 255) / 256;
        g2.o32 = at<float>(ws, pl.xs);  // spans the xs and obuf regions (GEMM-1 is done with xs)
        const int rc = mixed ? enqueue_mixed_gemms(g, g2, at<char>(ws, pl.xs), Rc, Rc, x_cal, w_gate, w_up, N, s)
                             : enqueue_expert_gemms(g, g2, Rc, pairs, 0, s);
        if (rc != EXFOLD_OK) return rc;
        cs.out = g2.o32;
    } else {
        FfnF32Params fp = f32_params(x_cal, w_gate, w_up, w_down, d, I, N, tile_rows);
        fp.offsets = offsets; fp.tile_start = work_start; fp.x_rows = m;
        fp.row_tok = opts->mode == 0 ? row_tok : nullptr;
        fp.out = at<float>(ws, pl.out);
        EXFOLD_CUDA(launch_ffn_f32(fp, Rc, sm_count(), s));
        cs.out = fp.out;
    }

    char* cb = at<char>(ws, pl.calib);
    cs.ids = ids; cs.status = status; cs.m = m; cs.Ke = Ke; cs.d = d; cs.N = N;
    cs.A = reinterpret_cast<double*>(cb); cs.Bv = cs.A + NN; cs.C = cs.Bv + NN;
    cs.H = cs.C + NN;
    cs.cnt = reinterpret_cast<int32_t*>(cs.H + N);
    cs.hc = cs.cnt + NN;
    if (opts->mode == 1 && Ke >= 32)  // many experts per token: Gram-product form of the same sums
        EXFOLD_CUDA(launch_calib_stats_common(cs, at<double>(ws, pl.calib_nrm), sm_count(), s));
    else
        EXFOLD_CUDA(launch_calib_stats(cs, sm_count(), s));
    EXFOLD_CUDA(launch_calib_finalize(cs, *opts, out->S, out->L, out->h, out->lnh, out->n_obs, counts + job, s));
    return EXFOLD_OK;
}

// The jobs' unobserved-expert counts, after the stream has drained
static int calibrate_collect(int n_jobs, int32_t* warn, cudaStream_t s) {
    const int* counts = result_words();
    EXFOLD_CUDA(cudaStreamSynchronize(s));
    int any = 0;
    for (int j = 0; j < n_jobs; ++j) {
        if (warn) warn[j] = counts[j];
        any |= counts[j] > 0;
    }
    return any ? EXFOLD_WARN_UNOBSERVED_EXPERT : EXFOLD_OK;
}

int exfold_calibrate(const exfold_layer* layer, const void* x_cal, const float* logits_cal, int64_t m,
                     const void* w_gate, const void* w_up, const void* w_down, const exfold_calib_opts* opts,
                     exfold_tables* out, void* ws, size_t ws_bytes, void* cuda_stream) {
    int rc = calibrate_check(layer, x_cal, logits_cal, m, w_gate, w_up, w_down, opts, out, ws, ws_bytes);
    if (rc == EXFOLD_OK) rc = calibrate_enqueue(layer, x_cal, logits_cal, m, w_gate, w_up, w_down, opts, out, ws, cuda_stream, 0);
    if (rc != EXFOLD_OK) return rc;
    return calibrate_collect(1, nullptr, reinterpret_cast<cudaStream_t>(cuda_stream));
}

int exfold_calibrate_layers(const exfold_layer* layer, const exfold_calib_job* jobs, int32_t n_jobs,
                            const exfold_calib_opts* opts, int32_t* unobserved, void* ws, size_t ws_bytes,
                            void* cuda_stream) {
    if (!valid_layer(layer) || !jobs || !opts || n_jobs < 1 || n_jobs > EXFOLD_MAX_CALIB_JOBS) return EXFOLD_ERR_INVALID_ARG;
    if (opts->mode != 0 && opts->mode != 1) return EXFOLD_ERR_INVALID_ARG;
    int64_t m_max = 0;
    for (int j = 0; j < n_jobs; ++j) {
        if (!jobs[j].out || jobs[j].m < 1) return EXFOLD_ERR_INVALID_ARG;
        m_max = std::max<int64_t>(m_max, jobs[j].m);
    }
    // The jobs run one after the other on the stream and share the workspace, sized for the largest one.
    const int Ke = opts->mode == 1 ? layer->n_experts : layer->top_k;
    if (ws_bytes < exfold_workspace_bytes(layer, m_max, Ke)) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    for (int j = 0; j < n_jobs; ++j) {
        const exfold_calib_job& b = jobs[j];
        int rc = calibrate_check(layer, b.x_cal, b.logits_cal, b.m, b.w_gate, b.w_up, b.w_down, opts, b.out, ws, ws_bytes);
        if (rc != EXFOLD_OK) return rc;
    }
    for (int j = 0; j < n_jobs; ++j) {
        const exfold_calib_job& b = jobs[j];
        int rc = calibrate_enqueue(layer, b.x_cal, b.logits_cal, b.m, b.w_gate, b.w_up, b.w_down, opts, b.out, ws, cuda_stream, j);
        if (rc != EXFOLD_OK) {  // the jobs before this one still write their tables and their counts
            cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(cuda_stream));
            return rc;
        }
    }
    return calibrate_collect(n_jobs, unobserved, reinterpret_cast<cudaStream_t>(cuda_stream));
}

// Router scores on the stream; `clear_status`: the call stands alone (clears the status record itself)
static int router_enqueue(const exfold_layer* layer, const void* x, const void* w_router, int64_t T, float* logits,
                          void* ws, size_t ws_bytes, cudaStream_t s, bool clear_status) {
    if (!valid_layer(layer) || !x || !w_router || !logits || !ws || T < 1) return EXFOLD_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(ws) & 255) != 0 || (reinterpret_cast<uintptr_t>(logits) & 15) != 0)
        return EXFOLD_ERR_INVALID_ARG;
    const exfold_layer& l = *layer;
    const int N = l.n_experts, d = l.hidden;
    if (T > (int64_t)1 << 30) return EXFOLD_ERR_UNSUPPORTED;
    exfold_layer lc = l;
    lc.n_shared = 0;
    const Plan pl = make_plan(lc, T, 1);
    if (ws_bytes < pl.total) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    DeviceStatus* status = at<DeviceStatus>(ws, pl.status);
    // fp32 layers, and bf16 batches of at most one row tile (decode): dot products in a fixed order
    if (l.dtype == EXFOLD_F32 || (T <= kTileM && aligned16(x) && aligned16(w_router))) {
        EXFOLD_CUDA(launch_router_simt(x, w_router, l.dtype, T, N, d, logits, clear_status ? status : nullptr, s));
        return EXFOLD_OK;
    }
    if (!aligned16(x) || !aligned16(w_router)) return EXFOLD_ERR_INVALID_ARG;
    RouterGemmParams g{};
    if (!make_tmap(&g.tm_x, x, (uint64_t)T, d, 128) || !make_tmap(&g.tm_wr, w_router, (uint64_t)N, d, (uint32_t)router_npad(N)))
        return EXFOLD_ERR_CUDA;
    g.logits = logits; g.T = (int)T; g.N = N; g.nkb = d / kGemmBK; g.clear_status = clear_status ? 1 : 0; g.status = status;
    EXFOLD_CUDA(launch_router_gemm(g, sm_count(), s));
    return EXFOLD_OK;
}

int exfold_router_logits(const exfold_layer* layer, const void* x, const void* w_router, int64_t T, float* logits,
                         void* ws, size_t ws_bytes, void* cuda_stream) {
    return router_enqueue(layer, x, w_router, T, logits, ws, ws_bytes, reinterpret_cast<cudaStream_t>(cuda_stream),
                          true);
}

int exfold_moe_prefill_layer(const exfold_layer* layer, const void* x, const void* w_router, int64_t T,
                             const void* w_gate, const void* w_up, const void* w_down, const exfold_tables* tables,
                             int32_t k_pre, float* logits, void* y, const exfold_prefill_meta* meta, void* ws,
                             size_t ws_bytes, void* cuda_stream) {
    if (!valid_layer(layer) || k_pre < 1 || k_pre > layer->top_k) return EXFOLD_ERR_INVALID_ARG;
    if (ws_bytes < exfold_workspace_bytes(layer, T < 1 ? 1 : T, k_pre)) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    int rc = router_enqueue(layer, x, w_router, T, logits, ws, ws_bytes, reinterpret_cast<cudaStream_t>(cuda_stream),
                            true);
    if (rc != EXFOLD_OK) return rc;
    // the routing kernel would clear the status record again: an error of the router GEMM must stay visible
    t_keep_status = true;
    rc = exfold_moe_prefill(layer, x, logits, T, w_gate, w_up, w_down, tables, k_pre, y, meta, ws, ws_bytes, cuda_stream);
    t_keep_status = false;
    return rc;
}

int exfold_moe_decode_layer(const exfold_layer* layer, const void* x, const void* w_router, int64_t B,
                            const void* w_gate, const void* w_up, const void* w_down, const exfold_tables* tables,
                            int32_t pool_m, float* logits, void* y, const exfold_decode_meta* meta, void* ws,
                            size_t ws_bytes, void* cuda_stream) {
    if (!valid_layer(layer) || !w_router || !logits) return EXFOLD_ERR_INVALID_ARG;
    if (B < 1 || B > kMaxDecodeBatch) return B < 1 ? EXFOLD_ERR_INVALID_ARG : EXFOLD_ERR_UNSUPPORTED;
    if (ws_bytes < exfold_workspace_bytes(layer, B, layer->top_k)) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    if ((reinterpret_cast<uintptr_t>(logits) & 15) != 0 || !aligned16(w_router)) return EXFOLD_ERR_INVALID_ARG;
    return decode_impl(layer, x, logits, B, w_gate, w_up, w_down, tables, nullptr, pool_m, y, meta, ws, ws_bytes,
                       cuda_stream, w_router);
}

int exfold_moe_prefill_host(const exfold_layer* layer, const void* x_host, const float* logits_host, int64_t T,
                            const void* w_gate, const void* w_up, const void* w_down, const exfold_tables* tables,
                            int32_t k_pre, void* y_host, const exfold_prefill_meta* meta, void* ws, size_t ws_bytes,
                            void* cuda_stream) {
    if (!valid_layer(layer) || !x_host || !logits_host || !y_host || !ws || T < 1) return EXFOLD_ERR_INVALID_ARG;
    if (k_pre < 1 || k_pre > layer->top_k) return EXFOLD_ERR_INVALID_ARG;
    const size_t main_bytes = exfold_workspace_bytes(layer, T, k_pre);
    const size_t el = layer->dtype == EXFOLD_BF16 ? 2 : 4;
    const size_t xb = (size_t)T * layer->hidden * el, lb = (size_t)T * layer->n_experts * 4;
    if (ws_bytes < main_bytes + exfold_host_staging_bytes(layer, T)) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    char* stage = reinterpret_cast<char*>(ws) + main_bytes;
    char* xd = stage;
    char* yd = xd + align_up(xb, 256);
    char* ld = yd + align_up(xb, 256);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    // Tokens are independent, so a long prompt goes through in chunks: chunk c+1 is copied in and chunk c-1 copied
    // out (two helper streams, both PCIe directions) while chunk c is computed on the caller's stream. Routing
    // metadata describes the whole call (one permutation over all routes), so a call that asks for it is not split.
    const int64_t chunk_tokens = 2048;
    int chunks = meta != nullptr ? 1 : (int)std::min<int64_t>(kMaxHostChunks, T / chunk_tokens);
    if (chunks <= 1) {
        EXFOLD_CUDA(cudaMemcpyAsync(xd, x_host, xb, cudaMemcpyHostToDevice, s));
        EXFOLD_CUDA(cudaMemcpyAsync(ld, logits_host, lb, cudaMemcpyHostToDevice, s));
        int rc = exfold_moe_prefill(layer, xd, reinterpret_cast<const float*>(ld), T, w_gate, w_up, w_down, tables,
                                    k_pre, yd, meta, ws, main_bytes, cuda_stream);
        if (rc != EXFOLD_OK) return rc;
        EXFOLD_CUDA(cudaMemcpyAsync(y_host, yd, xb, cudaMemcpyDeviceToHost, s));
        return EXFOLD_OK;
    }
    ThreadDeviceState* hp = host_helpers();  // created once per host thread and device
    if (!hp) return EXFOLD_ERR_CUDA;
    ThreadDeviceState& h = *hp;
    // the staging buffers may still be in use by earlier work on the caller's stream
    EXFOLD_CUDA(cudaEventRecord(h.start, s));
    EXFOLD_CUDA(cudaStreamWaitEvent(h.in, h.start, 0));
    EXFOLD_CUDA(cudaStreamWaitEvent(h.out, h.start, 0));
    const size_t row_x = (size_t)layer->hidden * el, row_l = (size_t)layer->n_experts * 4;
    const int64_t per = ((T + chunks - 1) / chunks + 127) / 128 * 128;  // whole row tiles per chunk, all tokens covered
    for (int c = 0; c < chunks; ++c) {
        const int64_t t0 = c * per, n = std::min<int64_t>(per, T - t0);
        if (n <= 0) break;
        EXFOLD_CUDA(cudaMemcpyAsync(xd + t0 * row_x, reinterpret_cast<const char*>(x_host) + t0 * row_x, n * row_x,
                                    cudaMemcpyHostToDevice, h.in));
        EXFOLD_CUDA(cudaMemcpyAsync(ld + t0 * row_l, reinterpret_cast<const char*>(logits_host) + t0 * row_l,
                                    n * row_l, cudaMemcpyHostToDevice, h.in));
        EXFOLD_CUDA(cudaEventRecord(h.copied[c], h.in));
    }
    for (int c = 0; c < chunks; ++c) {
        const int64_t t0 = c * per, n = std::min<int64_t>(per, T - t0);
        if (n <= 0) break;
        EXFOLD_CUDA(cudaStreamWaitEvent(s, h.copied[c], 0));
        t_keep_status = c > 0;  // an error recorded by an earlier chunk stays visible
        int rc = exfold_moe_prefill(layer, xd + t0 * row_x, reinterpret_cast<const float*>(ld + t0 * row_l), n, w_gate,
                                    w_up, w_down, tables, k_pre, yd + t0 * row_x, nullptr, ws, main_bytes, cuda_stream);
        t_keep_status = false;
        if (rc != EXFOLD_OK) return rc;
        EXFOLD_CUDA(cudaEventRecord(h.computed[c], s));
        EXFOLD_CUDA(cudaStreamWaitEvent(h.out, h.computed[c], 0));
        EXFOLD_CUDA(cudaMemcpyAsync(reinterpret_cast<char*>(y_host) + t0 * row_x, yd + t0 * row_x, n * row_x,
                                    cudaMemcpyDeviceToHost, h.out));
    }
    EXFOLD_CUDA(cudaEventRecord(h.done, h.out));
    EXFOLD_CUDA(cudaStreamWaitEvent(s, h.done, 0));  // the call is complete, in the caller's stream order, when y_host is
    return EXFOLD_OK;
}

int exfold_moe_decode_host(const exfold_layer* layer, const void* x_host, const float* logits_host, int64_t B,
                           const void* w_gate, const void* w_up, const void* w_down, const exfold_tables* tables,
                           int32_t pool_m, void* y_host, const exfold_decode_meta* meta, void* ws, size_t ws_bytes,
                           void* cuda_stream) {
    if (!valid_layer(layer) || !x_host || !logits_host || !y_host || !ws || B < 1) return EXFOLD_ERR_INVALID_ARG;
    const size_t main_bytes = exfold_workspace_bytes(layer, B, layer->top_k);
    const size_t el = layer->dtype == EXFOLD_BF16 ? 2 : 4;
    const size_t xb = (size_t)B * layer->hidden * el, lb = (size_t)B * layer->n_experts * 4;
    if (ws_bytes < main_bytes + exfold_host_staging_bytes(layer, B)) return EXFOLD_ERR_WORKSPACE_TOO_SMALL;
    char* stage = reinterpret_cast<char*>(ws) + main_bytes;
    char* xd = stage;
    char* yd = xd + align_up(xb, 256);
    char* ld = yd + align_up(xb, 256);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    EXFOLD_CUDA(cudaMemcpyAsync(xd, x_host, xb, cudaMemcpyHostToDevice, s));
    EXFOLD_CUDA(cudaMemcpyAsync(ld, logits_host, lb, cudaMemcpyHostToDevice, s));
    int rc = exfold_moe_decode(layer, xd, reinterpret_cast<const float*>(ld), B, w_gate, w_up, w_down, tables, pool_m,
                               yd, meta, ws, main_bytes, cuda_stream);
    if (rc != EXFOLD_OK) return rc;
    EXFOLD_CUDA(cudaMemcpyAsync(y_host, yd, xb, cudaMemcpyDeviceToHost, s));
    return EXFOLD_OK;
}

}  // extern "C"
