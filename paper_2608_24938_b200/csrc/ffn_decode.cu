// Decode: gate/up half of the expert FFN over the expert pool (Eq. 1 with the pool of Eq. 11 / 14), with the
// batch-level half of the routing in the kernel's prologue.
//
// Decode cost is the bytes of the distinct experts that are loaded ("Phase-specific budgets"), so every SM should
// stream weights from the first microsecond on and nothing else should cross HBM. One persistent CTA per SM. A
// work item is (pool expert, tile of <= 128 tokens, slice of s = 128 or 64 intermediate features):
//
//   acc[tokens, gate s | up s] = x[tokens, :] * [W_gate[slice, :]; W_up[slice, :]]^T        K = d
//   H[row(token, expert), slice] = silu(gate) * up   -> bf16, only for the tokens the expert serves
//
// Tokens are the 128-row M operand, read from x IN PLACE (all B tokens of the tile: no gathered copy; a token the
// expert does not serve costs nothing extra and is simply not stored), weights the N = 256 operand, which is the
// orientation in which a tcgen05.mma consumes weight bytes fastest (its cost follows M, not N). Above 128 tokens a
// group of few rows is one item with its rows gathered instead (kGatherRows below). The two halves of
// tensor memory alternate between items, so the SwiGLU epilogue of one item overlaps the MMAs of the next.
// H is compact: one row per distinct (token, pool expert) pair, grouped by pool rank, tokens ascending. The down
// projection then runs on the grouped GEMM-2 kernel with the whole intermediate dimension as K, which keeps the
// cross-CTA reduction out of memory: measured, a version that also did the down projection per slice spent more
// time on the fp32 reductions of its partial outputs (about 1.9 TB/s of reduction traffic is all L2 takes) than
// on the weights.
//
// The batch-level half of the routing runs in this kernel's prologue, redundantly in every CTA, from the per-token
// Top-K the previous kernel left: routed weights summed per expert in 2^-53 fixed point (exact, order-independent),
// pool by counting ranks on (score desc, id asc), minimum-loss target and scalar per source, remap of every slot,
// rows per group. With the dynamic pool and at most 128 tokens the work list is known once the pool is: the
// producer and MMA warps start streaming then, and the epilogue warps finish the routing beside them. The CTAs
// that own a group's first slice write its execution lists (row -> token, merged weight, slot -> row); CTA 0 writes
// the routing metadata and the group table.
//
// Routing prologue, dependency wait -> pool known -> first weights multiplied -> row lists done: 64 tokens 3.2 -> 5.9 -> 12 us
// before the members-only ranking, the eight-lane target search and the token masks; 256 tokens 4.5, 19 (nothing streams
// before the lists there), 17 us. Whole call then -> now: Qwen3 shape 64 tokens, pool 16 43.4 -> 42.4 us; 256 tokens with the
// router, pool 64 192 -> 180 (dense items), pool 16 74 -> 66 (also a fourth ring stage, from the slot tables' bytes).
// Then slots four to a load, ranks on the keys' upper halves, a list of the sources outside the pool with 64 candidates per
// round trip, no integer division per slot, and the schedule ahead of the dependency wait: 256 tokens 14.5 -> 9.7 us from the
// wait to the first item (call 149 -> 146.5 us), 120 tokens with the router, pool 16 53.9 -> 52.6, 32 tokens 48.5 -> 48.1.
//
// Item sizes: full slices of 128 features; the last partial round of full items is cut into halves (s = 64) when
// that lets more SMs share it, and a trailing 64-wide slice of I is a half by itself. Single rounds: 96- or 32-wide slices.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "ptx.cuh"

namespace exfold {

namespace {

constexpr int kFThreads = 224;   // warp 0 and 6: TMA producers, warp 1: MMA issuer, warps 2-5: epilogue
constexpr int kFBK = 64;         // K elements per ring stage (one 128-byte swizzle row)
constexpr int kFBBytes = 256 * kFBK * 2;   // weight part of a stage: 128 gate rows + 128 up rows
constexpr int kFMaxStages = 16;
// Above 128 tokens a group of at most kGatherRows rows is one item whose rows are gathered from x (TMA gather4, ~60-85
// cycles of the SM's copy engine per four rows, so 64 rows fit the ~1200 cycles in which an SM's share of HBM brings a stage
// of weights); a larger group runs as one dense item per token tile that it touches, which pulls its weights through the SM
// twice. 256 tokens with the router, Qwen3 shape, pool 64 (some 32 rows per group): kernel 116 -> 96 us, call 187 -> 151 us;
// with the limit at 32 rows 161 us, at 96 152.4, at 128 152.8.
// Where one item per (group, slice) leaves SMs idle, the two dense items of a group run at the same time on those, and the
// gathers only lengthen the one: the limit falls with the square of the share of SMs that gathered items would fill. Whole
// call dense / limit of 64 / this: 32 experts of 2048 x 512, 160 tokens, pool of 8 35.3 / 41.9 / 34.8 us, pool of 32 58.7 /
// 49.9 / 50.0; 13 + 1 experts of 832 x 768, 130 tokens, pool of 4 27.9 / 30.3 / 28.0; 16 + 1 of 3648 x 1664, 130 tokens,
// pool of 8 95.3 / 102.9 / 97.9; Qwen3 shape, 130 tokens, pool of 8 45.0 / 49.4 / 42.1 (pool of 16, all SMs but a third: 62.1 /
// 52.3 / 58.8).
constexpr int kGatherRows = 64;
constexpr int kGather = 2;
constexpr int kFTmemCols = 512;
constexpr int kFMaxPairs = 2 * kMaxGroups;      // (group, token tile) pairs: B <= 256 is at most two tiles
constexpr int kFSmemLimit = 227 * 1024 - 2048;  // dynamic shared memory the kernel may ask for
static_assert(kMaxDecodeBatch <= 256, "two token tiles per group at most");

__host__ __device__ constexpr int decode_ffn_stage_bytes(int a_rows, int alt) {
    return a_rows * kFBK * 2 + (alt == 32 ? kFBBytes / 4 : kFBBytes);
}

struct Scratch {  // per-batch routing state, one copy per CTA
    long long key[kMaxExperts];        // by union member: order-preserving integer image of score_e
    unsigned acc32[3 * kMaxExperts];   // sum_i w_{i,e} in 2^-53 units, as three 21-bit limbs
    int in_union[kMaxExperts];
    int rank_of[kMaxExperts];  // pool rank or -1
    int pool[kMaxExperts];     // pool experts by rank
    int target[kMaxExperts];
    float scale[kMaxExperts];  // static pool; dynamic pool: for the metadata only
    int goff[kFMaxPairs + 2];  // exclusive prefix over (group, token tile): first compact row
    int pairs[kFMaxPairs];     // the work list's rows: group * 4 + token tile, or + kGather (before that: the union's experts)
    int P, U, n_pairs;
};
constexpr int kFScratchFixed = (int)((sizeof(Scratch) + 15) / 16 * 16);

struct Item {
    int expert, g, mt, j0, s;  // mt: token tile, or kGather: all rows of the group, gathered
};

struct Sched {  // the same in every role of a CTA
    int n_pairs, nfull, has_half, f_keep, split, total;
    int alt, n_alt;  // n_alt > 0: every item is an alt-wide slice (96 or 32), n_alt per pair (see make_sched)
    int identity;  // pair p is (group p, token tile 0): no list needed
    int ctas;      // CTAs that take work: item w belongs to CTA w % ctas
};

// Two ways to deal F full items (plus a few natural halves) over the grid, both static:
//   (a) all CTAs, the last partial round of r full items cut into 2r halves when every half finds its own SM;
//   (b) only eff = ceil(F / rounds) CTAs, each exactly `rounds` items, so that all of them finish together.
// In units of the time one SM needs for a full item alone, a phase of n SMs working at once takes z * max(1, n / c)
// for items of size z: about c = 110 SMs of this kernel saturate HBM (measured: it streams ~55 GB/s per SM, ~6 TB/s together).
// (b) wins when the remainder would leave a few SMs working alone (448 items: 112 x 4 rather than 148 x 3 + 8 halves).
__device__ __forceinline__ Sched make_sched(int n_pairs, int I, int grid, int identity, int alt) {
    Sched sc;
    sc.identity = identity;
    sc.n_pairs = n_pairs;
    sc.nfull = I / 128;
    sc.has_half = (I % 128) != 0 ? 1 : 0;
    const int F = n_pairs * sc.nfull, H = n_pairs * sc.has_half;
    const float c = 110.0f;
    const int q = F / grid, r = F % grid;
    const bool can_split = r > 0 && 2 * r + H <= grid;
    // Less than one round of full items, too many to halve: 96-wide slices when they divide I and still fit one round.
    // What an SM streams is bounded by the bytes its ring keeps in flight over the loaded HBM latency (~60 GB/s), so a
    // single round goes faster on more SMs with smaller items (16 experts x 768: 128 items of 0.75 MB, not 96 of 1 MB).
    // Few groups, so that even 32-wide slices all have an SM to themselves (decided by the host, decode_ffn_alt): those.
    sc.alt = alt;
    sc.n_alt = 0;
    if (alt == 32 || (alt == 96 && q == 0 && r > 0 && !can_split && H == 0 && n_pairs * (I / 96) <= grid && I / 96 > sc.nfull)) {
        sc.n_alt = I / alt;
        sc.split = 0;
        sc.ctas = grid;
        sc.f_keep = 0;
        sc.total = n_pairs * sc.n_alt;
        return sc;
    }
    float ta = (float)q * fmaxf(1.0f, (float)grid / c);
    if (can_split) ta += 0.5f * fmaxf(1.0f, (float)(2 * r) / c);
    else if (r > 0) ta += fmaxf(1.0f, (float)r / c);
    const int rounds = (F + grid - 1) / grid;
    const int eff = rounds > 0 ? (F + rounds - 1) / rounds : grid;
    const float tb = (float)rounds * fmaxf(1.0f, (float)eff / c);
    if (F > 0 && tb < ta) {
        sc.split = 0;
        sc.ctas = eff;
    } else {
        sc.split = can_split ? r : 0;
        sc.ctas = grid;
    }
    sc.f_keep = F - sc.split;
    sc.total = sc.f_keep + 2 * sc.split + H;
    return sc;
}

__device__ __forceinline__ Item decode_item(int w, const Sched& sc, const Scratch& s, int N) {
    Item it;
    int pair;
    if (sc.n_alt > 0) {
        pair = w / sc.n_alt;
        it.j0 = (w - pair * sc.n_alt) * sc.alt;
        it.s = sc.alt;
    } else if (w < sc.f_keep) {
        pair = w / sc.nfull;
        it.j0 = (w - pair * sc.nfull) * 128;
        it.s = 128;
    } else if (w < sc.f_keep + 2 * sc.split) {
        const int u = w - sc.f_keep, f = sc.f_keep + (u >> 1);
        pair = f / sc.nfull;
        it.j0 = (f - pair * sc.nfull) * 128 + (u & 1) * 64;
        it.s = 64;
    } else {
        pair = w - sc.f_keep - 2 * sc.split;
        it.j0 = sc.nfull * 128;
        it.s = 64;
    }
    const int code = sc.identity ? pair * 4 : s.pairs[pair];
    it.g = code >> 2;
    it.mt = code & 3;
    it.expert = it.g < s.P ? s.pool[it.g] : N;  // group P is the shared expert
    return it;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
}

// NMT: token tiles of 128 (one kernel for both: 64 tokens 0.5 % slower, from the gathers' code)
template <int NMT>
__global__ void __launch_bounds__(kFThreads, 1) decode_ffn_kernel(const __grid_constant__ DecodeFfnParams p) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kFMaxStages];
    __shared__ __align__(8) uint64_t empty_bar[kFMaxStages];
    __shared__ __align__(8) uint64_t tfull_bar[2];
    __shared__ __align__(8) uint64_t tempty_bar[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ Sched sched_s;  // for the expected number of list entries
    __shared__ __align__(16) int s_rows[2][NMT == 2 ? kGatherRows : 4];  // per producer: the tokens of a gathered item

    unsigned char* tiles =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int stages = p.stages;
    const int a_bytes = p.a_rows * kFBK * 2;
    const int stage_bytes = decode_ffn_stage_bytes(p.a_rows, p.alt);
    Scratch& sc = *reinterpret_cast<Scratch*>(tiles + p.scratch_off);
    // two bytes per slot (its routed expert in the upper, the expert that runs it in the lower one) and, by pool rank, the
    // tokens each group serves as bit masks: what is not spent here is ring (256 tokens x 8 slots: 20 KB with ids and weights
    // as words, one stage of four)
    unsigned short* slots = reinterpret_cast<unsigned short*>(tiles + p.scratch_off + kFScratchFixed);
    uint32_t* tmask = reinterpret_cast<uint32_t*>(tiles + p.scratch_off + kFScratchFixed + align16((size_t)p.B * p.K * 2));

    // ---- set-up that does not depend on the previous kernel: overlaps its tail under programmatic launch
    if (threadIdx.x == 0) {
        ptx::prefetch_tmap(&p.tm_x);
        if (NMT == 2) ptx::prefetch_tmap(&p.tm_xg);
        ptx::prefetch_tmap(&p.tm_wg);
        ptx::prefetch_tmap(&p.tm_wu);
        if (p.alt) {
            ptx::prefetch_tmap(&p.tm_wg_alt);
            ptx::prefetch_tmap(&p.tm_wu_alt);
        }
        for (int s = 0; s < kFMaxStages; ++s) {
            ptx::mbar_init(&full_bar[s], 1);
            ptx::mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(&tfull_bar[s], 1);
            ptx::mbar_init(&tempty_bar[s], 4);
        }
        abort_s = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(&tmem_base_s, kFTmemCols);
        ptx::tmem_relinquish();
    }
    const int B = p.B, N = p.N, K = p.K, BK = B * K;
    const bool is_static = p.st_pool != nullptr;
    const int nmt = NMT == 2 ? 2 : (B + 127) >> 7;  // 1 as a run-time value: as a constant 0.4 % slower (64 tokens)
    // With the dynamic pool and one token tile every pool expert has a row (it is in the union), so the work list
    // is known as soon as the pool is: the producer and MMA warps leave for their roles then, and the epilogue
    // warps finish the routing (targets, remap, row lists, metadata) while the first weights stream in.
    const bool early = !is_static && nmt == 1;
    for (int e = threadIdx.x; e < N; e += kFThreads) {
        sc.acc32[3 * e] = sc.acc32[3 * e + 1] = sc.acc32[3 * e + 2] = 0u;
        sc.in_union[e] = 0;
        sc.rank_of[e] = -1;
    }
    const int W = nmt * 4;  // mask words per group
    for (int i = threadIdx.x; i < (N + 1) * W; i += kFThreads) tmask[i] = 0u;
    if (!is_static) {  // the tables into L2 while the previous kernel runs (only a hint: they are read after the wait)
        if (warp == 5 && lane * 32 < N) ptx::prefetch_l2(p.h + lane * 32);
        const size_t n_el = (size_t)N * N, lines = (n_el * 4 + 127) / 128;
        for (size_t i = (size_t)blockIdx.x * kFThreads + threadIdx.x; i < lines; i += (size_t)gridDim.x * kFThreads) {
            const size_t el = i * 32 < n_el ? i * 32 : n_el - 1;
            ptx::prefetch_l2(p.L + el);
            ptx::prefetch_l2(p.S + el);
        }
    }
    // The schedule of the list that is expected (every group one entry, the pool full): its divisions take a microsecond
    if (threadIdx.x == 96) sched_s = make_sched(min(p.M, min(N, BK)) + (p.n_shared ? 1 : 0), p.I, (int)gridDim.x, early ? 1 : 0, p.alt);
    ptx::tc_fence_before();
    __syncthreads();
    grid_dep_wait();  // the per-token Top-K of the previous kernel; the previous call's readers of the workspace

    // ---- routing, batch level (Eq. 11, 12, 14), the same in every CTA
    // (four slots to a load, a thread's loads first: one L2 round trip for 256 tokens x 8)
    auto add_slot = [&](int id, double wv) {
        // The routed weight in 2^-53 fixed point, added as three 21-bit limbs with 32-bit integer atomics (at most 256
        // addends per expert, so no limb overflows): exact, and independent of the order of arrival.
        const unsigned long long fx = (unsigned long long)(wv * 9007199254740992.0);
        atomicAdd(&sc.acc32[3 * id], (unsigned)(fx & 0x1FFFFFull));
        atomicAdd(&sc.acc32[3 * id + 1], (unsigned)((fx >> 21) & 0x1FFFFFull));
        atomicAdd(&sc.acc32[3 * id + 2], (unsigned)(fx >> 42));
        sc.in_union[id] = 1;
    };
    // The norms that this thread scores below, in the slots' round trip. Not before the wait: the caller may have written
    // the table on this stream right before the call.
    static_assert(kMaxExperts <= 2 * kFThreads, "two norms per thread");
    float h_e[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int e = threadIdx.x + u * kFThreads;
        h_e[u] = !is_static && e < N ? __ldg(p.h + e) : 0.f;
    }
    const int BK4 = BK >> 2;
    for (int s0 = threadIdx.x; s0 < BK4; s0 += kFThreads * 3) {
        int4 id[3];
        double2 wv[3][2];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const int s = s0 + u * kFThreads;
            if (s >= BK4) break;
            id[u] = reinterpret_cast<const int4*>(p.ids)[s];
            if (!is_static) {
                wv[u][0] = reinterpret_cast<const double2*>(p.w64)[2 * s];
                wv[u][1] = reinterpret_cast<const double2*>(p.w64)[2 * s + 1];
            }
        }
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const int s = s0 + u * kFThreads;
            if (s >= BK4) break;
            reinterpret_cast<uint2*>(slots)[s] = make_uint2((unsigned)id[u].x << 8 | (unsigned)id[u].y << 24,
                                                            (unsigned)id[u].z << 8 | (unsigned)id[u].w << 24);
            if (!is_static) {
                add_slot(id[u].x, wv[u][0].x);
                add_slot(id[u].y, wv[u][0].y);
                add_slot(id[u].z, wv[u][1].x);
                add_slot(id[u].w, wv[u][1].y);
            }
        }
    }
    if (threadIdx.x < (BK & 3)) {
        const int s = BK4 * 4 + threadIdx.x;
        const int id = p.ids[s];
        slots[s] = (unsigned short)(id << 8);
        if (!is_static) add_slot(id, p.w64[s]);
    }
    __syncthreads();
    if (is_static) {
        for (int e = threadIdx.x; e < N; e += kFThreads) {
            sc.target[e] = p.st_target[e];
            sc.scale[e] = p.st_scale[e];
        }
        for (int j = threadIdx.x; j < p.M; j += kFThreads) {
            const int e = p.st_pool[j];
            sc.pool[j] = e;
            sc.rank_of[e] = j;
        }
        if (threadIdx.x == 0) sc.P = p.M;
        __syncthreads();
    } else {
        // Eq. 11: score_e = h_e * sum_i w_{i,e} in double, for the union's experts (in ascending order), ranked through an
        // order-preserving integer key
        const int n_chunks = (N + 31) >> 5;
        int* member = sc.pairs;
        int* khi = reinterpret_cast<int*>(sc.scale);  // the keys' upper halves
        int U = 0;
        for (int c = 0; c < n_chunks; ++c) {
            const int e = c * 32 + lane;
            const bool in = e < N && sc.in_union[e];
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (in && c % (kFThreads / 32) == warp) {
                const int pos = U + __popc(m & ((1u << lane) - 1u));
                const unsigned long long acc = (unsigned long long)sc.acc32[3 * e] +
                                               ((unsigned long long)sc.acc32[3 * e + 1] << 21) +
                                               ((unsigned long long)sc.acc32[3 * e + 2] << 42);
                const long long key =
                    score_order_key((double)acc * (1.0 / 9007199254740992.0) * (double)(c < kFThreads / 32 ? h_e[0] : h_e[1]));
                member[pos] = e;
                sc.key[pos] = key;
                khi[pos] = (int)(key >> 32);
            }
            U += __popc(m);
        }
        if (threadIdx.x < (-U & 3)) khi[U + threadIdx.x] = INT_MIN;
        __syncthreads();
        // pool = best min(M, |U|) experts of the union by (score desc, id asc): rank by counting, several threads per
        // member, on the keys' upper halves four to a load; only a member whose half another one shares counts whole keys.
        // A member outside the pool is a source; rank - M is its place in the list.
        int lanes = 32;
        while (lanes > 1 && U * lanes > kFThreads) lanes >>= 1;
        const int sub = threadIdx.x & (lanes - 1);
        int* src = reinterpret_cast<int*>(sc.acc32);
        for (int i0 = 0; i0 < U; i0 += kFThreads / lanes) {
            const int i = i0 + (int)threadIdx.x / lanes;
            int better = 0, same = 0;
            if (i < U) {
                const int ki = khi[i];
#pragma unroll 4
                for (int o = sub; 4 * o < U; o += lanes) {
                    const int4 ko = reinterpret_cast<const int4*>(khi)[o];
                    better += (ko.x > ki) + (ko.y > ki) + (ko.z > ki) + (ko.w > ki);
                    same += (ko.x == ki) + (ko.y == ki) + (ko.z == ki) + (ko.w == ki);
                }
            }
            for (int o = lanes >> 1; o > 0; o >>= 1) {
                better += __shfl_xor_sync(0xffffffffu, better, o);
                same += __shfl_xor_sync(0xffffffffu, same, o);
            }
            if (i < U && sub == 0) {
                if (same > 1) {
                    const long long ki = sc.key[i];
                    better = 0;
                    for (int o = 0; o < U; ++o) {
                        const long long ko = sc.key[o];
                        better += (ko > ki || (ko == ki && o < i)) ? 1 : 0;  // members ascend: position order is id order
                    }
                }
                if (better < p.M) {
                    sc.rank_of[member[i]] = better;
                    sc.pool[better] = member[i];
                } else {
                    src[better - p.M] = member[i];
                }
            }
        }
        if (threadIdx.x == 0) {
            sc.P = U < p.M ? U : p.M;
            sc.U = U;
        }
        __syncthreads();
    }
    const bool mine = !early || (warp >= 2 && warp <= 5);  // threads that run the rest of the routing
    const int tid = early ? (int)threadIdx.x - 64 : (int)threadIdx.x, nth = early ? 128 : kFThreads;
    auto sync_group = [&]() {
        if (early) asm volatile("bar.sync 1, 128;" ::: "memory");
        else __syncthreads();
    };
    if (mine) {
        const int P = sc.P, G = P + (p.n_shared ? 1 : 0);
        const bool meta = p.pool_ids != nullptr && blockIdx.x == 0;  // the caller asked for the routing metadata
        if (!is_static) {
            // Eq. 12: a source in the pool keeps itself; any other takes its minimum-loss pool expert (ties -> lower
            // id; a NaN loss is never smaller, but the best-ranked expert's is where the search starts and stays).
            // Every CTA searches every source, so the sectors read count as much as the round trips: losses only (the chosen
            // target's scalar is read where a row's weight is made), and two, four or eight lanes per source, so that a lane
            // has at most eight candidates up to a pool of 64. 256 experts of 2048 x 512, pool of 16, 64 / 128 / 160 tokens:
            // eight lanes with losses and scalars 43.1 / 48.5 / 61.7 us per call, a thread per source 44.1 / 47.5 / 59.5, this
            // 39.3 / 44.2 / 58.8. Qwen3 shape, pool of 16, 256 tokens: 71.2, 73.8, 69.8. Only sources that occur in the
            // batch matter for the execution; the metadata has the whole table.
            for (int j = tid; j < P; j += nth) {
                sc.target[sc.pool[j]] = sc.pool[j];
                if (meta) sc.scale[sc.pool[j]] = 1.0f;
            }
            const int* src = reinterpret_cast<const int*>(sc.acc32);
            const int lg = P > 32 ? 3 : (P > 16 ? 2 : 1), lanes = 1 << lg, sub = tid & (lanes - 1);
            const int n_src = meta ? N : sc.U - P;
            for (int i0 = 0; i0 < n_src; i0 += nth >> lg) {
                const int i = i0 + (tid >> lg);
                const int s = i < n_src ? (meta ? i : src[i]) : -1;
                float bl = INFINITY, l[8];
                l[0] = 0.f;
                int bt = 0x7fffffff;
                if (s >= 0 && sc.rank_of[s] < 0) {
                    for (int j0 = sub + (((P - 1) >> (lg + 3)) << (lg + 3)); j0 >= 0; j0 -= 8 * lanes) {  // the best-ranked one last
                        int tt[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            tt[u] = j0 + (u << lg) < P ? sc.pool[j0 + (u << lg)] : -1;
                            l[u] = tt[u] >= 0 ? __ldg(p.L + (size_t)s * N + tt[u]) : 0.f;
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (tt[u] >= 0 && (l[u] < bl || (l[u] == bl && tt[u] < bt))) {
                                bl = l[u];
                                bt = tt[u];
                            }
                    }
                } else {
                    bt = s;  // every lane of the source alike
                }
                for (int o = lanes >> 1; o > 0; o >>= 1) {
                    const float ol = __shfl_xor_sync(0xffffffffu, bl, o);
                    const int ot = __shfl_xor_sync(0xffffffffu, bt, o);
                    if (ol < bl || (ol == bl && ot < bt)) {
                        bl = ol;
                        bt = ot;
                    }
                }
                if (s >= 0 && sub == 0) {
                    const bool stays = isnan(l[0]);
                    if (stays) bt = sc.pool[0];
                    sc.target[s] = bt;
                    if (meta) sc.scale[s] = bt == s ? 1.0f : __ldg(p.S + (size_t)s * N + bt);
                }
            }
            sync_group();
        }
        // Eq. 14: every slot in place; [B][K] layout kept. A token counts once per distinct target: a bit of its mask
        const unsigned inv_k = ((1u << 18) + K - 1) / K;  // s / K = s * inv_k >> 18: s * K < 2^17
        for (int s0 = tid; s0 < BK; s0 += 4 * nth) {
            int e[4], t[4], r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) e[u] = s0 + u * nth < BK ? slots[s0 + u * nth] >> 8 : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) t[u] = e[u] >= 0 ? sc.target[e[u]] : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) r[u] = e[u] >= 0 ? sc.rank_of[t[u]] : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e[u] < 0) continue;
                const int s = s0 + u * nth, i = (int)(((unsigned)s * inv_k) >> 18);
                slots[s] = (unsigned short)(e[u] << 8 | t[u]);
                atomicOr(&tmask[r[u] * W + (i >> 5)], 1u << (i & 31));
                if (meta) {
                    p.out_ids[s] = t[u];
                    p.out_w[s] = (float)(p.w64[s] * (double)sc.scale[e[u]]);
                }
            }
        }
        if (p.n_shared && tid < W) {
            const int left = B - tid * 32;
            tmask[P * W + tid] = left >= 32 ? 0xffffffffu : (left > 0 ? (1u << left) - 1u : 0u);
        }
        if (meta) {
            for (int e = tid; e < N; e += nth) {
                p.target[e] = sc.target[e];
                p.scale[e] = sc.scale[e];
                p.pool_ids[e] = e < P ? sc.pool[e] : -1;
            }
            if (tid < 8) {
                uint32_t m = 0;
                for (int b = 0; b < 32; ++b) {
                    const int e = tid * 32 + b;
                    if (e < N && sc.rank_of[e] >= 0) m |= 1u << b;
                }
                p.pool_mask[tid] = m;
            }
            if (tid == 0) *p.pool_size = P;
        }
        sync_group();
        // exclusive prefix over (group, tile) = first compact row of each; the work list's rows
        if (tid < 32) {
            const float fill = fminf(1.0f, (float)(G * ((p.I + 127) / 128)) / (float)gridDim.x);
            const int gather_limit = (int)(kGatherRows * fill * fill);
            int carry = 0, n = 0;
            for (int g0 = 0; g0 < G; g0 += 32) {
                const int g = g0 + tid;
                int v[2] = {0, 0};
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
                    if (g < G && mt < nmt) {
                        const uint4 m4 = *reinterpret_cast<const uint4*>(tmask + g * W + mt * 4);
                        v[mt] = __popc(m4.x) + __popc(m4.y) + __popc(m4.z) + __popc(m4.w);
                    }
                const int rows = v[0] + v[1];
                const bool gather = nmt == 2 && rows > 0 && rows <= gather_limit;
                const int entries = gather ? 1 : (v[0] > 0) + (v[1] > 0);
                int incl = rows;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, incl, o);
                    if (tid >= o) incl += u;
                }
                const unsigned one = __ballot_sync(0xffffffffu, entries > 0), two = __ballot_sync(0xffffffffu, entries > 1);
                const unsigned below = (1u << tid) - 1u;
                if (g < G) {
                    sc.goff[2 * g] = carry + incl - rows;
                    sc.goff[2 * g + 1] = carry + incl - v[1];
                    int q = n + __popc(one & below) + __popc(two & below);
                    if (gather) {
                        sc.pairs[q] = g * 4 + kGather;
                    } else {
                        if (v[0] > 0) sc.pairs[q++] = g * 4;
                        if (v[1] > 0) sc.pairs[q] = g * 4 + 1;
                    }
                }
                carry += __shfl_sync(0xffffffffu, incl, 31);
                n += __popc(one) + __popc(two);
            }
            if (tid == 0) {
                sc.goff[2 * G] = carry;
                sc.n_pairs = n;
            }
        }
        sync_group();
        if (blockIdx.x == 0) {  // group table of the down-projection kernel
            for (int g = tid; g <= G; g += nth) {
                p.grp_off[g] = sc.goff[2 * g];
                if (g < G) p.grp_expert[g] = g < P ? sc.pool[g] : N;
            }
            if (tid < 32) {
                int carry = 0;
                for (int g0 = 0; g0 < G; g0 += 32) {
                    const int g = g0 + tid;
                    const int v = g < G ? (sc.goff[2 * g + 2] - sc.goff[2 * g] + kTileM - 1) / kTileM : 0;
                    int incl = v;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int u = __shfl_up_sync(0xffffffffu, incl, o);
                        if (tid >= o) incl += u;
                    }
                    if (g < G) p.grp_tiles[g] = carry + incl - v;
                    carry += __shfl_sync(0xffffffffu, incl, 31);
                }
                if (tid == 0) {
                    p.grp_tiles[G] = carry;
                    p.n_groups[0] = G;
                    p.n_groups[1] = sc.goff[2 * G];
                    p.n_groups[2] = sc.goff[2 * P];  // first row of the shared expert's group
                }
            }
        }
    }
    if (!early) __syncthreads();
    ptx::tc_fence_after();

    const int n_list = early ? sc.P + (p.n_shared ? 1 : 0) : sc.n_pairs;
    Sched sched = sched_s;
    if (n_list != sched.n_pairs) sched = make_sched(n_list, p.I, (int)gridDim.x, early ? 1 : 0, p.alt);
    const int total = sched.total;
    const int w_begin = (int)blockIdx.x < sched.ctas ? (int)blockIdx.x : total, w_stride = sched.ctas;
    const uint32_t tmem_base = tmem_base_s;
    const int nkb = p.d / kFBK;
    volatile int* abort_flag = &abort_s;

    if (warp == 0 || warp == 6) {
        // ------------------------------------------------ TMA producers (k-block c belongs to producer c % 2)
        const int me = warp == 0 ? 0 : 1;
        int stage = 0, phase = 0, turn = 0;
        int ok = 1;
        if (NMT == 2 || ptx::elect_one()) {  // a whole warp where rows are gathered
            for (int w = w_begin; w < total && ok; w += w_stride) {
                const Item it = decode_item(w, sched, sc, N);
                int n4 = 0;  // groups of four rows to gather
                if (NMT == 2 && it.mt == kGather) {
                    int n = 0;
                    __syncwarp();
                    for (int q = 0; q < W; ++q) {
                        const uint32_t m = tmask[it.g * W + q];
                        if ((m >> lane) & 1u) s_rows[me][n + __popc(m & ((1u << lane) - 1u))] = q * 32 + lane;
                        n += __popc(m);
                    }
                    __syncwarp();
                    n4 = (n + 3) >> 2;
                    if (lane < 4 * n4 - n) s_rows[me][n + lane] = s_rows[me][0];  // the last four filled up
                    __syncwarp();
                }
                if (NMT == 1 || ptx::elect_one()) {
                    const int xrow = NMT == 2 && it.mt == 1 ? 128 : 0;
                    const int wrow = it.expert * p.I + it.j0;
                    const uint32_t tx = (uint32_t)((n4 > 0 ? n4 * 512 : a_bytes) + 2 * it.s * kFBK * 2);
                    for (int kb = 0; kb < nkb; ++kb) {
                        if (turn == me) {
                            if (!ptx::mbar_wait(&empty_bar[stage], phase ^ 1, abort_flag, p.status, 1)) {
                                ok = 0;
                                break;
                            }
                            unsigned char* a_dst = tiles + stage * stage_bytes;
                            unsigned char* b_dst = a_dst + a_bytes;
                            ptx::mbar_expect_tx(&full_bar[stage], tx);
                            if (n4 == 0) ptx::tma_load_2d(a_dst, &p.tm_x, &full_bar[stage], kb * kFBK, xrow);
                            if (it.s == 128) {
                                ptx::tma_load_2d(b_dst, &p.tm_wg, &full_bar[stage], kb * kFBK, wrow);
                                ptx::tma_load_2d(b_dst + 128 * kFBK * 2, &p.tm_wu, &full_bar[stage], kb * kFBK, wrow);
                            } else if (it.s == 64) {
                                ptx::tma_load_2d(b_dst, &p.tm_wg64, &full_bar[stage], kb * kFBK, wrow);
                                ptx::tma_load_2d(b_dst + 64 * kFBK * 2, &p.tm_wu64, &full_bar[stage], kb * kFBK, wrow);
                            } else {
                                ptx::tma_load_2d(b_dst, &p.tm_wg_alt, &full_bar[stage], kb * kFBK, wrow);
                                ptx::tma_load_2d(b_dst + it.s * kFBK * 2, &p.tm_wu_alt, &full_bar[stage], kb * kFBK, wrow);
                            }
                            for (int q = 0; q < n4; ++q) {
                                const int4 r = *reinterpret_cast<const int4*>(&s_rows[me][4 * q]);
                                ptx::tma_gather4(a_dst + q * 512, &p.tm_xg, &full_bar[stage], kb * kFBK, r.x, r.y, r.z, r.w);
                            }
                        }
                        turn ^= 1;
                        if (++stage == stages) {
                            stage = 0;
                            phase ^= 1;
                        }
                    }
                }
                if (NMT == 2) ok = __all_sync(0xffffffffu, ok);  // (whichever lane was elected and gave up)
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (ptx::elect_one()) {
            const uint32_t lo0 = (ptx::smem_u32(tiles) & 0x3FFFFu) >> 4;
            const uint32_t lo_step = (uint32_t)stage_bytes >> 4, lo_b = (uint32_t)a_bytes >> 4;
            const uint32_t desc_hi32 = (uint32_t)(ptx::make_kmajor_sw128_desc(0) >> 32);
            constexpr uint32_t idesc256 = ptx::make_idesc_bf16(128, 256), idesc128 = ptx::make_idesc_bf16(128, 128),
                               idesc192 = ptx::make_idesc_bf16(128, 192), idesc64 = ptx::make_idesc_bf16(128, 64);
            int stage = 0, phase = 0, item = 0;
            uint32_t a_lo = lo0;
            bool ok = true, ready = false;
            for (int w = w_begin; w < total && ok; w += w_stride, ++item) {
                const Item it = decode_item(w, sched, sc, N);
                const int as = item & 1, aphase = (item >> 1) & 1;
                if (!ptx::mbar_wait(&tempty_bar[as], aphase ^ 1, abort_flag, p.status, 2)) break;
                ptx::tc_fence_after();
                const uint32_t d_tmem = tmem_base + as * 256;
                const uint32_t idesc = it.s == 128 ? idesc256 : (it.s == 64 ? idesc128 : (it.s == 96 ? idesc192 : idesc64));
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!ready && !ptx::mbar_wait(&full_bar[stage], phase, abort_flag, p.status, 3)) {
                        ok = false;
                        break;
                    }
                    const int ns = stage + 1 == stages ? 0 : stage + 1;
                    const int nphase = ns == 0 ? phase ^ 1 : phase;
                    ready = ptx::umma_kblock_bf16(d_tmem, a_lo, a_lo + lo_b, desc_hi32, idesc, kb > 0 ? 1u : 0u,
                                                  &empty_bar[stage], &full_bar[ns], nphase);
                    a_lo = ns == 0 ? lo0 : a_lo + lo_step;
                    stage = ns;
                    phase = nphase;
                }
                if (ok) ptx::umma_commit(&tfull_bar[as]);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue warps (TMEM lane quadrant = warp % 4)
        const int q = warp & 3;
        const int row = q * 32 + lane;
        int item = 0;
        for (int w = w_begin; w < total; w += w_stride, ++item) {
            const Item it = decode_item(w, sched, sc, N);
            const int as = item & 1, aphase = (item >> 1) & 1;
            const bool shared_grp = it.g >= sc.P;
            bool valid;
            unsigned mq;  // this quadrant's rows that are stored
            int tok;
            int64_t rowpos;
            if (NMT == 2 && it.mt == kGather) {  // the group's rows in order
                valid = row < sc.goff[2 * it.g + 2] - sc.goff[2 * it.g];
                mq = __ballot_sync(0xffffffffu, valid);
                rowpos = sc.goff[2 * it.g] + row;
                tok = 0;
                if (it.j0 == 0 && valid) {  // the row-th token of the mask
                    int left = row, q8 = 0;
                    uint32_t m = tmask[it.g * W];
                    while (left >= __popc(m)) {
                        left -= __popc(m);
                        m = tmask[it.g * W + ++q8];
                    }
                    tok = q8 * 32 + (int)__fns(m, 0, left + 1);
                }
            } else {
                // Which tokens of the tile does this expert serve? All four quadrants, so that a warp knows how many rows
                // come before its own
                const uint4 m4 = *reinterpret_cast<const uint4*>(tmask + it.g * W + it.mt * 4);
                const unsigned m[4] = {m4.x, m4.y, m4.z, m4.w};
                int before = 0;
#pragma unroll
                for (int qq = 0; qq < 4; ++qq)
                    if (qq < q) before += __popc(m[qq]);
                mq = q == 0 ? m[0] : (q == 1 ? m[1] : (q == 2 ? m[2] : m[3]));
                valid = (mq >> lane) & 1u;
                tok = it.mt * 128 + row;
                rowpos = sc.goff[it.g * 2 + it.mt] + before + __popc(mq & ((1u << lane) - 1u));
            }
            if (it.j0 == 0 && valid) {
                // this CTA owns the group's first slice: it writes the group's rows of the execution lists
                float cw = 1.0f;
                if (!shared_grp) {
                    bool has = false;
                    for (int k = 0; k < K; ++k) {
                        const int s = tok * K + k;
                        const int id = slots[s] >> 8;
                        if ((slots[s] & 255) != it.expert) continue;  // duplicates merged, weights summed in slot order
                        const float scl = is_static ? sc.scale[id] : (id == it.expert ? 1.0f : __ldg(p.S + (size_t)id * N + it.expert));
                        const float wv = (float)(p.w64[s] * (double)scl);
                        cw = has ? __fadd_rn(cw, wv) : wv;
                        p.slot_row[s] = has ? -1 : (int32_t)rowpos;
                        has = true;
                    }
                }
                p.row_tok[rowpos] = tok;
                p.row_w[rowpos] = cw;
            }
            int ok = 1;
            if (lane == 0) ok = ptx::mbar_wait(&tfull_bar[as], aphase, abort_flag, p.status, 4) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            ptx::tc_fence_after();
            if (mq != 0u) {  // warp-uniform: some row of this quadrant is stored
                const uint32_t taddr = tmem_base + as * 256 + ((uint32_t)(q * 32) << 16);
                const int nch = it.s / 32;
#pragma unroll 1
                for (int c = 0; c < nch; ++c) {
                    uint32_t gv[32], uv[32];
                    ptx::tmem_ld32(taddr + c * 32, gv);
                    ptx::tmem_ld32(taddr + it.s + c * 32, uv);
                    ptx::tmem_ld_wait();
                    if (valid) {
                        uint32_t pk[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float g0 = __uint_as_float(gv[2 * j]), g1 = __uint_as_float(gv[2 * j + 1]);
                            const float u0 = __uint_as_float(uv[2 * j]), u1 = __uint_as_float(uv[2 * j + 1]);
                            const float h0 = __fdividef(g0, 1.0f + __expf(-g0)) * u0;
                            const float h1 = __fdividef(g1, 1.0f + __expf(-g1)) * u1;
                            pk[j] = pack_bf16x2(h0, h1);
                        }
                        __nv_bfloat16* dst = p.H + rowpos * p.I + it.j0 + c * 32;
                        ptx::st_global32(dst, pk);
                        ptx::st_global32(dst + 16, pk + 8);
                    }
                }
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&tempty_bar[as]);
        }
    }

    // ------------------------------------------------ teardown
    if (threadIdx.x == 64) grid_dep_launch();  // after the epilogue loop: the successor's CTAs would only compete
    ptx::tc_fence_before();
    __syncthreads();
    if (abort_s) __nanosleep(100000);  // let any copy still in flight land before shared memory is released
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kFTmemCols);
    }
}

}  // namespace

// Width of the slices beside 128 and 64 that a call may use (make_sched). 32 where every (group, 32 features) of the largest
// pool has an SM to itself: a group of I = 768 then streams on 24 SMs, not on 12 with halves.
// Whole call without / with: Qwen3 shape 16 tokens, pool 4 28.9 / 28.2 us, 128 tokens, pool 2 31.1 / 30.0, 200 tokens, pool 3
// 37.5 / 35.9; GLM shape 100 tokens, pool 1 50.5 / 47.3.
int decode_ffn_alt(int B, int max_groups, int I, int sms) {
    if (I % 32 == 0 && (int64_t)((B + 127) / 128) * max_groups * (I / 32) <= std::min(sms, kMaxCtas)) return 32;
    return I % 96 == 0 ? 96 : 0;
}

// Shared-memory plan: [ring: stages x (token box + 32 KB of weights, 8 KB when all slices are 32 wide)][routing state][slots,
// token masks]
size_t decode_ffn_smem_plan(int B, int K, int N, int alt, int* stages, int* scratch_off, int* a_rows) {
    const int ar = std::min(kTileM, (B + 31) / 32 * 32);
    const int stage_bytes = decode_ffn_stage_bytes(ar, alt);
    const int mask_words = (B + 127) / 128 * 4;
    const size_t scratch = kFScratchFixed + align16((size_t)B * K * 2) + (size_t)(N + 1) * mask_words * 4;
    const long avail = (long)kFSmemLimit - 1024 - (long)scratch;
    int st = (int)(avail / stage_bytes);
    if (st > kFMaxStages) st = kFMaxStages;
    *stages = st;
    *a_rows = ar;
    *scratch_off = st * stage_bytes;
    return 1024 + (size_t)st * stage_bytes + scratch;
}

cudaError_t launch_decode_ffn(const DecodeFfnParams& p, int sms, cudaStream_t s) {
    int stages, scratch_off, a_rows;
    const size_t smem = decode_ffn_smem_plan(p.B, p.K, p.N, p.alt, &stages, &scratch_off, &a_rows);
    if (stages < 2 || stages != p.stages || scratch_off != p.scratch_off) return cudaErrorInvalidValue;
    auto kernel = p.B > 128 ? decode_ffn_kernel<2> : decode_ffn_kernel<1>;
    cudaError_t err = ensure_smem(kernel, smem);
    if (err != cudaSuccess) return err;
    return launch_pdl(kernel, std::min(sms, kMaxCtas), kFThreads, smem, s, p);
}

}  // namespace exfold
