// Expert GEMMs of prefill and calibration on CTA pairs, whole 256-row tiles and ragged remainders in one pass.
//
// A group of r rows is r / 256 whole items and one ragged item of the r % 256 rows left (a whole one of masked rows above
// kRaggedMax = 224 of them, which take as long). Both kinds stage at most 32 KB per
// CTA and k-block (16 KB of weight rows, up to 16 KB of token rows) and differ in which operand is which:
//
//   whole    A = 256 token rows (128 per CTA), B = 256 weight rows: accumulator lane = token row, column = feature.
//   ragged   A = 256 weight rows (128 per CTA), B = the tokens, N = their number rounded up to 32 (half of them staged
//            by each CTA): accumulator lane = feature, column = token. The tensor pipe takes N / 256 of a whole item's time
//            (N / 2 cycles per K = 16 step, measured for N = 32 ... 256) and the stage only the tokens there are; as a row
//            tile of 128 or 256 rows the remainder would be computed and loaded in full, mostly for nothing.
//
// GEMM-1's ragged items: a CTA takes 64 features, gate rows in lanes 0-63 and up rows in lanes 64-127, so the two halves of a
// feature lie in different warps; warps q and q + 2 exchange half of their tokens each through shared memory.
//
// The items of a group that share a weight tile are neighbours in the work order, whole ones and the ragged one, so a weight
// tile crosses HBM once. Their times differ, so the items are dealt dynamically: a warp of the leader draws the next
// index from a counter in memory, decodes it and puts it into a ring of slots in both CTAs' shared memory.
//
// What bounds it: an SM takes in 64 bytes per cycle, which a whole item needs (32 KB per 512 cycles), so whole items run at
// 507-546 cycles per k-block; ragged items of 50 tokens at 530-570 where their weights come from memory. Whole prefill call on
// whole pairs of 128-row tiles and odd tiles in two passes side by side / this: GLM shape 16384 tokens 2576 / 2423 us, Mixtral shape
// 4096 tokens 1271 / 1187, Qwen3 shape 8192 tokens 400 / 381.
//
// Roles per CTA: warps 0 and 7 TMA producers (k-blocks dealt in turn; four of them are no faster: a k-block then takes each
// 1500 instead of 750 cycles), warp 1 MMA issuer (leader), warps 2-5 epilogue, warp 6 item scheduler (leader) or, in the
// peer, the return of its slots. Every wait is bounded.
#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"

namespace exfold {

namespace {

constexpr int kXBK = kGemmBK;
constexpr int kXWBytes = 128 * kXBK * 2;  // 16 KB: a CTA's weight rows of a k-block
constexpr int kXRing = 6 * 2 * kXWBytes;  // six k-blocks of a whole item
constexpr int kXBars = 16;                // barriers of the ring: more than the k-blocks in flight (ten of the smallest fit)
constexpr int kXOutBytes = 6144 + 128;  // per epilogue warp: exchange 2 x 2 KB and staging 2 KB, or staging 4 KB; 32 weights
constexpr int kXSmem = kXRing + 4 * kXOutBytes + 1024;
constexpr int kXProducers = 2;
constexpr int kXThreads = 192 + 32 * kXProducers;
constexpr int kXTmemCols = 512;
constexpr int kXSlots = 3;

struct MixItem {
    int row0, rows, n_idx, g;  // rows: 0 = no more items
    bool ragged;
};

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
}

// The operand ring is a circular buffer of bytes: a k-block takes what its item stages (18 KB for 32 tokens, 32 KB for a whole
// item), so that small items have more k-blocks in flight (a stage comes back ~2700 cycles after the MMAs that used it). All
// roles place the k-blocks alike: in order, none across the end, those of whole items at multiples of their size.
__device__ __forceinline__ int ring_start(int pos, bool ragged) {
    if (ragged) return pos;
    const int up = (pos + 2 * kXWBytes - 1) / (2 * kXWBytes) * (2 * kXWBytes);
    return up == kXRing ? 0 : up;
}
__device__ __forceinline__ int token_rows(int rows, bool ragged) { return ragged ? (rows + 31) / 32 * 16 : kTileM; }  // per CTA

// MODE 0: gate/up + SwiGLU -> H; MODE 1: down projection -> weighted bf16 rows (y or the per-route buffer) or fp32 rows
template <int MODE>
__global__ void __launch_bounds__(kXThreads, 1) grouped_gemm_mixed_kernel(const __grid_constant__ MixedGemmParams p) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kXBars];     // used in the leader
    __shared__ __align__(8) uint64_t empty_bar[kXBars];    // one per CTA, released by the leader's commits
    __shared__ __align__(8) uint64_t tfull_bar[2];         // one per CTA
    __shared__ __align__(8) uint64_t tempty_bar[2];        // used in the leader: 8 epilogue warps of the pair
    __shared__ __align__(8) uint64_t ifull_bar[kXSlots];   // one per CTA
    __shared__ __align__(8) uint64_t iempty_bar[kXSlots];  // used in the leader: the peer's slot is free
    __shared__ __align__(8) uint64_t iread_bar[kXSlots];   // one per CTA: its producers and epilogue warps have read the item
    __shared__ __align__(16) int4 s_item[kXSlots];
    __shared__ uint32_t s_at[kXProducers][kXBars];  // per producer: running start of each k-block in flight
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, fail_s[2];
    __shared__ int s_off[kMaxGroups + 1];
    __shared__ int s_units[kMaxGroups + 1];  // prefix of row tiles

    unsigned char* tiles =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int rank = (int)ptx::cluster_ctarank();  // 0 = leader
    if (threadIdx.x == 0) {
        ptx::prefetch_tmap(&p.g.tm_a);
        ptx::prefetch_tmap(&p.g.tm_b1);
        if (MODE == 0) ptx::prefetch_tmap(&p.g.tm_b0);
        for (int s = 0; s < kXBars; ++s) {
            ptx::mbar_init(&full_bar[s], 1);
            ptx::mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(&tfull_bar[s], 1);
            ptx::mbar_init(&tempty_bar[s], 8);
        }
        for (int s = 0; s < kXSlots; ++s) {
            ptx::mbar_init(&ifull_bar[s], 1);
            ptx::mbar_init(&iempty_bar[s], 1);
            ptx::mbar_init(&iread_bar[s], kXProducers + 4);
        }
        abort_s = fail_s[0] = fail_s[1] = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc_pair(&tmem_base_s, kXTmemCols);
        ptx::tmem_relinquish_pair();
    }
    grid_dep_wait();  // everything below reads what the routing kernels (or GEMM-1) wrote
    const int G = p.g.G;
    for (int i = threadIdx.x; i <= G; i += kXThreads) {
        s_off[i] = p.g.offsets[i];
        s_units[i] = p.g.work_start[i];
    }
    ptx::tc_fence_before();
    __syncthreads();
    // GEMM-1 beside an early launch of the shared expert's pairs of row tiles: only an odd last tile is left of that group,
    // the last one
    const int skip = MODE == 0 && p.g.shared_split == 2 ? p.g.n_routed : -1;
    if (skip >= 0) {
        if (threadIdx.x == 0) s_units[G] = s_units[G - 1] + (((s_off[G] - s_off[G - 1] + kTileM - 1) / kTileM) & 1);
        __syncthreads();
    }
    ptx::cluster_sync_all();  // both CTAs' barriers are initialised and their tensor memory allocated
    ptx::tc_fence_after();
    const uint32_t tmem_base = tmem_base_s;
    const int nt = p.g.n_ntiles;
    const int nkb = (MODE == 0 ? p.g.d : p.g.I) / kXBK;
    volatile int* abort_flag = &abort_s;

    // This cluster's next item, by one thread (sl, sp: slot and phase, advanced). A slot is free again once the CTA's producers and
    // epilogue warps have read it, the latter when the item's accumulator is complete, so that the MMA issuer has read it too.
    // (Arrivals with cluster scope are left to the idle warp 6 of the peer: they wait for what the thread has in flight, an MMA
    // issuer's MMAs for 2700 cycles per item, an epilogue warp's stores.)
    auto next_item = [&](int* sl, int* sp, MixItem* it) {
        if (!ptx::mbar_wait(&ifull_bar[*sl], *sp, abort_flag, p.g.status, 5)) return false;
        const int4 v = s_item[*sl];
        if (++*sl == kXSlots) {
            *sl = 0;
            *sp ^= 1;
        }
        it->row0 = v.x;
        it->rows = v.y & 0xffff;
        it->ragged = (v.y >> 16) != 0;
        it->n_idx = v.z;
        it->g = v.w;
        return it->rows > 0;
    };

    if (warp == 0 || warp > 6) {
        // ------------------------------------------------ TMA producers (both CTAs; k-block c belongs to producer c % 2)
        if (ptx::elect_one()) {
            const int me = warp == 0 ? 0 : warp - 6;
            int c = 0, pos = 0;            // the next k-block and where it goes
            int r = 0;                     // the oldest k-block that may still be in use
            uint32_t run = 0, oldest = 0;  // running start (pos without the wrap) of the two
            bool ok = true;
            MixItem it;
            int sl = 0, sp = 0;
            for (int slot = 0; ok && next_item(&sl, &sp, &it); slot = sl) {
                ptx::mbar_arrive(&iread_bar[slot]);
                const bool from_x = MODE == 0 && it.g >= p.g.n_routed;  // rows read from x itself, no gathered copy
                const int half = token_rows(it.rows, it.ragged), size = kXWBytes + half * kXBK * 2;
                const int arow = (from_x ? (it.row0 - p.g.R) % p.g.x_rows : it.row0) + rank * half;
                const CUtensorMap* tm_whole = from_x ? &p.g.tm_a2 : &p.g.tm_a;
                const CUtensorMap* tm_part = from_x ? p.tm_x_part : p.tm_a_part;
                const CUtensorMap* tm_b = MODE == 1 || rank == 1 ? &p.g.tm_b1 : &p.g.tm_b0;
                const int brow = MODE == 1 ? it.g * p.g.d + it.n_idx * 256 + rank * 128
                                           : it.g * p.g.I + it.n_idx * 128 + (it.ragged ? rank * 64 : 0);
                {
                    const int at = ring_start(pos, it.ragged);
                    run += (uint32_t)(at - pos) + (at < pos ? (uint32_t)kXRing : 0u);
                    pos = at;
                }
                for (int kb = 0; kb < nkb; ++kb) {
                    if (pos + size > kXRing) {
                        run += (uint32_t)(kXRing - pos);
                        pos = 0;
                    }
                    if (r == c) oldest = run;
                    if (c % kXProducers == me) {
                        // Room for this k-block: the older ones that have to be consumed first. They are consumed in order, so the
                        // wait is for the newest of them alone. (Its barrier cannot turn over again before this k-block is loaded,
                        // and the use before, 16 k-blocks earlier, was over when this thread's last k-block had room.)
                        int newest = -1;
                        while (run + (uint32_t)size - oldest > (uint32_t)kXRing) {
                            newest = r++;
                            oldest = r < c ? s_at[me][r % kXBars] : run;
                        }
                        if (newest >= 0 &&
                            !ptx::mbar_wait(&empty_bar[newest % kXBars], (newest / kXBars) & 1, abort_flag, p.g.status, 1)) {
                            ok = false;
                            break;
                        }
                        unsigned char* w_dst = tiles + pos;
                        unsigned char* t_dst = w_dst + kXWBytes;
                        uint64_t* fb = &full_bar[c % kXBars];
                        if (rank == 0) ptx::mbar_expect_tx(fb, 2u * (uint32_t)size);  // both CTAs' bytes
                        if (!it.ragged) {
                            ptx::tma_load_2d_pair(t_dst, tm_whole, fb, kb * kXBK, arow);
                            ptx::tma_load_2d_pair(w_dst, tm_b, fb, kb * kXBK, brow);
                        } else {
                            if (MODE == 0) {
                                ptx::tma_load_2d_pair(w_dst, &p.tm_b0_half, fb, kb * kXBK, brow);
                                ptx::tma_load_2d_pair(w_dst + 64 * kXBK * 2, &p.tm_b1_half, fb, kb * kXBK, brow);
                            } else {
                                ptx::tma_load_2d_pair(w_dst, &p.g.tm_b1, fb, kb * kXBK, brow);
                            }
                            int at = 0;  // half = 16 ... 112 rows: boxes of 64, 32 and 16
                            if (half & 64) {
                                ptx::tma_load_2d_pair(t_dst, tm_part, fb, kb * kXBK, arow);
                                at = 64;
                            }
                            if (half & 32) {
                                ptx::tma_load_2d_pair(t_dst + at * kXBK * 2, tm_part + 1, fb, kb * kXBK, arow + at);
                                at += 32;
                            }
                            if (half & 16) ptx::tma_load_2d_pair(t_dst + at * kXBK * 2, tm_part + 2, fb, kb * kXBK, arow + at);
                        }
                    }
                    s_at[me][c % kXBars] = run;
                    ++c;
                    run += (uint32_t)size;
                    pos += size;
                    if (pos == kXRing) pos = 0;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer (leader CTA only)
        if (rank == 0 && ptx::elect_one()) {
            const uint32_t lo0 = (ptx::smem_u32(tiles) & 0x3FFFFu) >> 4;
            const uint32_t desc_hi32 = (uint32_t)(ptx::make_kmajor_sw128_desc(0) >> 32);
            int pos = 0, bar = 0, phase = 0;
            bool ok = true, ready = false;
            MixItem it;
            int sl = 0, sp = 0;
            for (int k = 0; ok && next_item(&sl, &sp, &it); ++k) {
                const int as = k & 1, aphase = (k >> 1) & 1;
                if (!ptx::mbar_wait(&tempty_bar[as], aphase ^ 1, abort_flag, p.g.status, 2)) break;
                ptx::tc_fence_after();
                const uint32_t d_tmem = tmem_base + as * 256;
                const int half = token_rows(it.rows, it.ragged), size = kXWBytes + half * kXBK * 2;
                const uint32_t idesc = ptx::make_idesc_bf16(256, 0) | ((uint32_t)(half >> 2) << 17);  // N = 2 half
                const uint32_t a0 = lo0 + (it.ragged ? 0u : (uint32_t)kXWBytes >> 4), b0 = lo0 + (it.ragged ? (uint32_t)kXWBytes >> 4 : 0u);
                pos = ring_start(pos, it.ragged);
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!ready && !ptx::mbar_wait(&full_bar[bar], phase, abort_flag, p.g.status, 3)) {
                        ok = false;
                        break;
                    }
                    if (pos + size > kXRing) pos = 0;
                    const int nbar = bar + 1 == kXBars ? 0 : bar + 1;
                    const int nphase = nbar == 0 ? phase ^ 1 : phase;
                    ready = ptx::umma_kblock_bf16_pair(d_tmem, a0 + ((uint32_t)pos >> 4), b0 + ((uint32_t)pos >> 4), desc_hi32, idesc,
                                                       kb > 0 ? 1u : 0u, &empty_bar[bar], &full_bar[nbar], nphase);
                    pos += size;
                    if (pos == kXRing) pos = 0;
                    bar = nbar;
                    phase = nphase;
                }
                if (ok) ptx::umma_commit_pair(&tfull_bar[as], 3);
            }
        }
        __syncwarp();
    } else if (warp == 6 && rank == 0) {
        // ------------------------------------------------ item scheduler (leader CTA, whole warp)
        const int total = s_units[G] * nt, clusters = (int)gridDim.x >> 1;
        int i = (int)blockIdx.x >> 1, sl = 0, sp = 1;
        int next = 0;  // lane 0: the index after i, on its way while i is decoded
        for (;;) {
            if (lane == 0 && i < total) next = clusters + atomicAdd(p.queue, 1);
            int4 v = make_int4(0, 0, 0, 0);
            if (i < total) {
                int g = 0;  // groups whose items all come before i
                for (int g0 = 0; g0 < G; g0 += 32) {
                    const unsigned m = __ballot_sync(0xffffffffu, g0 + lane < G && s_units[min(g0 + lane, G - 1) + 1] * nt <= i);
                    g += __popc(m);
                    if (m != 0xffffffffu) break;
                }
                const int units = s_units[g + 1] - s_units[g], local = i - s_units[g] * nt;
                // the faster index is the one with fewer values: clusters that run together share the larger operand
                const bool rows_outer = units > nt;
                const int q = local / (rows_outer ? nt : units), j = rows_outer ? q : local - q * units;
                const int off = s_off[g], rows = s_off[g + 1] - off;
                const int whole = g == skip ? 0 : whole_items(rows);
                const int row0 = g == skip ? rows / 256 * 256 : j * 256;
                v.x = off + row0;
                v.y = min(256, rows - row0) | (j >= whole ? 1 << 16 : 0);
                v.z = rows_outer ? local - j * nt : q;
                v.w = g;
            }
            int ok = 1;
            if (lane == 0) {
                ok = ptx::mbar_wait(&iread_bar[sl], sp, abort_flag, p.g.status, 6) &&
                     ptx::mbar_wait<true>(&iempty_bar[sl], sp, abort_flag, p.g.status, 7);
                if (ok)
                    for (uint32_t r = 0; r < 2; ++r) ptx::st_async(&s_item[sl], v, &ifull_bar[sl], r);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok || i >= total) break;
            i = __shfl_sync(0xffffffffu, next, 0);
            if (++sl == kXSlots) {
                sl = 0;
                sp ^= 1;
            }
        }
    } else if (warp == 6) {
        // ------------------------------------------------ the peer's slots back to the leader
        if (ptx::elect_one()) {
            MixItem it;
            int sl = 0, sp = 0;
            for (int slot = 0, phase = 0; next_item(&sl, &sp, &it); slot = sl, phase = sp) {
                if (!ptx::mbar_wait(&iread_bar[slot], phase, abort_flag, p.g.status, 8)) break;
                ptx::mbar_arrive_leader_cluster(&iempty_bar[slot]);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue warps (TMEM lane quadrant = warp % 4)
        const int q = warp & 3;
        unsigned char* out_buf = tiles + kXRing + q * kXOutBytes;
        int xp = 0;  // which half of the exchange buffer
        int sl = 0, sp = 0;
        for (int k = 0;; ++k) {
            MixItem it{};
            int ok = 1, rr = 0;
            const int slot = sl;  // (lane 0's)
            const int as = k & 1, aphase = (k >> 1) & 1;
            if (lane == 0) {
                ok = next_item(&sl, &sp, &it) ? 1 : 0;
                rr = it.rows | (it.ragged ? 1 << 16 : 0);
            }
            rr = __shfl_sync(0xffffffffu, rr, 0);
            const int row0 = __shfl_sync(0xffffffffu, it.row0, 0), n_idx = __shfl_sync(0xffffffffu, it.n_idx, 0);
            const int rows = rr & 0xffff;
            const bool ragged = (rr >> 16) != 0;
            // GEMM-2: the target row and weight of this lane's row (ragged: of its first chunk), asked for before the wait
            const int my_row = ragged ? lane : rank * kTileM + q * 32 + lane;
            const bool weighted = MODE == 1 && p.g.o32 == nullptr;
            int drow = row0 + my_row;
            float wv = 0.f;
            if (weighted && my_row < rows) {
                wv = p.g.row_w[drow];
                if (!p.g.store_rows) drow = p.g.row_tok[drow];
            }
            if (lane == 0) {
                if (ok) ok = ptx::mbar_wait(&tfull_bar[as], aphase, abort_flag, p.g.status, 4) ? 1 : 0;
                if (!ok) fail_s[as] = 1;  // (a warp may be an item ahead of the one that reads the flag)
            }
            // The four warps go on together or not at all: the ragged items' exchange below has them wait for one another
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (*(volatile int*)&fail_s[as]) break;
            if (lane == 0) ptx::mbar_arrive(&iread_bar[slot]);
            ptx::tc_fence_after();
            const uint32_t taddr = tmem_base + as * 256 + ((uint32_t)(q * 32) << 16);
            if (!ragged) {  // lane = token row of this CTA, column = feature
                const bool valid = my_row < rows;
                const int grow = row0 + my_row;
                const unsigned vmask = __ballot_sync(0xffffffffu, valid);
                if (vmask == 0u) {
                    // no row of this quadrant is stored
                } else if (MODE == 0) {
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        const int col0 = n_idx * 128 + c * 32;
                        if (col0 >= p.g.I) break;
                        uint32_t gv[32], uv[32];
                        ptx::tmem_ld32(taddr + c * 32, gv);
                        ptx::tmem_ld32(taddr + 128 + c * 32, uv);
                        ptx::tmem_ld_wait();
                        uint32_t pk[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float g0 = __uint_as_float(gv[2 * j]), g1 = __uint_as_float(gv[2 * j + 1]);
                            const float u0 = __uint_as_float(uv[2 * j]), u1 = __uint_as_float(uv[2 * j + 1]);
                            pk[j] = pack_bf16x2(__fdividef(g0, 1.0f + __expf(-g0)) * u0, __fdividef(g1, 1.0f + __expf(-g1)) * u1);
                        }
                        if (valid) {
                            __nv_bfloat16* dst = p.g.H + (size_t)grow * p.g.I + col0;
                            ptx::st_global32(dst, pk);
                            ptx::st_global32(dst + 16, pk + 8);
                        }
                    }
                } else {
                    // GEMM-2's items are short where I is: the next chunk's load from tensor memory is in flight while this one's
                    // rows are stored
                    const int chunks = min(8, (p.g.d - n_idx * 256) >> 5);  // even: d is a multiple of 64
                    const bool raw = p.g.o32 != nullptr;                    // fp32 rows (calibration outputs)
                    const bool in_order = raw || p.g.store_rows;
                    const size_t row_bytes = (size_t)p.g.d * (raw ? 4 : 2);
                    char* base = (raw ? reinterpret_cast<char*>(p.g.o32 + n_idx * 256) : reinterpret_cast<char*>(p.g.y + n_idx * 256)) +
                                 (in_order ? (size_t)(row0 + rank * kTileM + q * 32) * row_bytes : 0);
                    auto put = [&](uint32_t (&v)[32], int c) {
                        if (raw) {
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                stage_put(out_buf, lane, j, make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]));
                            stage_flush_rows(out_buf, lane, vmask, base + c * 128, row_bytes);
                            return;
                        }
                        uint32_t pk[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            pk[j] = pack_bf16x2(wv * __uint_as_float(v[2 * j]), wv * __uint_as_float(v[2 * j + 1]));
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            stage_put(out_buf, lane, (c & 1) * 4 + j, make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]));
                        if (c & 1) {
                            if (in_order) stage_flush_rows(out_buf, lane, vmask, base + (c - 1) * 64, row_bytes);
                            else stage_flush(out_buf, lane, vmask, drow, base + (c - 1) * 64, row_bytes);
                        }
                    };
                    uint32_t va[32], vb[32];
                    ptx::tmem_ld32(taddr, va);
#pragma unroll
                    for (int c = 0; c < 8; c += 2) {
                        if (c >= chunks) break;
                        ptx::tmem_ld_wait(va);
                        ptx::tmem_ld32(taddr + (c + 1) * 32, vb);
                        put(va, c);
                        ptx::tmem_ld_wait(vb);
                        if (c + 2 < chunks) ptx::tmem_ld32(taddr + (c + 2) * 32, va);
                        put(vb, c + 1);
                    }
                }
            } else if (MODE == 0) {  // lane = feature (gate: q 0, 1; up: q 2, 3), column = token
                const int f0 = n_idx * 128 + rank * 64 + (q & 1) * 32;
                const bool is_up = q >= 2;
                unsigned char* stage_buf = out_buf + 4096;  // [16 tokens][32 features] bf16
                const int part = (rows + 31) / 32;
#pragma unroll 1
                for (int c = 0; c < part && f0 < p.g.I; ++c) {  // both warps of an exchange have the same f0
                    uint32_t v[32];
                    ptx::tmem_ld32(taddr + c * 32, v);
                    ptx::tmem_ld_wait();
                    uint32_t* mine = reinterpret_cast<uint32_t*>(out_buf + xp * 2048) + lane;
                    const uint32_t* theirs = reinterpret_cast<const uint32_t*>(out_buf + ((q ^ 2) - q) * kXOutBytes + xp * 2048) + lane;
                    xp ^= 1;
                    // the gate warp finishes tokens 0-15 of the chunk, the up warp tokens 16-31
#pragma unroll
                    for (int j = 0; j < 16; ++j) mine[j * 32] = is_up ? v[j] : v[16 + j];
                    if (q & 1) asm volatile("bar.sync 3, 64;" ::: "memory");
                    else asm volatile("bar.sync 2, 64;" ::: "memory");
                    const int t0 = c * 32 + (is_up ? 16 : 0);
                    uint32_t other[16];  // all of them read before the first store: the compiler cannot tell the buffers apart
#pragma unroll
                    for (int j = 0; j < 16; ++j) other[j] = theirs[j * 32];
                    __nv_bfloat16 h[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float o = __uint_as_float(other[j]), s = __uint_as_float(is_up ? v[16 + j] : v[j]);
                        const float g = is_up ? o : s, u = is_up ? s : o;
                        h[j] = __float2bfloat16_rn(__fdividef(g, 1.0f + __expf(-g)) * u);
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) reinterpret_cast<__nv_bfloat16*>(stage_buf)[j * 32 + lane] = h[j];
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 2; ++j) {  // four lanes store the 64 bytes of a token's row
                        const int t = j * 8 + (lane >> 2);
                        if (t0 + t < rows)
                            *reinterpret_cast<uint4*>(p.g.H + (size_t)(row0 + t0 + t) * p.g.I + f0 + (lane & 3) * 8) =
                                *reinterpret_cast<const uint4*>(stage_buf + t * 64 + (lane & 3) * 16);
                    }
                    __syncwarp();
                }
            } else {  // lane = output feature, column = token
                const int f0 = n_idx * 256 + rank * 128 + q * 32;
                float* wbuf = reinterpret_cast<float*>(out_buf + 6144);
                const int part = (rows + 31) / 32;
#pragma unroll 1
                for (int c = 0; c < part && f0 < p.g.d; ++c) {
                    const int t0 = c * 32;
                    int next_row = row0 + t0 + 32 + lane;  // the next chunk's
                    float next_w = 0.f;
                    if (weighted && t0 + 32 + lane < rows) {
                        next_w = p.g.row_w[next_row];
                        if (!p.g.store_rows) next_row = p.g.row_tok[next_row];
                    }
                    uint32_t v[32];
                    ptx::tmem_ld32(taddr + c * 32, v);
                    ptx::tmem_ld_wait();
                    if (p.g.o32 != nullptr) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) reinterpret_cast<uint32_t*>(out_buf)[j * 32 + lane] = v[j];
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 8; ++j) {  // eight lanes store the 128 bytes of a row
                            const int t = j * 4 + (lane >> 3);
                            if (t0 + t < rows)
                                *reinterpret_cast<uint4*>(p.g.o32 + (size_t)(row0 + t0 + t) * p.g.d + f0 + (lane & 7) * 4) =
                                    *reinterpret_cast<const uint4*>(out_buf + t * 128 + (lane & 7) * 16);
                        }
                    } else {
                        wbuf[lane] = wv;
                        __syncwarp();
                        float4 w4[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) w4[j] = reinterpret_cast<const float4*>(wbuf)[j];
                        const float* w = reinterpret_cast<const float*>(w4);
                        __nv_bfloat16 o[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j) o[j] = __float2bfloat16_rn(w[j] * __uint_as_float(v[j]));
#pragma unroll
                        for (int j = 0; j < 32; ++j) reinterpret_cast<__nv_bfloat16*>(out_buf)[j * 32 + lane] = o[j];
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 4; ++j) {  // four lanes store 64 bytes of a row
                            const int t = j * 8 + (lane >> 2);
                            const int target = __shfl_sync(0xffffffffu, drow, t);
                            if (t0 + t < rows)
                                *reinterpret_cast<uint4*>(p.g.y + (size_t)target * p.g.d + f0 + (lane & 3) * 8) =
                                    *reinterpret_cast<const uint4*>(out_buf + t * 64 + (lane & 3) * 16);
                        }
                    }
                    __syncwarp();
                    drow = next_row;
                    wv = next_w;
                }
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_leader(&tempty_bar[as]);
        }
    }

    // ------------------------------------------------ teardown
    if (threadIdx.x == 64) grid_dep_launch();  // after the epilogue loop, as in the one-CTA kernel
    ptx::tc_fence_before();
    __syncthreads();
    if (abort_s) __nanosleep(100000);  // let any copy still in flight land before shared memory is released
    ptx::cluster_sync_all();           // the peer is done with this CTA's shared and tensor memory
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc_pair(tmem_base, kXTmemCols);
    }
}

template <int MODE>
cudaError_t launch_mixed_t(const MixedGemmParams& p, int grid, cudaStream_t s) {
    cudaError_t err = ensure_smem(grouped_gemm_mixed_kernel<MODE>, kXSmem);
    if (err != cudaSuccess) return err;
    return launch_pdl_cluster(grouped_gemm_mixed_kernel<MODE>, std::max(2, grid & ~1), kXThreads, kXSmem, 2, s, p);
}

}  // namespace

cudaError_t launch_grouped_gemm1_mixed(const MixedGemmParams& p, int grid, cudaStream_t s) { return launch_mixed_t<0>(p, grid, s); }
cudaError_t launch_grouped_gemm2_mixed(const MixedGemmParams& p, int grid, cudaStream_t s) { return launch_mixed_t<1>(p, grid, s); }

}  // namespace exfold
