// Expert FFN of fp32 layers (Eq. 1) on the CUDA cores: tensor cores would round fp32 inputs.
//
// A cluster of 8 CTAs (4 or 2 where there are many tiles of a small layer) per row tile (up to tile_rows sorted rows of one
// expert). Phase 0: CTA r computes its share of the intermediate features, gate and up, for all rows of the tile, and leaves silu(gate) * up in shared memory. Phase 1,
// after a cluster barrier: CTA r computes its share of the output features with all of I as K. The activation crosses the
// cluster through distributed shared memory and never goes to memory; one launch does the whole FFN, and a tile's weights
// are read once per tile instead of once per row. Two kernels:
//
//   short tiles (8 rows)  Bound by latency and the weights' bytes. The lanes of a warp lie along K and load the weights
//       straight into registers, a group of 4 weight rows at a time with the next group's loads in flight (phase 1's first
//       ones before the cluster barrier); the tokens lie in shared memory whole. The 4 x 8 sums of a group are reduced over
//       the lanes by halving exchanges (31 shuffles), which leaves one sum per lane. Activations are written to every
//       CTA's copy of H as they are computed.
//   tall tiles (16 or 32 rows)  Bound by the multiply-adds. 32-wide K chunks pass through two shared-memory stages, the
//       next chunk's loads in registers meanwhile (cp.async moves only ~17 bytes per cycle and SM in 16-byte pieces: it
//       took longer than the arithmetic). A warp covers 4 TM rows x 8 NW weight rows, its lanes 4 rows x 8 weight rows,
//       so that a 16-byte shared-memory read of a warp touches at most 128 distinct bytes (one wavefront) and TM + NW of
//       them feed 4 TM NW multiply-adds; TM = NW = 4 with two warps along 32 rows, TM = 4, NW = 2 for 16 rows. The
//       remaining warps lie along the features; where a CTA has too few features for them they split K (partial sums
//       meet in shared memory, in order). A CTA keeps its slice of H and the others read it chunk by chunk.
//
// Sums: a few products in a row, partial sums added in order - the error of a two-level sum, as with a warp per output.
// Measured (one CTA per route with a warp per output feature -> cp.async stages for every tile height -> now): tiny layer,
// 64 rows of 128 x 256 24 -> 12.4 -> 7.6 us; one token, 9 experts of 512 x 384, whole call 171 -> 40 -> 33; tall: 400 rows
// of 768 x 1024 750 -> 158 -> 149 us (12.7 TFLOP/s); 2048 rows of 256 x 512 270 -> 130 -> 123. What bounds the tall form now
// is shared-memory reads (a 16-byte read costs a wavefront per quarter warp, so 32 for the 64 multiply-adds they feed).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "ptx.cuh"
#include "route_token.cuh"

#include <cooperative_groups.h>

namespace exfold {

namespace {

namespace cg = cooperative_groups;

constexpr int kMaxCl = 8;  // CTAs per row tile, at most
constexpr int kThreads = 256;  // 8 warps
constexpr int kKC = 32;        // tall tiles: K elements per stage
constexpr int kLd = kKC + 4;   // row pitch in floats: 16-byte aligned, the rows of a warp's read hit distinct banks
// Four consecutive floats, `left` of which exist (<= 0: none), the others zero. VEC: 16-byte aligned, all or none
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* src, int left) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (VEC) {
        if (left > 0) v = __ldg(reinterpret_cast<const float4*>(src));
    } else {
        if (left > 0) v.x = __ldg(src);
        if (left > 1) v.y = __ldg(src + 1);
        if (left > 2) v.z = __ldg(src + 2);
        if (left > 3) v.w = __ldg(src + 3);
    }
    return v;
}

// The group, rows and expert of a row tile: every group's tile range in one round trip. False: past the last tile
struct Tile {
    int g, row0, rows, expert;
};
__device__ __forceinline__ bool find_tile(const FfnF32Params& p, int tile, Tile* s) {
    if (threadIdx.x == 0) s->g = -1;
    __syncthreads();
    const int gd = p.n_groups_dev != nullptr ? *p.n_groups_dev : p.G;
    for (int g = threadIdx.x; g < p.G; g += kThreads) {
        const int t0 = p.tile_start[g], t1 = p.tile_start[g + 1], o0 = p.offsets[g], o1 = p.offsets[g + 1];
        const int e = p.grp_expert != nullptr ? p.grp_expert[g] : g;
        if (g < gd && tile >= t0 && tile < t1) {
            s->g = g;
            s->row0 = o0 + (tile - t0) * p.tile_rows;
            s->rows = min(p.tile_rows, o1 - s->row0);
            s->expert = e;
        }
    }
    __syncthreads();
    return s->g >= 0;
}
__device__ __forceinline__ int64_t token_of(const FfnF32Params& p, int64_t row) {
    return p.row_tok != nullptr ? (int64_t)p.row_tok[row] : row % p.x_rows;
}
__device__ __forceinline__ float swiglu(float g, float u) { return (g / (1.0f + expf(-g))) * u; }

// ---------------------------------------------------------------- short tiles
constexpr int kSR = 8;  // token rows of a tile
constexpr int kSW = 4;  // weight rows of a group: phase 0 two features' gate rows and up rows, phase 1 four columns

// Sum over the lanes of 32 values by halving exchanges: lane l ends up with the sum of value l
template <int N, int OFF>
__device__ __forceinline__ void lane_sums(float* v, int lane) {
    if constexpr (OFF > 0) {
        const bool up = (lane & OFF) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const float keep = up ? v[i + N / 2] : v[i], send = up ? v[i] : v[i + N / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, OFF);
        }
        lane_sums<N / 2, OFF / 2>(v, lane);
    }
}

// Prefill of at most kRoutedTokens tokens on a grid of one wave: every cluster routes all of them, a token per warp of the
// cluster at a time, hands the routes round through distributed shared memory and picks the rows of its tile; the first cluster
// writes the metadata, each tile its part of the permutation. One kernel instead of three, each of which waited for the one
// before and for its lists: tiny layer, 64 tokens 14.4 -> 9.6 us per call, one token
// 12.3 -> 8.9, with the router before it 16.0 -> 12.3.
constexpr int kRoutedTokens = 128;
constexpr int kRoutedSlots = 512;  // routes, at most
constexpr int kRoutedExperts = 128;
struct PrefillRouteSmem {
    short id[kRoutedSlots];
    float w[kRoutedSlots];
    int cnt[kMaxExperts];
    int warp_sum[kThreads / 32];
    int skip;  // the tile's first route of its expert
    int tok[kSR];
    float rw[kSR];
};

template <int CL, int NPL>
__device__ __forceinline__ bool route_tile(const FfnF32Route& rt, cg::cluster_group& cluster, int tile, PrefillRouteSmem& sm, Tile* st) {
    const PrefillRouteParams& p = rt.r;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rank = (int)cluster.block_rank();
    const int T = (int)p.T, N = p.N, Kp = p.Kp, Ko = p.K - p.Kp, n = T * Kp;
    const bool first = blockIdx.x < CL;  // this cluster writes the metadata
    constexpr int kWarps = kThreads / 32;
    sm.cnt[threadIdx.x] = 0;  // N <= 256 = kThreads
    if (threadIdx.x == 0) st->g = -1;
    cluster.barrier_arrive();
    grid_dep_wait();
    if (p.status != nullptr && blockIdx.x == 0 && threadIdx.x < 4) reinterpret_cast<int*>(p.status)[threadIdx.x] = 0;
    bool started = false;
    for (int t = warp * CL + rank; t < T; t += CL * kWarps) {
        float v[NPL];
#pragma unroll
        for (int q = 0; q < NPL; ++q) v[q] = lane + 32 * q < N ? p.logits[(size_t)t * N + lane + 32 * q] : -INFINITY;
        const TokenRoute r = route_token<NPL>(p, v, lane);
        if (!started) cluster.barrier_wait();  // before the first remote write: all CTAs of the cluster have started
        started = true;
        if (r.kept) {
#pragma unroll
            for (int c = 0; c < CL; ++c) {
                cluster.map_shared_rank(sm.id, c)[t * Kp + r.rank] = (short)r.id;
                cluster.map_shared_rank(sm.w, c)[t * Kp + r.rank] = r.w;
            }
            if (first) {
                p.ids[t * Kp + r.rank] = r.id;
                p.w[t * Kp + r.rank] = r.w;
            }
        } else if (r.omitted && first) {
            p.omit_src[t * Ko + (r.rank - Kp)] = r.id;
            p.omit_tgt[t * Ko + (r.rank - Kp)] = r.tgt;
        }
    }
    if (!started) cluster.barrier_wait();
    cluster.sync();  // every copy of the routes is complete
    for (int i = threadIdx.x; i < n; i += kThreads) atomicAdd(&sm.cnt[sm.id[i]], 1);
    __syncthreads();
    // a thread per expert: its rows and tiles, prefixes of both in one word
    const int mine = sm.cnt[threadIdx.x], packed = mine | (mine + kSR - 1) / kSR << 16;
    int incl = packed;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) sm.warp_sum[warp] = incl;
    __syncthreads();
    int before = incl - packed, all = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        if (w < warp) before += sm.warp_sum[w];
        all += sm.warp_sum[w];
    }
    const int off = before & 0xffff, t0 = before >> 16, routed_tiles = all >> 16;
    if (first && rank == 0) {
        if ((int)threadIdx.x < N) rt.offsets[threadIdx.x] = off;
        if (threadIdx.x == 0) {
            rt.offsets[N] = n;
            if (rt.n_shared) rt.offsets[N + 1] = n + T;
        }
    }
    if (tile >= routed_tiles) {  // the shared expert's rows: the tokens in order, weight 1
        const int j0 = (tile - routed_tiles) * kSR;
        if (!rt.n_shared || j0 >= T) return false;
        if (threadIdx.x == 0) *st = Tile{N, n + j0, min(kSR, T - j0), N};
        if (threadIdx.x < kSR && j0 + (int)threadIdx.x < T) {
            sm.tok[threadIdx.x] = j0 + threadIdx.x;
            sm.rw[threadIdx.x] = 1.0f;
            if (rank == 0) {
                rt.row_tok[n + j0 + threadIdx.x] = j0 + threadIdx.x;
                rt.row_w[n + j0 + threadIdx.x] = 1.0f;
            }
        }
        __syncthreads();
        return true;
    }
    if (tile >= t0 && tile < t0 + (packed >> 16)) {
        const int k = (tile - t0) * kSR;
        *st = Tile{(int)threadIdx.x, off + k, min(kSR, mine - k), (int)threadIdx.x};
        sm.skip = k;
    }
    __syncthreads();
    if (warp == 0) {  // the expert's routes in (token, slot) order
        const int e = st->g, k = sm.skip, row0 = st->row0;
        for (int c0 = 0, seen = 0; c0 < n && seen < k + kSR; c0 += 32) {
            const int r = c0 + lane;
            const bool hit = r < n && sm.id[r] == e;
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            const int at = seen + __popc(m & ((1u << lane) - 1u)) - k;
            if (hit && at >= 0 && at < kSR) {
                sm.tok[at] = r / Kp;
                sm.rw[at] = sm.w[r];
                if (rank == 0) {
                    rt.perm[row0 + at] = r;
                    rt.inv_pos[r] = row0 + at;
                    rt.row_tok[row0 + at] = r / Kp;
                    rt.row_w[row0 + at] = sm.w[r];
                }
            }
            seen += __popc(m);
        }
    }
    __syncthreads();
    return true;
}

// Decode on a grid of one wave, likewise: every cluster takes the Top-K of all tokens (a token per warp at a time), sums the
// routed weights, ranks the pool, finds the targets (an expert per warp at a time), remaps the slots and picks the rows of its
// tile; the first cluster writes the metadata, each tile its part of the lists that the sum after it reads. The arithmetic is
// decode_route_kernel's. Whole call before / now: tiny layer 16 tokens 16.1 / 12.7 us, one 15.5 / 12.3, 74 19.9 / 15.0.
struct DecodeRouteSmem {
    double w64[kRoutedSlots];
    long long key[kRoutedExperts];           // order-preserving image of the expert's score
    unsigned long long acc[kRoutedExperts];  // sum_i w_{i,e} in 2^-53 units: exact, order-independent
    short id[kRoutedSlots];
    float wrm[kRoutedSlots];  // remapped weights
    int in_union[kRoutedExperts];
    int rank_of[kRoutedExperts];  // pool rank or -1
    int pool[kRoutedExperts];
    int target[kRoutedExperts];
    float scale[kRoutedExperts];
    unsigned mask[kRoutedExperts][kRoutedTokens / 32];  // by pool rank: the tokens with a row
    int warp_sum[kThreads / 32];
    int skip, P;
    int tok[kSR];
    float rw[kSR];
};

template <int CL, int NPL>
__device__ __forceinline__ bool route_tile(const DecodeRouteParams& p, cg::cluster_group& cluster, int tile, DecodeRouteSmem& sm, Tile* st) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = (int)cluster.block_rank();
    const int B = p.B, N = p.N, K = p.K, M = p.M, n = B * K;
    const bool first = blockIdx.x < CL, meta = first && rank == 0;
    const bool is_static = p.st_pool != nullptr;
    constexpr int kWarps = kThreads / 32;
    for (int e = tid; e < N; e += kThreads) {
        sm.acc[e] = 0ull;
        sm.in_union[e] = 0;
        sm.rank_of[e] = -1;
    }
    for (int i = tid; i < kRoutedExperts * (kRoutedTokens / 32); i += kThreads) (&sm.mask[0][0])[i] = 0u;
    if (tid == 0) st->g = -1;
    cluster.barrier_arrive();
    grid_dep_wait();
    if (p.status != nullptr && blockIdx.x == 0 && tid < 4) reinterpret_cast<int*>(p.status)[tid] = 0;
    bool started = false;
    for (int i = warp * CL + rank; i < B; i += CL * kWarps) {  // Eq. 2
        float v[NPL];
#pragma unroll
        for (int q = 0; q < NPL; ++q) v[q] = lane + 32 * q < N ? p.logits[(size_t)i * N + lane + 32 * q] : -INFINITY;
        int id;
        const double w = warp_topk_softmax<NPL>(v, N, K, lane, &id);
        if (!started) cluster.barrier_wait();  // before the first remote write: all CTAs of the cluster have started
        started = true;
        if (lane < K) {
#pragma unroll
            for (int c = 0; c < CL; ++c) {
                cluster.map_shared_rank(sm.id, c)[i * K + lane] = (short)id;
                cluster.map_shared_rank(sm.w64, c)[i * K + lane] = w;
            }
        }
    }
    if (!started) cluster.barrier_wait();
    cluster.sync();  // every copy of the routes is complete
    if (is_static) {
        for (int e = tid; e < N; e += kThreads) {
            sm.target[e] = p.st_target[e];
            sm.scale[e] = p.st_scale[e];
        }
        for (int j = tid; j < M; j += kThreads) {
            const int e = p.st_pool[j];
            sm.pool[j] = e;
            sm.rank_of[e] = j;
        }
        if (tid == 0) sm.P = M;
        __syncthreads();
    } else {
        for (int s = tid; s < n; s += kThreads) {
            const int e = sm.id[s];
            atomicAdd(&sm.acc[e], (unsigned long long)(sm.w64[s] * 9007199254740992.0));
            sm.in_union[e] = 1;
        }
        __syncthreads();
        // Eq. 11: score_e = h_e * sum_i w_{i,e}; a thread per expert counts the better ones (score desc, id asc)
        int in = 0;
        if (tid < N) {
            in = sm.in_union[tid];
            sm.key[tid] = score_order_key((double)sm.acc[tid] * (1.0 / 9007199254740992.0) * (double)p.h[tid]);
        }
        const int usz = __syncthreads_count(in);
        if (in) {
            const long long ke = sm.key[tid];
            int better = 0;
            for (int o = 0; o < N; ++o)
                better += sm.in_union[o] && (sm.key[o] > ke || (sm.key[o] == ke && o < tid)) ? 1 : 0;
            if (better < M) {
                sm.rank_of[tid] = better;
                sm.pool[better] = tid;
            }
        }
        if (tid == 0) sm.P = usz < M ? usz : M;
        __syncthreads();
        // Eq. 12, a warp of the cluster per source expert: itself if in the pool, else its minimum-loss pool expert
        const int P = sm.P;
        for (int s = warp * CL + rank; s < N; s += CL * kWarps) {
            int bt = s;
            float sc = 1.0f;
            if (sm.rank_of[s] < 0) {  // warp-uniform
                const float* row = p.L + (size_t)s * N;
                float bl = INFINITY;
                int bj = 0x7fffffff;
                for (int j = lane; j < P; j += 32) {
                    const int t = sm.pool[j];
                    const float l = __ldg(row + t);
                    if (bj == 0x7fffffff || l < bl || (l == bl && t < bj)) {
                        bl = l;
                        bj = t;
                    }
                }
                bt = warp_argmin(bj != 0x7fffffff, float_order_key(bl), bj);
                sc = __ldg(p.S + (size_t)s * N + bt);
            }
            if (lane < CL) {
                cluster.map_shared_rank(sm.target, lane)[s] = bt;
                cluster.map_shared_rank(sm.scale, lane)[s] = sc;
            }
        }
        cluster.sync();  // the targets are in every copy
    }
    const int P = sm.P;
    for (int s = tid; s < n; s += kThreads) {  // Eq. 14
        const int e = sm.id[s], t = sm.target[e], i = s / K;
        const float wv = (float)(sm.w64[s] * (double)sm.scale[e]);
        sm.id[s] = (short)t;
        sm.wrm[s] = wv;
        if (sm.rank_of[t] >= 0) atomicOr(&sm.mask[sm.rank_of[t]][i >> 5], 1u << (i & 31));
        if (meta) {
            p.ids[s] = t;
            p.w[s] = wv;
        }
    }
    if (meta) {
        for (int e = tid; e < N; e += kThreads) {
            p.target[e] = sm.target[e];
            p.scale[e] = sm.scale[e];
            p.pool_ids[e] = e < P ? sm.pool[e] : -1;
        }
        if (tid < 8) {
            uint32_t m = 0;
            for (int b = 0; b < 32; ++b) {
                const int e = tid * 32 + b;
                if (e < N && sm.rank_of[e] >= 0) m |= 1u << b;
            }
            p.pool_mask[tid] = m;
        }
        if (tid == 0) *p.pool_size = P;
    }
    __syncthreads();
    // a thread per group: its rows and tiles, prefixes of both in one word
    int mine = 0;
    if (tid < P)
#pragma unroll
        for (int q = 0; q < kRoutedTokens / 32; ++q) mine += __popc(sm.mask[tid][q]);
    const int packed = mine | (mine + kSR - 1) / kSR << 16;
    int incl = packed;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) sm.warp_sum[warp] = incl;
    __syncthreads();
    int before = incl - packed, all = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        if (w < warp) before += sm.warp_sum[w];
        all += sm.warp_sum[w];
    }
    const int off = before & 0xffff, t0 = before >> 16, rows = all & 0xffff, pool_tiles = all >> 16;
    if (meta && tid == 0) {
        p.n_groups[0] = P + (p.n_shared ? 1 : 0);
        p.n_groups[1] = rows + (p.n_shared ? B : 0);
        p.n_groups[2] = rows;  // first row of the shared expert's group
    }
    if (tile >= pool_tiles) {  // the shared expert's rows: the tokens in order, weight 1
        const int j0 = (tile - pool_tiles) * kSR;
        if (!p.n_shared || j0 >= B) return false;
        if (tid == 0) *st = Tile{P, rows + j0, min(kSR, B - j0), N};
        if (tid < kSR && j0 + tid < B) {
            sm.tok[tid] = j0 + tid;
            if (rank == 0) {
                p.row_tok[rows + j0 + tid] = j0 + tid;
                p.row_w[rows + j0 + tid] = 1.0f;
            }
        }
        __syncthreads();
        return true;
    }
    if (tile >= t0 && tile < t0 + (packed >> 16)) {
        const int k = (tile - t0) * kSR;
        *st = Tile{tid, off + k, min(kSR, mine - k), sm.pool[tid]};
        sm.skip = k;
    }
    __syncthreads();
    if (warp == 0) {  // the group's tokens in order
        const int g = st->g, e = st->expert, k = sm.skip, row0 = st->row0;
        for (int q = 0, seen = 0; q < kRoutedTokens / 32; ++q) {
            const unsigned m = sm.mask[g][q];
            const int i = q * 32 + lane, at = seen + __popc(m & ((1u << lane) - 1u)) - k;
            if (((m >> lane) & 1u) && at >= 0 && at < kSR) {
                float ws = 0.f;
                int slot = -1;  // a token's first slot with this target has the row, the others are merged into it
                for (int a = 0; a < K; ++a)
                    if (sm.id[i * K + a] == e) {
                        ws = slot >= 0 ? __fadd_rn(ws, sm.wrm[i * K + a]) : sm.wrm[i * K + a];
                        if (rank == 0) p.slot_row[i * K + a] = slot >= 0 ? -1 : row0 + at;
                        if (slot < 0) slot = a;
                    }
                sm.tok[at] = i;
                if (rank == 0) {
                    p.row_tok[row0 + at] = i;
                    p.row_w[row0 + at] = ws;
                }
            }
            seen += __popc(m);
        }
    }
    __syncthreads();
    return true;
}

struct NoRoute {};  // the tiles' rows come from lists that kernels before it wrote
struct NoRouteSmem {
    int tok[1];
    float rw[1];
};
template <typename R>
struct RouteSmemOf {
    using type = NoRouteSmem;
};
template <>
struct RouteSmemOf<FfnF32Route> {
    using type = PrefillRouteSmem;
};
template <>
struct RouteSmemOf<DecodeRouteParams> {
    using type = DecodeRouteSmem;
};

// R: who routes the tokens; NPL: their scores per lane
template <int CL, bool VEC, typename R, int NPL>
__global__ void __launch_bounds__(kThreads) ffn_f32_short_kernel(FfnF32Params p, const __grid_constant__ R rt) {
    extern __shared__ __align__(16) float smem[];
    __shared__ Tile s_tile;
    __shared__ typename RouteSmemOf<R>::type rs;
    constexpr bool kRoutes = NPL > 0;
    const int d = p.d, I = p.I, xld = (d + 127) / 128 * 128, hld = p.hld;  // whole 128-wide K chunks
    float* xs = smem;             // [8][xld]
    float* hs = smem + kSR * xld;  // [8][hld]
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWarps = kThreads / 32;
    if constexpr (kRoutes) {
        if (!route_tile<CL, NPL>(rt, cluster, (int)(blockIdx.x / CL), rs, &s_tile)) return;  // the whole cluster
    } else {
        grid_dep_wait();
        if (!find_tile(p, (int)(blockIdx.x / CL), &s_tile)) return;  // the whole cluster
        cluster.barrier_arrive();  // waited for before the first remote write: all CTAs of the cluster have started
    }
    const int rows = s_tile.rows;
    const int64_t row0 = s_tile.row0;
    const size_t e = s_tile.expert;
    const int per0 = (I + CL - 1) / CL, per1 = (d + CL - 1) / CL;

    // Lane's elements of K chunk c: VEC 4 consecutive ones, else 4 that are 32 apart
    auto load_w = [&](const float* row, bool in, int c, int K) {
        if (VEC) return load4<true>(row + c * 128 + lane * 4, in ? K - c * 128 - lane * 4 : 0);
        float4 v;
        const int k = c * 128 + lane;
        v.x = in && k < K ? __ldg(row + k) : 0.f;
        v.y = in && k + 32 < K ? __ldg(row + k + 32) : 0.f;
        v.z = in && k + 64 < K ? __ldg(row + k + 64) : 0.f;
        v.w = in && k + 96 < K ? __ldg(row + k + 96) : 0.f;
        return v;
    };
    auto load_t = [&](const float* row, int c) {
        if (VEC) return *reinterpret_cast<const float4*>(row + c * 128 + lane * 4);
        const float* q = row + c * 128 + lane;
        return make_float4(q[0], q[32], q[64], q[96]);
    };
    // item (group gi of this CTA, chunk c) of a phase: the four weight rows' elements
    auto load_item = [&](int phase, int gi, int c, float4 (&w)[kSW]) {
#pragma unroll
        for (int q = 0; q < kSW; ++q) {
            if (phase == 0) {
                const int f = rank * per0 + gi * 2 + (q & 1);
                const bool in = f < min(I, (rank + 1) * per0);
                w[q] = load_w((q < 2 ? p.wg : p.wu) + (e * I + (in ? f : 0)) * (size_t)d, in, c, d);
            } else {
                const int col = rank * per1 + gi * kSW + q;
                const bool in = col < min(d, (rank + 1) * per1);
                w[q] = load_w(p.wd + (e * d + (in ? col : 0)) * (size_t)I, in, c, I);
            }
        }
    };
    float4 w[kSW], nxt[kSW];
    const int n0 = max(0, min(I, (rank + 1) * per0) - rank * per0), n1 = max(0, min(d, (rank + 1) * per1) - rank * per1);
    if (warp * 2 < n0) load_item(0, warp, 0, nxt);  // the first weights before the tokens, whose addresses take a round trip
    for (int t = warp; t < kSR; t += kWarps) {
        const float* src = p.x + (t < rows ? (kRoutes ? (int64_t)rs.tok[t] : token_of(p, row0 + t)) : 0) * d;
        for (int k = lane * 4; k < xld; k += 128)
            *reinterpret_cast<float4*>(xs + t * xld + k) = load4<VEC>(src + k, t < rows ? d - k : 0);
    }
    for (int i = threadIdx.x; i < kSR * (hld - I); i += kThreads)  // columns past I: read by the last chunk
        hs[i / (hld - I) * hld + I + i % (hld - I)] = 0.f;
    __syncthreads();
    bool started = kRoutes;

#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
        const int K = phase == 0 ? d : I, nc = (K + 127) / 128;
        const int groups = phase == 0 ? (n0 + 1) / 2 : (n1 + kSW - 1) / kSW;
        const float* ts = phase == 0 ? xs : hs;
        const int tld = phase == 0 ? xld : hld;
        if (phase == 1) {
            if (warp < groups) load_item(1, warp, 0, nxt);
            if (!started) cluster.barrier_wait();
            grid_dep_launch();  // not earlier: the next kernel's CTAs would only take this grid's places
            cluster.sync();     // every CTA's share of H is in every copy
        }
#pragma unroll 1
        for (int gi = warp; gi < groups; gi += kWarps) {
            float acc[kSW * kSR];
#pragma unroll
            for (int i = 0; i < kSW * kSR; ++i) acc[i] = 0.f;
#pragma unroll 1
            for (int c = 0; c < nc; ++c) {
#pragma unroll
                for (int q = 0; q < kSW; ++q) w[q] = nxt[q];
                const bool last = c + 1 == nc;
                if (!last || gi + kWarps < groups) load_item(phase, last ? gi + kWarps : gi, last ? 0 : c + 1, nxt);
#pragma unroll
                for (int t = 0; t < kSR; ++t) {
                    const float4 x = load_t(ts + t * tld, c);
#pragma unroll
                    for (int q = 0; q < kSW; ++q) {
                        float a = acc[q * kSR + t];
                        a = fmaf(w[q].x, x.x, a);
                        a = fmaf(w[q].y, x.y, a);
                        a = fmaf(w[q].z, x.z, a);
                        acc[q * kSR + t] = fmaf(w[q].w, x.w, a);
                    }
                }
            }
            lane_sums<32, 16>(acc, lane);
            const int t = lane & 7, q = lane >> 3;  // this lane's sum: weight row q of the group, token t
            if (phase == 0) {
                if (!started) {
                    cluster.barrier_wait();
                    started = true;
                }
                // lanes 0-15 hold gate, 16-31 up of the same (feature, token): both compute, each writes to half of the CTAs
                const float other = __shfl_xor_sync(0xffffffffu, acc[0], 16);
                const float h = lane < 16 ? swiglu(acc[0], other) : swiglu(other, acc[0]);
                const int fl = gi * 2 + (q & 1);
                if (fl < n0)
#pragma unroll
                    for (int c = 0; c < CL / 2; ++c)
                        cluster.map_shared_rank(hs, c + (lane < 16 ? 0 : CL / 2))[t * hld + rank * per0 + fl] = h;
            } else if (gi * kSW + q < n1 && t < rows) {
                const int col = rank * per1 + gi * kSW + q;
                if (p.y != nullptr) p.y[(int64_t)(kRoutes ? rs.tok[t] : p.row_tok[row0 + t]) * d + col] = (kRoutes ? rs.rw[t] : p.row_w[row0 + t]) * acc[0];
                else p.out[(row0 + t) * d + col] = acc[0];
            }
        }
    }
}

// ---------------------------------------------------------------- tall tiles
// k steps wk, wk + nk, ... of one chunk (8 steps of 4): part = products of the chunk, acc += part
template <int TM, int NW>
__device__ __forceinline__ void mac_chunk(const float* ws, const float* xs, int x_pitch, int wk, int nk,
                                          float (&acc)[TM][NW]) {
    float part[TM][NW];
#pragma unroll
    for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int q = 0; q < NW; ++q) part[r][q] = 0.f;
#pragma unroll 2
    for (int st = wk; st < kKC / 4; st += nk) {
        float4 w[NW], x[TM];
#pragma unroll
        for (int q = 0; q < NW; ++q) w[q] = *reinterpret_cast<const float4*>(ws + q * 8 * kLd + st * 4);
#pragma unroll
        for (int r = 0; r < TM; ++r) x[r] = *reinterpret_cast<const float4*>(xs + r * 4 * x_pitch + st * 4);
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int q = 0; q < NW; ++q) {
                part[r][q] = fmaf(w[q].x, x[r].x, part[r][q]);
                part[r][q] = fmaf(w[q].y, x[r].y, part[r][q]);
                part[r][q] = fmaf(w[q].z, x[r].z, part[r][q]);
                part[r][q] = fmaf(w[q].w, x[r].w, part[r][q]);
            }
    }
#pragma unroll
    for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int q = 0; q < NW; ++q) acc[r][q] += part[r][q];
}

template <int CL, int TM, int NW, int RW, bool VEC>
__global__ void __launch_bounds__(kThreads, 2) ffn_f32_tall_kernel(FfnF32Params p) {
    constexpr int BM = 4 * TM * RW;              // rows of the tile
    constexpr int kAcross = 8 / RW;              // warps along the features and along K
    constexpr int WR = kAcross * 8 * NW;         // weight rows of a stage, at most
    constexpr int kStage = (WR + BM) * kLd;      // floats
    constexpr int SR = WR / 32;                  // weight rows a thread copies per chunk, at most
    static_assert(TM * NW * kThreads <= 2 * kStage, "partial sums fit the stages");
    static_assert(BM <= 32, "one token row per staging thread");
    extern __shared__ __align__(16) float smem[];
    __shared__ Tile s_tile;
    float* hs = smem + 2 * kStage;  // [tile_rows][hld]: this CTA's slice of H
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lr = lane >> 3, lf = lane & 7, wr = warp / kAcross, wa = warp % kAcross;
    const int d = p.d, I = p.I, fpc = p.fpc, hld = p.hld;
    grid_dep_wait();
    if (!find_tile(p, (int)(blockIdx.x / CL), &s_tile)) return;  // the whole cluster
    const int rows = s_tile.rows;
    const int64_t row0 = s_tile.row0;
    const size_t e = s_tile.expert;

    // What this thread copies in every chunk, fixed for a pass: SR weight rows of the stage and one token row, from
    // w_src / x_src on, w_len / x_len floats ahead of it in the first chunk (none for rows that are not there)
    const int vk = (threadIdx.x & 7) * 4, vr = threadIdx.x >> 3;  // 32 rows of 8 vectors per sweep
    const bool x_in = vr < BM && vr < rows;
    const float* w_src[SR];
    int w_len[SR];
    const float* x_src = x_in ? p.x + token_of(p, row0 + vr) * d + vk : p.x;
    const int x_len = x_in ? d - vk : 0;

#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
        if (phase == 1) {
            grid_dep_launch();  // not earlier: the next kernel's CTAs would only take this grid's places
            cluster.sync();     // every slice of H is in place
        }
        // phase 0: H[:, rank's features] = silu(x W_gate^T) * (x W_up^T); phase 1: out[:, rank's columns] = H W_down^T
        const int K = phase == 0 ? d : I, per = phase == 0 ? fpc : (d + CL - 1) / CL;
        const int lo = rank * per, hi = min(phase == 0 ? I : d, lo + per);
        // A power of two of warps (n_wf) lies along the stage's weight rows, the others split K; afterwards the warps with
        // wk == 0 hold the sums of token rows wr * 4 TM + 4 r + lr and stage rows wf * 8 NW + 8 q + lf.
        int n_wf = 1;
        while (n_wf < kAcross && n_wf * 8 * NW < (phase == 0 ? 2 : 1) * (hi - lo)) n_wf *= 2;
        const int wf = wa & (n_wf - 1), wk = wa / n_wf, nk = kAcross / n_wf, n_rows = n_wf * 8 * NW;
        const int step = phase == 0 ? n_rows / 2 : n_rows;  // features (a gate and an up row each) or columns per pass
        const int nc = (K + kKC - 1) / kKC;
#pragma unroll 1
        for (int f0 = lo; f0 < hi; f0 += step) {
#pragma unroll
            for (int q = 0; q < SR; ++q) {  // a warp's stage rows in phase 0: 4 NW gate rows, then the same features' up rows
                const int r = vr + 32 * q, in_warp = r % (8 * NW);
                const int f = phase == 0 ? f0 + r / (8 * NW) * (4 * NW) + in_warp % (4 * NW) : f0 + r;
                const float* base = phase == 1 ? p.wd : (in_warp < 4 * NW ? p.wg : p.wu);
                const bool in = r < n_rows && f < hi;
                w_src[q] = base + (e * (size_t)(phase == 0 ? I : d) + (in ? f : 0)) * K + vk;
                w_len[q] = in ? K - vk : 0;
            }
            float4 wv[SR], xv;
            auto load = [&](int c) {
#pragma unroll
                for (int q = 0; q < SR; ++q) wv[q] = load4<VEC>(w_src[q] + c * kKC, w_len[q] - c * kKC);
                if (phase == 0) {
                    xv = load4<VEC>(x_src + c * kKC, x_len - c * kKC);
                } else {
                    // a chunk lies in one CTA's slice (fpc is a multiple of 32); features past I (never written) are zero
                    xv = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (x_in) {
                        const int owner = (c * kKC) / fpc, k = c * kKC + vk;
                        xv = *reinterpret_cast<const float4*>(cluster.map_shared_rank(hs, owner) + vr * hld + (k - owner * fpc));
                        if (k >= I) xv.x = 0.f;
                        if (k + 1 >= I) xv.y = 0.f;
                        if (k + 2 >= I) xv.z = 0.f;
                        if (k + 3 >= I) xv.w = 0.f;
                    }
                }
            };
            auto store = [&](float* st) {
#pragma unroll
                for (int q = 0; q < SR; ++q) *reinterpret_cast<float4*>(st + (vr + 32 * q) * kLd + vk) = wv[q];
                if (vr < BM) *reinterpret_cast<float4*>(st + (WR + vr) * kLd + vk) = xv;
            };
            float acc[TM][NW];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int q = 0; q < NW; ++q) acc[r][q] = 0.f;
            load(0);
            __syncthreads();  // the previous pass is done with the stages
            store(smem);
#pragma unroll 1
            for (int c = 0; c < nc; ++c) {
                __syncthreads();  // chunk c is in place; chunk c - 1, whose stage takes chunk c + 1, is used up
                if (c + 1 < nc) load(c + 1);
                const float* ws = smem + (c & 1) * kStage;
                mac_chunk<TM, NW>(ws + (wf * 8 * NW + lf) * kLd, ws + (WR + wr * 4 * TM + lr) * kLd, kLd, wk, nk, acc);
                if (c + 1 < nc) store(smem + ((c + 1) & 1) * kStage);
            }
            if (nk > 1) {  // partial sums of the K parts, added in order
                __syncthreads();
                float* red = smem + (wr * kAcross + wa) * (TM * NW * 32) + lane;
                if (wk > 0)
#pragma unroll
                    for (int i = 0; i < TM * NW; ++i) red[i * 32] = acc[i / NW][i % NW];
                __syncthreads();
                if (wk == 0)
#pragma unroll 1
                    for (int k = 1; k < nk; ++k)
#pragma unroll
                        for (int i = 0; i < TM * NW; ++i) acc[i / NW][i % NW] += red[(k * n_wf * TM * NW + i) * 32];
            }
            if (wk != 0) continue;
#pragma unroll
            for (int r = 0; r < TM; ++r) {
                const int row = (wr * TM + r) * 4 + lr;
                if (phase == 0) {
#pragma unroll
                    for (int q = 0; q < NW / 2; ++q) {
                        const int f = f0 + wf * 4 * NW + q * 8 + lf;
                        if (f < lo + fpc && row < p.tile_rows) hs[row * hld + f - lo] = swiglu(acc[r][q], acc[r][q + NW / 2]);
                    }
                } else if (row < rows) {
                    const float w = p.y != nullptr ? p.row_w[row0 + row] : 1.0f;
                    float* dst = p.y != nullptr ? p.y + (int64_t)p.row_tok[row0 + row] * d : p.out + (row0 + row) * d;
#pragma unroll
                    for (int q = 0; q < NW; ++q) {
                        const int c = f0 + (wf * NW + q) * 8 + lf;
                        if (c < hi) dst[c] = p.y != nullptr ? w * acc[r][q] : acc[r][q];
                    }
                }
            }
        }
    }
    cluster.sync();  // no CTA leaves while another may still read its slice of H
}

constexpr size_t kSmemLimit = 227 * 1024 - 1024;
int features_per_cta(int I, int cl) { return ((I + cl - 1) / cl + kKC - 1) / kKC * kKC; }
size_t short_bytes(int d, int I) { return (size_t)kSR * ((d + 127) / 128 * 128 + (I + 127) / 128 * 128 + 4) * sizeof(float); }
// CTAs of the short form that run at once, of `bytes` of shared memory each: two to an SM (what their registers allow) while an SM
// holds twice the memory (d + I up to 3580, 3130 where decode is routed in it), else one; in clusters of eight some nine tenths
int64_t short_wave(size_t bytes, int sms) { return (int64_t)sms * (2 * (bytes + 1024) <= 228 * 1024 ? 184 : 92) / 100; }
size_t tall_bytes(int tile_rows, int I, int cl) {  // two stages of 128 weight rows and the form's token rows, then the slice of H
    const int form_rows = tile_rows > 16 ? 32 : 16;
    return ((size_t)2 * (128 + form_rows) * kLd + (size_t)tile_rows * (features_per_cta(I, cl) + 4)) * sizeof(float);
}

template <int CL, typename K, typename... Args>
cudaError_t launch_t(K kernel, size_t smem, int64_t tiles, cudaStream_t s, const Args&... args) {
    cudaError_t err = ensure_smem(kernel, smem);
    if (err != cudaSuccess) return err;
    return launch_pdl_cluster(kernel, (unsigned)(tiles * CL), kThreads, smem, CL, s, args...);
}
template <int CL, bool VEC>
cudaError_t launch_form(FfnF32Params p, int64_t tiles, cudaStream_t s) {
    if (p.tile_rows == kSR && short_bytes(p.d, p.I) <= kSmemLimit) {
        p.hld = (p.I + 127) / 128 * 128 + 4;
        return launch_t<CL>(ffn_f32_short_kernel<CL, VEC, NoRoute, 0>, short_bytes(p.d, p.I), tiles, s, p, NoRoute{});
    }
    p.fpc = features_per_cta(p.I, CL);
    p.hld = p.fpc + 4;
    const size_t smem = tall_bytes(p.tile_rows, p.I, CL);
    if (p.tile_rows > 16) return launch_t<CL>(ffn_f32_tall_kernel<CL, 4, 4, 2, VEC>, smem, tiles, s, p);
    return launch_t<CL>(ffn_f32_tall_kernel<CL, 4, 2, 1, VEC>, smem, tiles, s, p);
}
bool vec_loads(const FfnF32Params& p) {
    auto a16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    return p.I % 4 == 0 && a16(p.x) && a16(p.wg) && a16(p.wu) && a16(p.wd);
}
template <bool VEC, typename R>
cudaError_t launch_routed(FfnF32Params p, const R& rt, int N, int64_t tiles, cudaStream_t s) {
    p.hld = (p.I + 127) / 128 * 128 + 4;
    if (N <= 32) return launch_t<kMaxCl>(ffn_f32_short_kernel<kMaxCl, VEC, R, 1>, short_bytes(p.d, p.I), tiles, s, p, rt);
    return launch_t<kMaxCl>(ffn_f32_short_kernel<kMaxCl, VEC, R, 4>, short_bytes(p.d, p.I), tiles, s, p, rt);
}
template <int CL>
cudaError_t launch_cl(const FfnF32Params& p, int64_t tiles, cudaStream_t s) {
    return vec_loads(p) ? launch_form<CL, true>(p, tiles, s) : launch_form<CL, false>(p, tiles, s);
}

// y[i][c] = sum_j w(row) out[row][c] over the token's rows in slot order (row = inv_pos[i][j], -1: merged into an earlier
// slot), plus the shared expert's row
__global__ void __launch_bounds__(128) combine_f32_kernel(const float* __restrict__ out, const int32_t* __restrict__ inv_pos,
                                                          const float* __restrict__ row_w, int64_t Tn, int Kr, int d,
                                                          int n_shared, const int32_t* __restrict__ shared0_dev,
                                                          float* __restrict__ y) {
    const int64_t i = blockIdx.x;
    grid_dep_launch();
    grid_dep_wait();
    const int64_t shared0 = shared0_dev != nullptr ? (int64_t)*shared0_dev : Tn * Kr;
    for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4) {  // d is a multiple of 4
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int j = 0; j < Kr; ++j) {
            const int row = inv_pos[i * Kr + j];
            if (row < 0) continue;
            const float w = row_w[row];
            const float4 v = *reinterpret_cast<const float4*>(out + (size_t)row * d + c);
            acc.x = fmaf(w, v.x, acc.x);
            acc.y = fmaf(w, v.y, acc.y);
            acc.z = fmaf(w, v.z, acc.z);
            acc.w = fmaf(w, v.w, acc.w);
        }
        if (n_shared) {
            const float4 v = *reinterpret_cast<const float4*>(out + (size_t)(shared0 + i) * d + c);
            acc.x += v.x;
            acc.y += v.y;
            acc.z += v.z;
            acc.w += v.w;
        }
        *reinterpret_cast<float4*>(y + i * d + c) = acc;
    }
}

}  // namespace

static int64_t short_tiles(int64_t rows, int G) { return std::min<int64_t>(rows, rows / kSR + G); }  // at most

// Rows per tile: a tile computes all of its rows, so short groups want short tiles (and more of them to fill the SMs); a
// tile's weights are read once per tile, so long groups want long ones. The short form is the faster one for as long as its
// tiles are a few waves of clusters at most: five where the alternative is 16-row tiles or the layer is small, else three (counted
// with the K chunks that sizes between multiples of 128 compute in vain). Whole call with tall / short tiles: tiny layer prefill (K' = 1)
// 75 tokens 20.3 / 12.0 us, 342 23.5 / 19.4, 509 35.0 / 22.8, (K' = 2) 456 40.4 / 28.3, 770 (6 waves) 34.6 / 39.2; decode of 116
// tokens, pool of 3 35.2 / 21.9; 28 experts of 320 x 960, 41 tokens, pool of 8 85 / 53; 9 of 384 x 736, 79 tokens 85 / 60; 8 of
// 2048 x 1536, 293 tokens (1.3 waves) 491 / 458; 8 + 1 of 160 x 480, 204 tokens x 2 (4.3 waves) 47.7 / 53.3; 30 + 1 of 96 x 128, 871
// tokens (K' = 3, 13 waves) 39 / 56.
// Where an SM holds one such CTA only, a wave is half as many tiles and a second one as long as a wave of 16-row tiles and a half: one
// wave, two where the alternative is 32 rows. 8 experts of 2048 x 2048, 16 tiles 623 / 299, 22 tiles 438 / 523, 28 434 / 535; of 1024 x
// 4096, 22 tiles 441 / 560; 2 of 2048 x 2048, 93 rows each 629 / 500, 6 of 1024 x 4096, 63 each (53 tiles) 637 / 958.
// Short tiles need the tokens and H in shared memory whole (d + I up to ~7000); tall ones are halved while the slice of H does not
// fit (32 rows: I above ~11 000).
int ffn_f32_tile_rows(int64_t rows, int G, int d, int I, int sms) {
    const size_t bytes = short_bytes(d, I);
    const bool rows16 = rows <= (int64_t)48 * G;  // else the alternative is 32
    if (bytes <= kSmemLimit) {
        if (rows <= (int64_t)kSR * G) return kSR;
        const int64_t wave = short_wave(bytes, sms);
        const int waves = wave < sms ? (rows16 ? 1 : 2) : (rows16 || (int64_t)d * I <= 48 * 1024 ? 5 : 3);
        const int64_t computed = (int64_t)((d + 127) / 128 * 128) * ((I + 127) / 128 * 128);  // K chunks are computed whole
        if (short_tiles(rows, G) * kMaxCl * computed <= wave * waves * d * I) return kSR;
    }
    int tile_rows = rows16 ? 16 : 32;
    while (tile_rows > 1 && tall_bytes(tile_rows, I, kMaxCl) > kSmemLimit) tile_rows /= 2;
    return tile_rows;
}

// CTAs per row tile. Two CTAs share an SM, so that clusters run in waves (fragmented by the chip's partitions to some nine
// tenths; a last wave that is nearly empty costs half of one), each of which takes a fixed 8 us and, in proportion to a CTA's
// share of the layer, 0.28 + 0.037 per row and weight row of 1000: few tiles want eight CTAs each, many tiles of a small
// layer fewer, in fewer waves. The tiles are estimated from the rows (over as many groups as random rows meet). Whole prefill
// call with 8, 4 and 2 CTAs, and with one CTA per route before there were row tiles: 195 experts of 64 x 64, 943 tokens x 3
// 78.4, 46.7, 32.5, 67.8 us; 60 of 128 x 256, 500 x 4 85.9, 64.7, 52.4, 123.3; 60 of 512 x 512 255.8, 260.9, 283.1, 795.8; 16 of
// 128 x 256, 64 x 2 17.1, 18.9, 23.1, 42.1. Over 90 shapes of 64 x 64 to 1024 x 2048 and 12 to 371 tiles the choice is 3.1 %
// above the best of the three, 11 % below eight CTAs always.
static int cluster_ctas(int64_t rows, int64_t tiles, const FfnF32Params& p, int sms) {
    const double r = (double)rows, used = p.G * (1.0 - std::exp(-r / p.G));  // groups with a row
    const double est = std::min((double)tiles, std::max(used, r / p.tile_rows + used / 2));
    const double share = (double)p.d * p.I * (0.28 + 0.037 * p.tile_rows) / 1000.0;
    int best = kMaxCl;
    double best_t = 1e30;
    for (int cl = kMaxCl; cl >= 2; cl /= 2) {
        if (cl < kMaxCl && tall_bytes(p.tile_rows, p.I, cl) > kSmemLimit) break;
        const double x = est * cl / (1.84 * sms), t = (x <= 1.0 ? 1.0 : 0.5 * (std::ceil(x) + x + 0.3)) * (8.0 + share / cl);
        if (t < 0.9 * best_t) {  // fewer only for a clear gain
            best_t = t;
            best = cl;
        }
    }
    return best;
}

cudaError_t launch_ffn_f32(const FfnF32Params& p, int64_t rows, int sms, cudaStream_t s) {
    if (rows == 0) return cudaSuccess;
    const int64_t tiles = std::min<int64_t>(rows, rows / p.tile_rows + p.G);
    const int cl = cluster_ctas(rows, tiles, p, sms);
    return cl == 8 ? launch_cl<8>(p, tiles, s) : (cl == 4 ? launch_cl<4>(p, tiles, s) : launch_cl<2>(p, tiles, s));
}

// One wave of clusters (each repeats the routing), and the routes of all tokens in shared memory. (8 + 1 experts of 2048 x 1536, 93
// tokens, 32 tiles: the state leaves one CTA to an SM, two waves, 402 us; lists from kernels of their own and two CTAs 273)
bool ffn_f32_routes(bool decode, int64_t T, int64_t rows, int G, int N, int slots, int d, int I, int tile_rows, int sms) {
    const size_t bytes = short_bytes(d, I) + (decode ? sizeof(DecodeRouteSmem) : sizeof(PrefillRouteSmem)) + 256;
    return tile_rows == kSR && bytes <= kSmemLimit && T <= kRoutedTokens && T * slots <= kRoutedSlots && N <= kRoutedExperts &&
           short_tiles(rows, G) * kMaxCl <= short_wave(bytes, sms);
}
cudaError_t launch_ffn_f32_routed(const FfnF32Params& p, const FfnF32Route& rt, int64_t rows, cudaStream_t s) {
    const int64_t tiles = short_tiles(rows, p.G);
    return vec_loads(p) ? launch_routed<true>(p, rt, rt.r.N, tiles, s) : launch_routed<false>(p, rt, rt.r.N, tiles, s);
}
cudaError_t launch_ffn_f32_routed(const FfnF32Params& p, const DecodeRouteParams& rt, int64_t rows, cudaStream_t s) {
    const int64_t tiles = short_tiles(rows, p.G);
    return vec_loads(p) ? launch_routed<true>(p, rt, rt.N, tiles, s) : launch_routed<false>(p, rt, rt.N, tiles, s);
}

cudaError_t launch_combine_f32(const float* out, const int32_t* inv_pos, const float* row_w, int64_t T, int Kr, int d,
                               int n_shared, const int32_t* shared0_dev, float* y, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    return launch_pdl(combine_f32_kernel, (unsigned)T, 128, 0, s, out, inv_pos, row_w, T, Kr, d, n_shared, shared0_dev, y);
}

}  // namespace exfold
