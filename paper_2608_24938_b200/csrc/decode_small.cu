// Decode of small batches (bf16 layers, at most 8 tokens): routing, expert pool and expert FFN in two kernels. Prefill calls
// of at most 8 tokens run the same two on the routes that the prefill routing kernel left.
//
// A small batch reads the weights of a few experts and does next to no arithmetic on them, so its time is the weights'
// bytes over HBM plus every fixed cost on the way. The four-kernel chain of larger batches (route_decode.cu,
// ffn_decode.cu, the grouped down projection, the per-token sum) pays for four dependent launches, for 128-row tensor
// tiles of which a row or two is used, and for few work items (8 experts x 768 features: 96 of 148 SMs stream). Here
//
//   gate/up kernel  every CTA takes the tokens' Top-K (a warp per token), the pool (Eq. 11), targets (Eq. 12) and the remap
//       (Eq. 14) itself from the router scores, then streams its share of the pool's gate and up weights against the
//       tokens and writes the compact rows of H; the first weights are requested as soon as the pool is known;
//   down kernel     streams W_down for 16 output columns per work item over ALL experts of the pool, so a token's experts
//       are added in registers in fp32 and y is written once: no per-expert rows, no separate sum.
//
// Weights go from global memory straight into the fragments of mma.sync m16n8k16: a lane loads 32 contiguous bytes of a
// weight row (4 lanes a whole 128-byte line), and since the K order inside a product does not matter, those 16 elements
// serve as the lane's K positions of four MMAs while the tokens, the 8-column operand, use the same order. A work item
// is 16 weight rows (gate/up: 8 features' gate rows and up rows, so that SwiGLU needs no exchange); the warps of a CTA
// split K and meet in shared memory. Two 64-wide K chunks per warp are in flight while the previous two are multiplied:
// 16 warps x 4 KB per SM, ~25 bytes per cycle and SM at the loaded HBM latency, which is HBM's rate. The legacy matrix
// instruction suffices: at 48 GB/s of weights per SM it is busy a few percent of the time.
//
// Measured, four-kernel chain -> this (whole call): Qwen3 shape, 1 token 33.2 -> 21.4 us, 8 tokens with a pool of 32 53.8 -> 44.9;
// Mixtral shape, 1 token 167 -> 124 (5.7 TB/s); GLM shape, 8 tokens with a pool of 32 213 -> 201.
// Prefill of 1 token 38.7 -> 18.8 (Mixtral shape 220 -> 126), of 8 tokens (Top-6, router) 96 -> 82. With two 8-column operands,
// a decode of 16 tokens took 57 us against the chain's 42 (the per-CTA routing grows with the tokens), so the line is at 8.
#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"
#include "route_token.cuh"

#include <cooperative_groups.h>

namespace exfold {

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;  // gate/up kernel, two CTAs per SM
constexpr int kWarps = kThreads / 32;
constexpr int kMaxDownWarps = 16;
constexpr int kKC = 64;     // K elements per chunk: one 128-byte line of a weight row
constexpr int kUnroll = 2;  // chunks per stage
constexpr int kTB = kSmallDecodeBatch;
static_assert(kTB == 8, "the tokens are the 8 columns of the MMA, and the 8 warps rank one each");

// 32 bytes of weights, read once: not kept in L1
__device__ __forceinline__ void ld_stream(uint32_t (&r)[8], const __nv_bfloat16* p) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "l"(p));
}
__device__ __forceinline__ void ld_rows(uint32_t (&r)[8], const __nv_bfloat16* p) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void zero8(uint32_t (&r)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = 0u;
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// One 64-wide K chunk: lo / hi = this lane's 16 elements of weight rows (lane / 4) and (lane / 4) + 8, b = of token lane / 4
__device__ __forceinline__ void mma_chunk(float (&c)[4], const uint32_t (&lo)[8], const uint32_t (&hi)[8], const uint32_t (&b)[8]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) mma_bf16(c, lo[2 * i], hi[2 * i], lo[2 * i + 1], hi[2 * i + 1], b[2 * i], b[2 * i + 1]);
}
__device__ __forceinline__ void add4(float4& s, const float4& v) {
    s.x += v.x;
    s.y += v.y;
    s.z += v.z;
    s.w += v.w;
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}

struct SmallState {  // routing state of the batch, one copy per CTA
    long long key[kMaxExperts];       // by union member: order-preserving integer image of its score
    unsigned acc32[3 * kMaxExperts];  // by expert: sum_i w_{i,e} in 2^-53 units, as three 21-bit limbs
    int in_union[kMaxExperts];
    int member[kMaxExperts];          // the batch's experts, ascending
    int rank[kMaxExperts];            // by union member: pool rank (the choice when the union exceeds M; metadata)
    int grp_of[kMaxExperts];          // by expert: group or -1
    int target[kMaxExperts];
    float scale[kMaxExperts];
    int grp[kMaxGroups];              // expert of each group: the pool's experts, ascending; the shared expert (N) last
    unsigned mask[kMaxGroups];        // tokens that each group serves
    int off[kMaxGroups];              // first compact row of each group
    int warp_cnt[2][kWarps];
    int G, rows;
};
constexpr int kStateBytes = (int)((sizeof(SmallState) + 15) / 16 * 16);
constexpr int kXPad = 8;  // elements between token rows: the two token rows a quarter warp reads lie in distinct banks

// Positions of the threads with `flag` in thread order (all threads call; list is readable after the next barrier):
// list[pos] = tid. Returns the count.
__device__ __forceinline__ int compact_threads(bool flag, int* warp_cnt, int* list, int* pos_out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    if (lane == 0) warp_cnt[warp] = __popc(m);
    __syncthreads();
    int base = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const int c = warp_cnt[w];
        if (w < warp) base += c;
        all += c;
    }
    *pos_out = base + __popc(m & ((1u << lane) - 1u));
    if (flag) list[*pos_out] = (int)threadIdx.x;
    return all;
}

// GIVEN: prefill, the routes and their weights are final (or found here, a token per warp, as prefill does); else Top-K, pool and
// remap happen here
struct NoRoute {};
template <bool GIVEN, typename R>  // R: PrefillRouteParams where the kernel routes prefill tokens (an argument that decode does without)
__global__ void __launch_bounds__(kThreads, 2) decode_small_gateup_kernel(DecodeSmallParams p, R route) {
    constexpr bool kRoutes = sizeof(R) > sizeof(NoRoute);
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ float4 s_red[2][kWarps][32];
    SmallState& sc = *reinterpret_cast<SmallState*>(smem);
    const int B = p.B, N = p.N, K = p.K, BK = B * K, d = p.d, I = p.I;
    double* w64 = reinterpret_cast<double*>(smem + kStateBytes);   // [B * K]
    int* ids = reinterpret_cast<int*>(w64 + BK);                    // [B * K] routed experts, then remapped ones
    float* wrm = reinterpret_cast<float*>(ids + BK);                // [B * K] remapped weights
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(smem + kStateBytes + align16((size_t)BK * 16));  // [B][d + pad]
    const int xld = d + kXPad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool is_static = !GIVEN && p.st_pool != nullptr;
    // the CTA with the fewest work items writes the metadata and the lists
    const bool scribe = blockIdx.x == gridDim.x - 1, meta = !GIVEN && p.pool_ids != nullptr && scribe;
    sc.acc32[3 * tid] = sc.acc32[3 * tid + 1] = sc.acc32[3 * tid + 2] = 0u;
    sc.in_union[tid] = 0;
    sc.grp_of[tid] = -1;
    for (int g = tid; g < kMaxGroups; g += kThreads) sc.mask[g] = 0u;
    grid_dep_wait();
    if (p.status != nullptr && scribe && tid < 4) reinterpret_cast<int*>(p.status)[tid] = 0;

    // ---- Eq. 2: a warp per token (or the result of the top-k kernel when that computed the scores)
    float v[8];
    const float* logits = p.logits;
    if constexpr (kRoutes) logits = route.logits;
    const bool ranks = (kRoutes || !GIVEN) && logits != nullptr && warp < B;
    if (ranks) {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = lane + 32 * q < N ? logits[(size_t)warp * N + lane + 32 * q] : -INFINITY;
    }
    // not before the wait: the caller may have written the table on this stream right before the call
    const float h_e = !GIVEN && !is_static && tid < N ? __ldg(p.h + tid) : 0.f;
    for (int t = 0; t < B; ++t)  // lands while the routing below runs
        for (int c = tid * 8; c < d; c += kThreads * 8) cp_async16(xs + t * xld + c, p.x + (size_t)t * d + c);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if constexpr (kRoutes) {
        if (ranks) {
            const TokenRoute r = route_token<8>(route, v, lane);
            if (r.kept) {
                ids[warp * K + r.rank] = r.id;
                wrm[warp * K + r.rank] = r.w;
            }
        }
    } else if (!GIVEN && ranks) {
        int id;
        const double w = warp_topk_softmax<8>(v, N, K, lane, &id);
        if (lane < K) {
            ids[warp * K + lane] = id;
            w64[warp * K + lane] = w;
        }
    }
    if ((GIVEN && !kRoutes) || logits == nullptr)
        for (int s = tid; s < BK; s += kThreads) {
            ids[s] = p.ids[s];
            if (GIVEN) wrm[s] = p.w_in[s];
            else w64[s] = p.w64[s];
        }
    __syncthreads();

    // ---- Eq. 11: weights summed per expert in 2^-53 fixed point (three 21-bit limbs: exact, order-independent)
    int U = 0, P;  // union size, pool size
    if (is_static) {
        if (tid < N) {
            sc.target[tid] = p.st_target[tid];
            sc.scale[tid] = p.st_scale[tid];
        }
        if (tid < p.M) sc.in_union[p.st_pool[tid]] = 1;  // here: the pool
        __syncthreads();
        const bool pooled = sc.in_union[tid] != 0;
        int g;
        P = compact_threads(pooled, sc.warp_cnt[0], sc.grp, &g);
        if (pooled) sc.grp_of[tid] = g;
    } else {
        for (int s = tid; s < BK; s += kThreads) {
            const int e = ids[s];
            sc.in_union[e] = 1;
            if (GIVEN) continue;
            const unsigned long long fx = (unsigned long long)(w64[s] * 9007199254740992.0);
            atomicAdd(&sc.acc32[3 * e], (unsigned)(fx & 0x1FFFFFull));
            atomicAdd(&sc.acc32[3 * e + 1], (unsigned)((fx >> 21) & 0x1FFFFFull));
            atomicAdd(&sc.acc32[3 * e + 2], (unsigned)(fx >> 42));
        }
        __syncthreads();
        const bool is_member = sc.in_union[tid] != 0;
        int mine;
        U = compact_threads(is_member, sc.warp_cnt[0], sc.member, &mine);
        bool pooled = is_member;
        if (!GIVEN && (U > p.M || p.pool_ids != nullptr)) {
            // pool = best M experts of the union by (score desc, id asc): rank by counting over the members
            if (is_member) {
                const unsigned long long acc = (unsigned long long)sc.acc32[3 * tid] +
                                               ((unsigned long long)sc.acc32[3 * tid + 1] << 21) +
                                               ((unsigned long long)sc.acc32[3 * tid + 2] << 42);
                sc.key[mine] = score_order_key((double)acc * (1.0 / 9007199254740992.0) * (double)h_e);
            }
            __syncthreads();
            int lanes = 32;  // threads per member
            while (lanes > 1 && U * lanes > kThreads) lanes >>= 1;
            const int i = tid / lanes, sub = tid & (lanes - 1);
            int better = 0;
            if (i < U) {
                const long long ki = sc.key[i];
                for (int o = sub; o < U; o += lanes) {
                    const long long ko = sc.key[o];
                    better += (ko > ki || (ko == ki && o < i)) ? 1 : 0;  // members ascend, so position order is id order
                }
            }
            for (int o = lanes >> 1; o > 0; o >>= 1) better += __shfl_xor_sync(0xffffffffu, better, o);
            if (i < U && sub == 0) sc.rank[i] = better;
            __syncthreads();
            pooled = is_member && sc.rank[mine] < p.M;
        }
        int g;
        P = compact_threads(pooled, sc.warp_cnt[1], sc.grp, &g);
        if (pooled) {
            sc.grp_of[tid] = g;
            sc.target[tid] = tid;
            sc.scale[tid] = 1.0f;
        }
    }
    if (tid == 0 && p.n_shared) {
        sc.grp[P] = N;
        sc.mask[P] = (1u << B) - 1u;
    }
    __syncthreads();

    // ---- gate/up: item = (group, 8 features). Every expert of a dynamic pool serves a token, so the first weights are
    // requested here and arrive while the remap below runs.
    const int fblocks = I / 8, nch = d / kKC;
    const int nst = (nch + kWarps * kUnroll - 1) / (kWarps * kUnroll);
    const int lr = lane >> 2, lk = (lane & 3) * 16;
    auto load = [&](int item, int st, uint32_t (&a)[kUnroll][2][8]) {
        const int g = item / fblocks, f = (item - g * fblocks) * 8 + lr;
        const size_t row = (size_t)sc.grp[g] * I + f;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int c = warp + kWarps * (st * kUnroll + u);
            if (c < nch) {
                ld_stream(a[u][0], p.wg + row * d + c * kKC + lk);
                ld_stream(a[u][1], p.wu + row * d + c * kKC + lk);
            }
        }
    };
    uint32_t nxt[kUnroll][2][8];
    int G = P + p.n_shared;
    if (!is_static && (int)blockIdx.x < G * fblocks) load(blockIdx.x, 0, nxt);

    if (!GIVEN && !is_static) {
        // Eq. 12 for the batch's experts outside the pool (all experts for the metadata): a warp per source, loss and
        // scalar of every candidate in one round trip, two sources at a time. A NaN loss is never smaller, but the
        // best-ranked expert's is where the search starts and stays.
        const int n_src = meta ? N : (U > P ? U : 0);
        for (int i0 = warp; i0 < n_src; i0 += 2 * kWarps) {
            int s2[2], bj[2];
            float bl[2], bs[2];
            unsigned nan = 0;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = i0 + u * kWarps;
                s2[u] = i < n_src ? (meta ? i : sc.member[i]) : -1;
                if (s2[u] >= 0 && sc.grp_of[s2[u]] >= 0) s2[u] = -1;  // in the pool: itself
                bl[u] = INFINITY;
                bs[u] = 0.f;
                bj[u] = 0x7fffffff;
                if (s2[u] >= 0)
                    for (int j = lane; j < P; j += 32) {
                        const int t = sc.grp[j];
                        const float l = __ldg(p.L + (size_t)s2[u] * N + t), sv = __ldg(p.S + (size_t)s2[u] * N + t);
                        nan |= isnan(l) ? 1u << u : 0u;
                        if (l < bl[u] || (l == bl[u] && t < bj[u])) {
                            bl[u] = l;
                            bs[u] = sv;
                            bj[u] = t;
                        }
                    }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (s2[u] < 0) continue;  // warp-uniform
                int bt = warp_argmin(bj[u] != 0x7fffffff, float_order_key(bl[u]), bj[u]);
                const unsigned who = __ballot_sync(0xffffffffu, bj[u] == bt);
                float scl = __shfl_sync(0xffffffffu, bs[u], __ffs(who) - 1);
                if (__any_sync(0xffffffffu, (nan >> u) & 1u)) {
                    int first = 0;
                    while (sc.rank[first] != 0) ++first;
                    first = sc.member[first];
                    if (isnan(__ldg(p.L + (size_t)s2[u] * N + first))) {
                        bt = first;
                        scl = __ldg(p.S + (size_t)s2[u] * N + first);
                    }
                }
                if (lane == 0) {
                    sc.target[s2[u]] = bt;
                    sc.scale[s2[u]] = scl;
                }
            }
        }
        __syncthreads();
    }
    // Eq. 14: every slot in place; tokens that each group serves
    for (int s = tid; s < BK; s += kThreads) {
        const int e = ids[s], t = GIVEN ? e : sc.target[e];
        atomicOr(&sc.mask[sc.grp_of[t]], 1u << (s / K));
        if (GIVEN) continue;
        const float wv = (float)(w64[s] * (double)sc.scale[e]);
        ids[s] = t;
        wrm[s] = wv;
        if (meta) {
            p.out_ids[s] = t;
            p.out_w[s] = wv;
        }
    }
    if (meta) {
        if (tid < N) {
            p.target[tid] = sc.target[tid];
            p.scale[tid] = sc.scale[tid];
            if (tid >= P) p.pool_ids[tid] = -1;
        }
        if (is_static) {
            if (tid < P) p.pool_ids[tid] = p.st_pool[tid];
        } else if (tid < U && sc.rank[tid] < p.M) {
            p.pool_ids[sc.rank[tid]] = sc.member[tid];
        }
        const unsigned m = __ballot_sync(0xffffffffu, sc.grp_of[tid] >= 0);
        if (lane == 0) p.pool_mask[warp] = m;
        if (tid == 0) *p.pool_size = P;
    }
    __syncthreads();
    if (warp == 0) {  // compact rows; groups of a static pool without rows are left out
        int carry = 0, n = 0;
        for (int g0 = 0; g0 < G; g0 += 32) {
            const int g = g0 + lane;
            const unsigned m = g < G ? sc.mask[g] : 0u;
            const int c = __popc(m), e = g < G ? sc.grp[g] : 0;
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            const unsigned some = __ballot_sync(0xffffffffu, c > 0);
            const int at = n + __popc(some & ((1u << lane) - 1u));
            __syncwarp();
            if (c > 0) {  // at <= g: never ahead of what is still to be read
                sc.grp[at] = e;
                sc.mask[at] = m;
                sc.off[at] = carry + incl - c;
            }
            __syncwarp();
            carry += __shfl_sync(0xffffffffu, incl, 31);
            n += __popc(some);
        }
        if (lane == 0) {
            sc.G = n;
            sc.rows = carry;
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // the tokens
    __syncthreads();
    G = sc.G;
    const int total = G * fblocks;
    if (scribe) {  // execution lists of the down kernel
        for (int i = tid; i < G * B; i += kThreads) {
            const int g = i / B, t = i - g * B, e = sc.grp[g];
            const unsigned m = sc.mask[g];
            if (!((m >> t) & 1u)) continue;
            float w = 1.0f;
            if (e < N) {  // slots with the same target merged, weights added in slot order
                bool has = false;
                for (int k = 0; k < K; ++k)
                    if (ids[t * K + k] == e) {
                        w = has ? __fadd_rn(w, wrm[t * K + k]) : wrm[t * K + k];
                        has = true;
                    }
            }
            const int row = sc.off[g] + __popc(m & ((1u << t) - 1u));
            p.row_tok[row] = t;
            p.row_w[row] = w;
            p.row_grp[row] = g;
        }
        for (int g = tid; g < G; g += kThreads) p.grp_expert[g] = sc.grp[g];
        if (tid == 0) {
            p.n_groups[0] = G;
            p.n_groups[1] = sc.rows;
        }
    }
    if (is_static && (int)blockIdx.x < total) load(blockIdx.x, 0, nxt);

    int par = 0;
    for (int item = blockIdx.x; item < total; item += gridDim.x, par ^= 1) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int st = 0; st < nst; ++st) {
            uint32_t cur[kUnroll][2][8];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    cur[u][0][i] = nxt[u][0][i];
                    cur[u][1][i] = nxt[u][1][i];
                }
            const bool last = st + 1 == nst;
            const int ni = last ? item + (int)gridDim.x : item;
            if (ni < total) load(ni, last ? 0 : st + 1, nxt);
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int c = warp + kWarps * (st * kUnroll + u);
                if (c >= nch) break;  // warp-uniform
                uint32_t b[8];
                if (lr < B) {
                    const uint4* src = reinterpret_cast<const uint4*>(xs + lr * xld + c * kKC + lk);
                    const uint4 v0 = src[0], v1 = src[1];
                    b[0] = v0.x; b[1] = v0.y; b[2] = v0.z; b[3] = v0.w;
                    b[4] = v1.x; b[5] = v1.y; b[6] = v1.z; b[7] = v1.w;
                } else {
                    zero8(b);
                }
                mma_chunk(acc, cur[u][0], cur[u][1], b);
            }
        }
        s_red[par][warp][lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        __syncthreads();
        if (warp == (item / (int)gridDim.x) % kWarps) {  // the items' ends dealt over the warps; the others go on
            const int g = item / fblocks, f = (item - g * fblocks) * 8 + lr;
            const unsigned m = sc.mask[g];
            float4 s = s_red[par][0][lane];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) add4(s, s_red[par][w][lane]);
            const int t = (lane & 3) * 2;  // s.x, s.y: gate of feature f, tokens t and t + 1; s.z, s.w: up
            const float h0 = __fdividef(s.x, 1.0f + __expf(-s.x)) * s.z, h1 = __fdividef(s.y, 1.0f + __expf(-s.y)) * s.w;
            const int row = sc.off[g] + __popc(m & ((1u << t) - 1u));
            const bool in0 = (m >> t) & 1u, in1 = (m >> (t + 1)) & 1u;
            if (in0) p.H[(size_t)row * I + f] = __float2bfloat16_rn(h0);
            if (in1) p.H[(size_t)(row + (in0 ? 1 : 0)) * I + f] = __float2bfloat16_rn(h1);
        }
    }
    grid_dep_launch();
}

// Work item = 16 output columns, K = all features of all groups; `split` CTAs (a cluster) share an item's K.
__global__ void __launch_bounds__(32 * kMaxDownWarps, 1) decode_small_down_kernel(DecodeSmallParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ float4 s_red[kMaxDownWarps][32];
    const int B = p.B, d = p.d, I = p.I, split = p.split;
    // [max_groups][8 / 2]: compact rows of two tokens (-1: not served) in .x and .y, their weights in .z and .w
    int4* s_rw = reinterpret_cast<int4*>(smem);
    int* s_exp = reinterpret_cast<int*>(s_rw + p.max_groups * (kTB / 2));  // [max_groups]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_thr = (int)blockDim.x, n_warps = n_thr >> 5;
    const int part = (int)blockIdx.x % split, c0 = (int)blockIdx.x / split * 16;
    for (int i = tid; i < p.max_groups * (kTB / 2); i += n_thr) s_rw[i] = make_int4(-1, -1, 0, 0);
    __syncthreads();
    grid_dep_wait();
    const int G = p.n_groups[0], rows = p.n_groups[1];
    for (int r = tid; r < p.max_rows; r += n_thr) {  // lists up to their bound in one round trip, then cut
        const int t = p.row_tok[r], g = p.row_grp[r];
        const float w = p.row_w[r];
        if (r < rows) {
            int* at = reinterpret_cast<int*>(s_rw + g * (kTB / 2) + (t >> 1)) + (t & 1);
            at[0] = r;
            at[2] = __float_as_int(w);
        }
    }
    for (int g = tid; g < p.max_groups; g += n_thr) {
        const int e = p.grp_expert[g];
        if (g < G) s_exp[g] = e;
    }
    __syncthreads();
    const int per = I / kKC, nch = G * per;  // chunks of all groups
    const int lr = lane >> 2, lk = (lane & 3) * 16;
    const int first = part * n_warps + warp, step = split * n_warps;
    uint32_t a[kUnroll][2][8], hb[kUnroll][8], an[kUnroll][2][8], hn[kUnroll][8];
    auto load = [&](int j0) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int j = j0 + u * step;
            if (j >= nch) continue;
            const int g = j / per, kc = (j - g * per) * kKC + lk;
            const __nv_bfloat16* w = p.wd + ((size_t)s_exp[g] * d + c0 + lr) * I + kc;
            ld_stream(an[u][0], w);
            ld_stream(an[u][1], w + (size_t)8 * I);
            const int row = reinterpret_cast<const int*>(s_rw + g * (kTB / 2) + (lr >> 1))[lr & 1];
            if (row >= 0) ld_rows(hn[u], p.H + (size_t)row * I + kc);
            else zero8(hn[u]);
        }
    };
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    load(first);
    for (int j0 = first; j0 < nch; j0 += kUnroll * step) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                a[u][0][i] = an[u][0][i];
                a[u][1][i] = an[u][1][i];
                hb[u][i] = hn[u][i];
            }
        load(j0 + kUnroll * step);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int j = j0 + u * step;
            if (j >= nch) break;  // warp-uniform
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            mma_chunk(c, a[u][0], a[u][1], hb[u]);
            const int4 rw = s_rw[j / per * (kTB / 2) + (lane & 3)];
            if (rw.x >= 0) {  // not for a token that the group does not serve: its zeros make NaN of infinite weights
                acc[0] = fmaf(__int_as_float(rw.z), c[0], acc[0]);
                acc[2] = fmaf(__int_as_float(rw.z), c[2], acc[2]);
            }
            if (rw.y >= 0) {
                acc[1] = fmaf(__int_as_float(rw.w), c[1], acc[1]);
                acc[3] = fmaf(__int_as_float(rw.w), c[3], acc[3]);
            }
        }
    }
    s_red[warp][lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    grid_dep_launch();
    __syncthreads();
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp == 0) {
        sum = s_red[0][lane];
        for (int w = 1; w < n_warps; ++w) add4(sum, s_red[w][lane]);
    }
    if (split > 1) {  // the cluster's parts in order
        cg::cluster_group cluster = cg::this_cluster();
        if (warp == 0) s_red[0][lane] = sum;
        cluster.sync();
        if (warp == 0 && part == 0)
            for (int q = 1; q < split; ++q) add4(sum, cluster.map_shared_rank(&s_red[0][0], q)[lane]);
        cluster.sync();  // no CTA leaves while its part may still be read
    }
    if (warp == 0 && part == 0) {
        const int t = (lane & 3) * 2, c = c0 + lr;  // sum.x, .y: column c, tokens t and t + 1; .z, .w: column c + 8
        if (t < B) {
            p.y[(size_t)t * d + c] = __float2bfloat16_rn(sum.x);
            p.y[(size_t)t * d + c + 8] = __float2bfloat16_rn(sum.z);
        }
        if (t + 1 < B) {
            p.y[(size_t)(t + 1) * d + c] = __float2bfloat16_rn(sum.y);
            p.y[(size_t)(t + 1) * d + c + 8] = __float2bfloat16_rn(sum.w);
        }
    }
}

size_t gateup_bytes(int B, int K, int d) {
    return kStateBytes + align16((size_t)B * K * 16) + (size_t)B * (d + kXPad) * 2;
}

}  // namespace

// The tokens lie in shared memory twice per SM (two CTAs); 32-byte weight loads
bool decode_small_fits(int B, int K, int d, const void* wg, const void* wu, const void* wd) {
    auto a32 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 31) == 0; };
    return B <= kSmallDecodeBatch && gateup_bytes(B, K, d) <= 100 * 1024 && a32(wg) && a32(wu) && a32(wd);
}

cudaError_t launch_decode_small(DecodeSmallParams p, const PrefillRouteParams* route, int sms, cudaStream_t s) {
    const size_t smem = gateup_bytes(p.B, p.K, p.d);
    auto gateup = [&](auto kernel, const auto& r) {
        const cudaError_t e = ensure_smem(kernel, smem);
        return e != cudaSuccess ? e : launch_pdl(kernel, std::min(2 * sms, p.max_groups * (p.I / 8)), kThreads, smem, s, p, r);
    };
    cudaError_t err = route != nullptr ? gateup(decode_small_gateup_kernel<true, PrefillRouteParams>, *route)
                      : p.w_in != nullptr ? gateup(decode_small_gateup_kernel<true, NoRoute>, NoRoute{})
                                          : gateup(decode_small_gateup_kernel<false, NoRoute>, NoRoute{});
    if (err != cudaSuccess) return err;
    // Down kernel, 16 warps per SM: one CTA of 16 warps when there are no more items than SMs (a cluster per item when
    // there are at most half as many), else two CTAs of 8 warps
    const int items = p.d / 16;
    const int warps = items <= sms ? kMaxDownWarps : kMaxDownWarps / 2;
    p.split = 1;
    while (p.split < 8 && items * p.split * 2 <= sms) p.split *= 2;
    const size_t smem2 = (size_t)p.max_groups * (kTB * 8 + 4);
    err = ensure_smem(decode_small_down_kernel, smem2);
    if (err != cudaSuccess) return err;
    if (p.split > 1) return launch_pdl_cluster(decode_small_down_kernel, items * p.split, 32 * warps, smem2, p.split, s, p);
    return launch_pdl(decode_small_down_kernel, items, 32 * warps, smem2, s, p);
}

}  // namespace exfold
