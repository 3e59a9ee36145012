// Offline calibration of the pairwise scalar projector (Eq. 6-9): per ordered pair (s,t) of
// experts observed on the same calibration token, with u = E_s(x), v = E_t(x) and token
// weight w = |u|, accumulate A = sum w<v,u>, B = sum w|v|^2, C = sum w|u|^2 in double;
// then S = clip(A / (B + lambda)), L = max(0, C - 2 S A + S^2 B) / (C + eps).
#include "common.cuh"
#include "ptx.cuh"

#include <algorithm>

namespace exfold {

namespace {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Sum of NV values over the warp by halving exchanges (reduce-scatter: NV/2 + NV/4 + ... shuffles instead of 5 NV).
// On return out[idx] (shared memory) holds the sum of value idx; the caller synchronises the warp.
template <int N, int OFF>
__device__ __forceinline__ void reduce_scatter_step(double* v, int lane) {
    if constexpr (OFF > 0) {
        constexpr int HALF = (N + 1) / 2;
        const bool up = (lane & OFF) != 0;
#pragma unroll
        for (int i = 0; i < HALF; ++i) {
            const double lo = v[i], hi = i + HALF < N ? v[i + HALF] : 0.0;
            v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, OFF);
        }
        reduce_scatter_step<HALF, OFF / 2>(v, lane);
    }
}
// index of slot i of this lane after the steps above (-1: none)
template <int N, int OFF>
__device__ __forceinline__ int reduce_scatter_index(int i, int lane) {
    if constexpr (OFF > 0) {
        constexpr int HALF = (N + 1) / 2;
        const int r = reduce_scatter_index<HALF, OFF / 2>(i, lane);
        if (r < 0) return -1;
        const int idx = r + ((lane & OFF) ? HALF : 0);
        return idx < N ? idx : -1;
    } else {
        return i < N ? i : -1;
    }
}
template <int NV>
__device__ __forceinline__ void warp_sums(double (&v)[NV], double* out, int lane) {
    constexpr int LEFT = (NV + 31) / 32;
    reduce_scatter_step<NV, 16>(v, lane);
#pragma unroll
    for (int i = 0; i < LEFT; ++i) {
        const int idx = reduce_scatter_index<NV, 16>(i, lane);
        if (idx >= 0) out[idx] = v[i];
    }
}

constexpr int kStatsThreads = 128;
constexpr int kStatsRows = 8;  // largest Top-K whose Gram triangle (36 sums) is held in one warp's registers

__device__ __forceinline__ int64_t stats_row(const CalibStatsParams& p, int64_t i, int a) {
    return p.inv_pos ? (int64_t)p.inv_pos[i * p.Ke + a] : i * p.tok_stride + a * p.slot_stride;
}
__device__ __forceinline__ void add_pair(const CalibStatsParams& p, int s, int t, double wi, double uu, double vu,
                                         double vv) {
    const size_t pq = (size_t)s * p.N + t;
    atomicAdd(&p.A[pq], wi * vu);
    atomicAdd(&p.Bv[pq], wi * vv);
    atomicAdd(&p.C[pq], wi * uu);
    atomicAdd(&p.cnt[pq], 1);
}

// Pair sums of a token per warp, KE = Top-K <= 8: the token's KE output rows are read once, converted to double once, and all
// KE (KE + 1) / 2 inner products accumulate in registers. Bound by reading the rows (4 KE d bytes per token). The rows come by
// bulk copies into a ring of three stages of 256 columns per warp (lane a fetches row a; the next token's rows follow without a
// gap): with 192 KB per SM twice the bytes are in flight that registers could hold beside the sums, and the
// double-precision units work meanwhile. 8192 tokens x 8 rows x 2048 columns: a warp per ordered pair 619 us, rows through
// registers with one chunk ahead 137 (134 alone under a profiler), this 101 alone (98 without the atomics).
constexpr int kRingWarps = 8;  // of a CTA, at most
constexpr int kRingStages = 3;
constexpr int kRingCols = 256;
// CTAs per SM, as many as their rings leave room for. Whole calibration with one / these: 64 experts of 1024 x 512, 2048 tokens, Top-3
// 95.1 / 93.3 us, 8 of 4096 x 1024, 2048 tokens, Top-4 249 / 245.
template <int KE>
constexpr int kRingCtas = KE == 2 ? 4 : KE == 3 ? 3 : KE == 4 ? 2 : 1;

// The rows are read once: they are the first to leave L2, before the weights (a layer of 50 MB calibrated again and again, Top-1, 2048
// tokens: 83.4 -> 75.3 us)
__device__ __forceinline__ uint64_t evict_first_policy() {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
                     ptx::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(ptx::smem_u32(bar)), "l"(policy)
                 : "memory");
}

template <int KE>
__global__ void __launch_bounds__(32 * kRingWarps, kRingCtas<KE>) calib_stats_kernel(CalibStatsParams p) {
    constexpr int NV = KE * (KE + 1) / 2;
    extern __shared__ __align__(128) float ring_all[];
    __shared__ double s_gram[kRingWarps][NV];
    __shared__ __align__(8) uint64_t bars[kRingWarps][kRingStages];
    __shared__ int abort_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* ring = ring_all + (size_t)warp * kRingStages * KE * kRingCols;
    if (lane == 0) {
        for (int s = 0; s < kRingStages; ++s) ptx::mbar_init(&bars[warp][s], 1);
        ptx::fence_mbar_init();
    }
    if (threadIdx.x == 0) abort_s = 0;
    __syncthreads();
    grid_dep_launch();
    grid_dep_wait();
    const int d = p.d, n_chunks = (d + kRingCols - 1) / kRingCols;
    const int n_warps = (int)blockDim.x >> 5;
    const uint64_t policy = evict_first_policy();
    const int64_t step = (int64_t)gridDim.x * n_warps, i0 = (int64_t)blockIdx.x * n_warps + warp;
    // the loads run ahead of the sums: chunk lc of token li into stage ls
    int64_t li = i0;
    int lc = 0, ls = 0;
    const float* row = li < p.m && lane < KE ? p.out + stats_row(p, li, lane) * d : nullptr;
    auto load = [&]() {
        if (li >= p.m) return;
        const int c0 = lc * kRingCols, cols = min(kRingCols, d - c0);
        if (lane == 0) ptx::mbar_expect_tx(&bars[warp][ls], (uint32_t)(KE * cols * 4));
        __syncwarp();
        if (lane < KE) bulk_load(ring + (ls * KE + lane) * kRingCols, row + c0, (uint32_t)cols * 4, &bars[warp][ls], policy);
        if (++ls == kRingStages) ls = 0;
        if (++lc == n_chunks) {
            lc = 0;
            li += step;
            if (li < p.m && lane < KE) row = p.out + stats_row(p, li, lane) * d;
        }
    };
#pragma unroll
    for (int s = 0; s < kRingStages; ++s) load();
    int cs = 0, cphase = 0;
    for (int64_t i = i0; i < p.m; i += step) {
        double acc[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = 0.0;
        for (int k = 0; k < n_chunks; ++k) {
            const bool ok = ptx::mbar_wait(&bars[warp][cs], cphase, &abort_s, p.status, 9);
            if (!__all_sync(0xffffffffu, ok)) {
                __nanosleep(100000);  // let any copy still in flight land before shared memory is released
                return;
            }
            const float* st = ring + cs * KE * kRingCols;
            const int cols = min(kRingCols, d - k * kRingCols);
            for (int c = lane * 4; c < cols; c += 128) {
                float4 cur[KE];
#pragma unroll
                for (int a = 0; a < KE; ++a) cur[a] = *reinterpret_cast<const float4*>(st + a * kRingCols + c);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    double o[KE];
#pragma unroll
                    for (int a = 0; a < KE; ++a)
                        o[a] = (double)(q == 0 ? cur[a].x : q == 1 ? cur[a].y : q == 2 ? cur[a].z : cur[a].w);
                    int v = 0;
#pragma unroll
                    for (int a = 0; a < KE; ++a)
#pragma unroll
                        for (int b = a; b < KE; ++b, ++v) acc[v] = fma(o[a], o[b], acc[v]);
                }
            }
            __syncwarp();  // the stage is used up
            load();
            if (++cs == kRingStages) {
                cs = 0;
                cphase ^= 1;
            }
        }
        double* g = s_gram[warp];
        warp_sums<NV>(acc, g, lane);
        __syncwarp();
        auto at = [](int a, int b) {  // place of (a, b) in the upper triangle
            const int lo = a < b ? a : b, hi = a < b ? b : a;
            return lo * KE - lo * (lo - 1) / 2 + (hi - lo);
        };
        const int32_t* ids = p.ids + i * KE;
        for (int q = lane; q < KE * KE; q += 32) {
            const int a = q / KE, b = q - a * KE;
            const double uu = g[at(a, a)], wi = sqrt(uu);
            if (a == b) {
                atomicAdd(&p.H[ids[a]], wi);
                atomicAdd(&p.hc[ids[a]], 1);
            } else {
                add_pair(p, ids[a], ids[b], wi, uu, g[at(a, b)], g[at(b, b)]);
            }
        }
        __syncwarp();
    }
}

// The same for one row per token, or two of at most 2048 columns: a warp per token, 16 bytes per lane and row with the next chunk in
// flight, into registers. The ring's barriers and its walk over the tokens cost a token more than so few copies bring. Whole
// calibration with the ring / this: 32 experts of 2048 x 128, Top-1, 2048 and 8192 tokens 75.3 / 67.9, 115.0 / 102.4 us, Top-2, 8192
// 154 / 140; 64 of 1024 x 512, Top-2, 2048 tokens 92.7 / 88.4; the other way 8 of 4096 x 1024, Top-2, 64, 512 and 2048 tokens 91.6 /
// 97.6, 102.6 / 107.0, 150.4 / 158.0.
template <int KE>
__global__ void __launch_bounds__(kStatsThreads) calib_stats_short_kernel(CalibStatsParams p) {
    constexpr int NV = KE * (KE + 1) / 2;
    __shared__ double s_gram[kStatsThreads / 32][NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_dep_launch();
    grid_dep_wait();
    const int64_t i = (int64_t)blockIdx.x * (kStatsThreads / 32) + warp;
    if (i >= p.m) return;
    const int d = p.d;
    const float* row[KE];
#pragma unroll
    for (int a = 0; a < KE; ++a) row[a] = p.out + stats_row(p, i, a) * d;
    double acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = 0.0;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 nxt[KE];
    int c = lane * 4;
#pragma unroll
    for (int a = 0; a < KE; ++a) nxt[a] = c < d ? __ldcs(reinterpret_cast<const float4*>(row[a] + c)) : zero;
    for (; c < d; c += 128) {
        float4 cur[KE];
#pragma unroll
        for (int a = 0; a < KE; ++a) {
            cur[a] = nxt[a];
            nxt[a] = c + 128 < d ? __ldcs(reinterpret_cast<const float4*>(row[a] + c + 128)) : zero;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            double o[KE];
#pragma unroll
            for (int a = 0; a < KE; ++a)
                o[a] = (double)(q == 0 ? cur[a].x : q == 1 ? cur[a].y : q == 2 ? cur[a].z : cur[a].w);
            int v = 0;
#pragma unroll
            for (int a = 0; a < KE; ++a)
#pragma unroll
                for (int b = a; b < KE; ++b, ++v) acc[v] = fma(o[a], o[b], acc[v]);
        }
    }
    double* g = s_gram[warp];
    warp_sums<NV>(acc, g, lane);
    __syncwarp();
    auto at = [](int a, int b) {  // place of (a, b) in the upper triangle
        const int lo = a < b ? a : b, hi = a < b ? b : a;
        return lo * KE - lo * (lo - 1) / 2 + (hi - lo);
    };
    const int32_t* ids = p.ids + i * KE;
    for (int q = lane; q < KE * KE; q += 32) {
        const int a = q / KE, b = q - a * KE;
        const double uu = g[at(a, a)], wi = sqrt(uu);
        if (a == b) {
            atomicAdd(&p.H[ids[a]], wi);
            atomicAdd(&p.hc[ids[a]], 1);
        } else {
            add_pair(p, ids[a], ids[b], wi, uu, g[at(a, b)], g[at(b, b)]);
        }
    }
}

// Larger Top-K: a warp takes four source rows against four target rows of a token (blocks I <= J of the slots) and their
// eight squared norms; a row is then read by ceil(Ke / 4) warps, mostly from L1 / L2.
__global__ void __launch_bounds__(kStatsThreads) calib_stats_tiled_kernel(CalibStatsParams p, int nb) {
    constexpr int NV = 24;  // 16 products, 4 + 4 norms
    __shared__ double s_sum[kStatsThreads / 32][NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_dep_launch();
    grid_dep_wait();
    const int64_t w = (int64_t)blockIdx.x * (kStatsThreads / 32) + warp;
    const int tiles = nb * (nb + 1) / 2;
    const int64_t i = w / tiles;
    if (i >= p.m) return;
    int I = 0, J = (int)(w - i * tiles);
    while (J >= nb - I) {
        J -= nb - I;
        ++I;
    }
    J += I;
    const int Ke = p.Ke, d = p.d;
    const float* u[4];
    const float* v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // slots past Ke repeat the last one; their sums are not used
        u[r] = p.out + stats_row(p, i, min(4 * I + r, Ke - 1)) * d;
        v[r] = p.out + stats_row(p, i, min(4 * J + r, Ke - 1)) * d;
    }
    double acc[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) acc[q] = 0.0;
    for (int c = lane * 4; c < d; c += 128) {
        float4 fu[4], fv[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            fu[r] = *reinterpret_cast<const float4*>(u[r] + c);
            fv[r] = *reinterpret_cast<const float4*>(v[r] + c);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            double du[4], dv[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                du[r] = (double)(q == 0 ? fu[r].x : q == 1 ? fu[r].y : q == 2 ? fu[r].z : fu[r].w);
                dv[r] = (double)(q == 0 ? fv[r].x : q == 1 ? fv[r].y : q == 2 ? fv[r].z : fv[r].w);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[4 * a + b] = fma(du[a], dv[b], acc[4 * a + b]);
                acc[16 + a] = fma(du[a], du[a], acc[16 + a]);
                acc[20 + a] = fma(dv[a], dv[a], acc[20 + a]);
            }
        }
    }
    double* g = s_sum[warp];
    warp_sums<NV>(acc, g, lane);
    __syncwarp();
    const int32_t* ids = p.ids + i * Ke;
    const int a = (lane >> 2) & 3, b = lane & 3;  // lanes 0-15: source from I, target from J; 16-31: the other direction
    const int sa = 4 * I + a, sb = 4 * J + b;
    if (sa >= Ke || sb >= Ke) return;
    const double na = g[16 + a], nb2 = g[20 + b], prod = g[4 * a + b];
    if (I == J) {
        if (lane >= 16) return;
        if (sa == sb) {
            atomicAdd(&p.H[ids[sa]], sqrt(na));
            atomicAdd(&p.hc[ids[sa]], 1);
        } else {
            add_pair(p, ids[sa], ids[sb], sqrt(na), na, prod, nb2);
        }
    } else if (lane < 16) {
        add_pair(p, ids[sa], ids[sb], sqrt(na), na, prod, nb2);
    } else {
        add_pair(p, ids[sb], ids[sa], sqrt(nb2), nb2, prod, na);
    }
}

__global__ void calib_finalize_kernel(CalibStatsParams p, exfold_calib_opts o, float* S, float* L, float* h,
                                      float* lnh, int32_t* n_obs, int32_t* unobserved) {
    const int N = p.N;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    grid_dep_launch();
    grid_dep_wait();
    if (idx < N * N) {
        const int s = idx / N, t = idx % N;
        float sv, lv;
        if (s == t) {
            sv = 1.0f;
            lv = 0.0f;
        } else if (p.cnt[idx] == 0) {
            sv = 0.0f;
            lv = 1e30f;
        } else {
            double a = p.A[idx], b = p.Bv[idx], c = p.C[idx];
            double sc = a / (b + (double)o.lambda);
            if (sc < (double)o.clip_lo) sc = (double)o.clip_lo;
            if (sc > (double)o.clip_hi) sc = (double)o.clip_hi;
            double num = c - 2.0 * sc * a + sc * sc * b;
            if (num < 0.0) num = 0.0;
            sv = (float)sc;
            lv = (float)(num / (c + (double)o.eps));
        }
        S[idx] = sv;
        L[idx] = lv;
        if (n_obs) n_obs[idx] = p.cnt[idx];
    }
    if (blockIdx.x == 0) {  // norms: a thread per expert (N <= 256 = the block; one thread alone: 128 experts 58 us, now 5)
        __shared__ double s_h[kMaxExperts];
        __shared__ double s_mean;
        const int e = threadIdx.x;
        const int n_e = e < N ? p.hc[e] : 0;
        const double he = n_e > 0 ? p.H[e] / (double)n_e : 0.0;
        if (e < N) s_h[e] = he;
        const int un = N - __syncthreads_count(n_e > 0);
        if (e == 0) {
            double hsum = 0.0;
            for (int o = 0; o < N; ++o) hsum += s_h[o];
            s_mean = un < N ? hsum / (N - un) : 1.0;
            *unobserved = un;
        }
        __syncthreads();
        if (e < N) {
            const float hf = (float)(n_e > 0 ? he : s_mean);
            h[e] = hf;
            lnh[e] = (float)log((double)hf);
        }
    }
}

// ids[i][e] = e: every expert sees every token (common-input calibration)
__global__ void iota_ids_kernel(int32_t* ids, int64_t m, int N) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m * N) ids[i] = (int32_t)(i % N);
}

// ---- common-input mode (slot a = expert a for every token), many experts: the pair sums as Gram products.
// A[s][t] = sum_i w_is <o_is, o_it>,  B[s][t] = sum_i w_is |o_it|^2,  C[s][t] = sum_i w_is^3,  w_is = |o_is|.
// Only A needs the off-diagonal inner products; B and C follow from the per-token squared norms.

// nrm[i][a] = |o_ia|^2 in double; one warp per (token, expert)
__global__ void __launch_bounds__(256) calib_norms_kernel(CalibStatsParams p, double* __restrict__ nrm) {
    const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (w >= p.m * p.Ke) return;
    const int64_t i = w / p.Ke;
    const int a = (int)(w % p.Ke);
    const float* u = p.out + (i * p.tok_stride + a * p.slot_stride) * p.d;
    double uu = 0.0;
    for (int c = lane; c < p.d; c += 32) {
        const double uc = (double)u[c];
        uu += uc * uc;
    }
    uu = warp_sum_d(uu);
    if (lane == 0) nrm[w] = uu;
}

// Each CTA walks its share of the tokens and keeps a 128 x 128 block of A in registers (4 x 4 per thread,
// 32 x 32 threads); 16-column chunks of the token's outputs are staged in shared memory, the source side
// already scaled by its weight w_is (in double, so nothing is rounded before the double accumulation).
__global__ void __launch_bounds__(1024, 1) calib_gram_kernel(CalibStatsParams p, const double* __restrict__ nrm) {
    __shared__ double sa[128][17];
    __shared__ float sb[128][17];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int lx = threadIdx.x & 15, ly = threadIdx.x >> 4;  // loader coordinates: 16 columns x 64 rows
    const int Ke = p.Ke, d = p.d, N = p.N;
    for (int ab = 0; ab < Ke; ab += 128)
        for (int bb = 0; bb < Ke; bb += 128) {
            double acc[4][4];
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) acc[ii][jj] = 0.0;
            for (int64_t i = blockIdx.x; i < p.m; i += gridDim.x) {
                for (int c0 = 0; c0 < d; c0 += 16) {
                    __syncthreads();
                    const bool cin = c0 + lx < d;
                    for (int r = ly; r < 128; r += 64) {
                        const int a = ab + r, b = bb + r;
                        double av = 0.0;
                        float bv = 0.f;
                        if (cin && a < Ke)
                            av = sqrt(nrm[i * Ke + a]) *
                                 (double)p.out[(i * p.tok_stride + a * p.slot_stride) * d + c0 + lx];
                        if (cin && b < Ke) bv = p.out[(i * p.tok_stride + b * p.slot_stride) * d + c0 + lx];
                        sa[r][lx] = av;
                        sb[r][lx] = bv;
                    }
                    __syncthreads();
#pragma unroll 4
                    for (int c = 0; c < 16; ++c) {
                        double a4[4], b4[4];
#pragma unroll
                        for (int ii = 0; ii < 4; ++ii) a4[ii] = sa[ty + 32 * ii][c];
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj) b4[jj] = (double)sb[tx + 32 * jj][c];
#pragma unroll
                        for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                            for (int jj = 0; jj < 4; ++jj) acc[ii][jj] += a4[ii] * b4[jj];
                    }
                }
            }
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int a = ab + ty + 32 * ii, b = bb + tx + 32 * jj;
                    if (a < Ke && b < Ke && a != b) atomicAdd(&p.A[(size_t)a * N + b], acc[ii][jj]);
                }
        }
}

// B, C, the pair counts and the per-expert norm sums from the squared norms; one thread per ordered pair
__global__ void __launch_bounds__(256) calib_common_finish_kernel(CalibStatsParams p, const double* __restrict__ nrm) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int Ke = p.Ke, N = p.N;
    if (idx >= Ke * Ke) return;
    const int s = idx / Ke, t = idx % Ke;
    double bsum = 0.0, csum = 0.0, hsum = 0.0;
    for (int64_t i = 0; i < p.m; ++i) {
        const double ns = nrm[i * Ke + s], nt = nrm[i * Ke + t];
        const double w = sqrt(ns);
        bsum += w * nt;
        csum += w * ns;
        hsum += w;
    }
    if (s == t) {
        p.H[s] = hsum;
        p.hc[s] = (int32_t)p.m;
    } else {
        const size_t pq = (size_t)s * N + t;
        p.Bv[pq] = bsum;
        p.C[pq] = csum;
        p.cnt[pq] = (int32_t)p.m;
    }
}

// common-input mode: group e = all m tokens in order
__global__ void calib_common_rows_kernel(int32_t* offsets, int32_t* work_start, int64_t m, int N, int tile_rows) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g <= N) {
        offsets[g] = (int32_t)(g * m);
        work_start[g] = (int32_t)(g * row_tiles((int)m, tile_rows));
    }
}

}  // namespace

cudaError_t launch_calib_common_rows(int32_t* offsets, int32_t* work_start, int64_t m, int N, int tile_rows, cudaStream_t s) {
    calib_common_rows_kernel<<<(N + 1 + 255) / 256, 256, 0, s>>>(offsets, work_start, m, N, tile_rows);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_calib_stats_common(const CalibStatsParams& p, double* nrm, int sms, cudaStream_t s) {
    if (p.m == 0) return cudaSuccess;
    const int64_t warps = p.m * p.Ke;
    calib_norms_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(p, nrm);
    count_launch();
    calib_gram_kernel<<<(unsigned)std::min<int64_t>(p.m, sms), 1024, 0, s>>>(p, nrm);
    count_launch();
    calib_common_finish_kernel<<<(p.Ke * p.Ke + 255) / 256, 256, 0, s>>>(p, nrm);
    count_launch();
    return cudaGetLastError();
}

template <int KE>
static cudaError_t launch_stats(const CalibStatsParams& p, int sms, cudaStream_t s) {
    // few tokens: fewer warps to a CTA, so that every SM has some
    const int warps = (int)std::min<int64_t>((p.m + sms - 1) / sms, kRingWarps);
    const size_t smem = (size_t)warps * kRingStages * KE * kRingCols * sizeof(float);
    cudaError_t err = ensure_smem(calib_stats_kernel<KE>, smem);
    if (err != cudaSuccess) return err;
    const int64_t blocks = std::min<int64_t>((p.m + warps - 1) / warps, (int64_t)sms * kRingCtas<KE>);
    return launch_pdl(calib_stats_kernel<KE>, (unsigned)blocks, 32 * warps, smem, s, p);
}
cudaError_t launch_calib_stats(const CalibStatsParams& p, int sms, cudaStream_t s) {
    if (p.m == 0) return cudaSuccess;
    constexpr int kWarps = kStatsThreads / 32;
    const unsigned short_grid = (unsigned)((p.m + kWarps - 1) / kWarps);
    if (p.Ke > kStatsRows) {
        const int nb = (p.Ke + 3) / 4;
        const int64_t warps = p.m * (nb * (nb + 1) / 2);
        return launch_pdl(calib_stats_tiled_kernel, (unsigned)((warps + kWarps - 1) / kWarps), kStatsThreads, 0, s, p, nb);
    }
    switch (p.Ke) {
        case 1: return launch_pdl(calib_stats_short_kernel<1>, short_grid, kStatsThreads, 0, s, p);
        case 2:
            if (p.d <= 2048) return launch_pdl(calib_stats_short_kernel<2>, short_grid, kStatsThreads, 0, s, p);
            return launch_stats<2>(p, sms, s);
        case 3: return launch_stats<3>(p, sms, s);
        case 4: return launch_stats<4>(p, sms, s);
        case 5: return launch_stats<5>(p, sms, s);
        case 6: return launch_stats<6>(p, sms, s);
        case 7: return launch_stats<7>(p, sms, s);
        default: return launch_stats<8>(p, sms, s);
    }
}

cudaError_t launch_calib_finalize(const CalibStatsParams& p, const exfold_calib_opts& o, float* S, float* L,
                                  float* h, float* lnh, int32_t* n_obs, int32_t* unobserved, cudaStream_t s) {
    const int n = p.N * p.N;
    return launch_pdl(calib_finalize_kernel, (n + 255) / 256, 256, 0, s, p, o, S, L, h, lnh, n_obs, unobserved);
}

cudaError_t launch_iota_ids(int32_t* ids, int64_t m, int N, cudaStream_t s) {
    const int64_t n = m * N;
    if (n == 0) return cudaSuccess;
    iota_ids_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(ids, m, N);
    count_launch();
    return cudaGetLastError();
}

}  // namespace exfold
