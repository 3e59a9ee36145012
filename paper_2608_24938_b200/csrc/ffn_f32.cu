// Expert FFN of fp32 layers (Eq. 1) on the CUDA cores: tensor cores would round fp32 inputs.
//
// A cluster of 8 CTAs per row tile (up to tile_rows sorted rows of one expert). Phase 0: CTA r computes its eighth of the
// intermediate features, gate and up, for all rows of the tile, and keeps silu(gate) * up in shared memory. Phase 1,
// after a cluster barrier: CTA r computes its eighth of the output features with all of I as K. The activation crosses the
// cluster through distributed shared memory: small tiles (up to kPushBytes) are written to every CTA's copy as they are
// computed, so that phase 1 waits for nothing but weights; of larger ones a CTA keeps its slice and the others read it
// chunk by chunk. The activation never goes to memory, one launch does the whole FFN, and a tile's weights are read once
// per tile instead of once per row.
//
// What bounds it: with few rows (the tiny layer: 8 rows per expert, 128 x 256) latency, hence eight CTAs per tile, one
// launch, the K split below, and ONE copy of the main loop for both phases (a kernel that runs for a few microseconds
// also waits for its own instructions); with many rows the multiply-adds. A warp covers 4 TM rows x 8 NW weight rows, its
// lanes 4 rows x 8 weight rows, so that a 16-byte shared-memory read of a warp touches at most 128 distinct bytes (one
// wavefront) and TM + NW of them feed 4 TM NW multiply-adds. Tiles of 32 rows: TM = NW = 4, two warps along the rows; of
// 16 rows: TM = 4, NW = 2; of 8 rows: TM = NW = 2. The remaining warps lie along the features; where a CTA has too few
// features for them they split K (partial sums meet in shared memory, in order). Sums: the products of one 32-wide chunk
// in a row, chunks added in order - the error of a two-level sum, as with a warp per output before.
// Measured against one CTA per route with a warp per output feature: tiny layer, 64 rows 24 -> 12 us; 400 rows of
// 768 x 1024 750 -> 158 us (12 TFLOP/s); 2048 rows of 256 x 512 270 -> 130 us.
#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"

#include <cooperative_groups.h>

namespace exfold {

namespace {

namespace cg = cooperative_groups;

constexpr int kCl = 8;         // CTAs per row tile
constexpr int kThreads = 256;  // 8 warps
constexpr int kKC = 32;        // K elements per stage
constexpr int kLd = kKC + 4;   // row pitch in floats: 16-byte aligned, the rows of a warp's read hit distinct banks
// Short tiles wait for weights (a chunk's copies take 700-1500 cycles, its multiply-adds ~100): six stages; longer ones
// compute: three, and two CTAs per SM.
__host__ __device__ constexpr int stages_of(int form_rows) { return form_rows == 8 ? 6 : 3; }

__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Four consecutive floats into shared memory, `left` of which exist (<= 0: none): the others are zero, nothing is read for
// them. VEC: 16-byte aligned, all or none. `base` is any readable, aligned address.
template <bool VEC>
__device__ __forceinline__ void stage4(uint32_t dst, const float* src, int left, const float* base) {
    if (VEC) {
        cp_async16(dst, left > 0 ? src : base, left > 0);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) cp_async4(dst + 4 * j, left > j ? src + j : base, left > j);
    }
}

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

template <int TM, int NW, int RW, bool VEC>
__global__ void __launch_bounds__(kThreads) ffn_f32_kernel(FfnF32Params p) {
    constexpr int BM = 4 * TM * RW;              // rows of the tile
    constexpr int kAcross = 8 / RW;              // warps along the features and along K
    constexpr int WR = kAcross * 8 * NW;         // weight rows of a stage, at most
    constexpr int kStage = (WR + BM) * kLd;      // floats
    constexpr int S = stages_of(BM);
    constexpr int SR = WR / 32;                  // weight rows a thread copies per chunk, at most
    static_assert(TM * NW * kThreads <= S * kStage, "partial sums fit the stages");
    static_assert(BM <= 32, "one token row per staging thread");
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_g, s_row0, s_rows;
    float* hs = smem + S * kStage;  // [tile_rows][hld]: this CTA's slice of H, or (push) all of H
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tile = (int)(blockIdx.x / kCl);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lr = lane >> 3, lf = lane & 7, wr = warp / kAcross, wa = warp % kAcross;
    const int d = p.d, I = p.I, fpc = p.fpc, hld = p.hld;
    const bool push = p.push != 0;
    if (threadIdx.x == 0) s_g = -1;
    grid_dep_wait();
    __syncthreads();
    {  // which group owns this tile: every group's tile range in one round trip
        const int gd = p.n_groups_dev != nullptr ? *p.n_groups_dev : p.G;
        for (int g = threadIdx.x; g < p.G; g += kThreads) {
            const int t0 = p.tile_start[g], t1 = p.tile_start[g + 1], o0 = p.offsets[g], o1 = p.offsets[g + 1];
            if (g < gd && tile >= t0 && tile < t1) {
                s_g = g;
                s_row0 = o0 + (tile - t0) * p.tile_rows;
                s_rows = min(p.tile_rows, o1 - s_row0);
            }
        }
    }
    __syncthreads();
    if (s_g < 0) return;  // the whole cluster: past the last tile
    cluster.barrier_arrive();  // waited for before the first access to another CTA's shared memory: all CTAs have started
    bool started = false;
    const int rows = s_rows;
    const int64_t row0 = s_row0;
    const size_t e = p.grp_expert != nullptr ? p.grp_expert[s_g] : s_g;

    // What this thread copies in every chunk, fixed for a pass: SR weight rows of the stage and one token row, from
    // w_src / x_src on, w_len / x_len floats ahead of it in the first chunk (none for rows that are not there)
    const int vk = (threadIdx.x & 7) * 4, vr = threadIdx.x >> 3;  // 32 rows of 8 vectors per sweep
    const bool x_in = vr < BM && vr < rows;
    const uint32_t w_dst = ptx::smem_u32(smem) + (uint32_t)(vr * kLd + vk) * 4u;
    const float* w_src[SR];
    int w_len[SR];
    const float* x_src = p.x;
    if (x_in) {
        const int64_t tok = p.row_tok != nullptr ? (int64_t)p.row_tok[row0 + vr] : (row0 + vr) % p.x_rows;
        x_src = p.x + tok * d + vk;
    }
    const int x_len = x_in ? d - vk : 0;

#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
        if (phase == 1) {
            if (push)  // the last chunk's columns past I
                for (int i = threadIdx.x; i < p.tile_rows * (hld - I); i += kThreads)
                    hs[i / (hld - I) * hld + I + i % (hld - I)] = 0.f;
            if (!started) cluster.barrier_wait();
            grid_dep_launch();  // not earlier: the next kernel's CTAs would only take this grid's places
            cluster.sync();     // every slice of H is in place
        }
        // phase 0: H[:, rank's features] = silu(x W_gate^T) * (x W_up^T); phase 1: out[:, rank's columns] = H W_down^T
        const int K = phase == 0 ? d : I, per = phase == 0 ? fpc : (d + kCl - 1) / kCl;
        const int lo = rank * per, hi = min(phase == 0 ? I : d, lo + per);
        // A power of two of warps (n_wf) lies along the stage's weight rows, the others split K; afterwards the warps with
        // wk == 0 hold the sums of token rows wr * 4 TM + 4 r + lr and stage rows wf * 8 NW + 8 q + lf.
        int n_wf = 1;
        while (n_wf < kAcross && n_wf * 8 * NW < (phase == 0 ? 2 : 1) * (hi - lo)) n_wf *= 2;
        const int wf = wa & (n_wf - 1), wk = wa / n_wf, nk = kAcross / n_wf, n_rows = n_wf * 8 * NW;
        const int step = phase == 0 ? n_rows / 2 : n_rows;  // features (a gate and an up row each) or columns per pass
        const bool x_local = phase == 1 && push;
        const int nc = (K + kKC - 1) / kKC;
#pragma unroll 1
        for (int f0 = lo; f0 < hi; f0 += step) {
#pragma unroll
            for (int q = 0; q < SR; ++q) {  // a warp's stage rows in phase 0: 4 NW gate rows, then the same features' up rows
                const int r = vr + 32 * q, in_warp = r % (8 * NW);
                const int f = phase == 0 ? f0 + r / (8 * NW) * (4 * NW) + in_warp % (4 * NW) : f0 + r;
                const float* base = phase == 1 ? p.wd : (in_warp < 4 * NW ? p.wg : p.wu);
                w_src[q] = base + (e * (size_t)(phase == 0 ? I : d) + f) * K + vk;
                w_len[q] = r < n_rows && f < hi ? K - vk : 0;
            }
            float acc[TM][NW];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int q = 0; q < NW; ++q) acc[r][q] = 0.f;
            __syncthreads();  // the previous pass is done with the stages
            int st_in = 0, st_out = 0;
#pragma unroll 1
            for (int c = 1 - S; c < nc; ++c) {  // chunk c + S - 1 is requested, chunk c (once >= 0) is consumed
                if (c >= 0) {
                    cp_wait<S - 2>();
                    __syncthreads();
                }
                const int cn = c + S - 1;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                const uint32_t off = (uint32_t)(st_in * kStage) * 4u;
                if (cn < nc) {
#pragma unroll
                    for (int q = 0; q < SR; ++q)
                        if (vr + 32 * q < n_rows)
                            stage4<VEC>(w_dst + off + (uint32_t)(32 * q * kLd) * 4u, w_src[q] + cn * kKC, w_len[q] - cn * kKC, p.x);
                    if (phase == 0) {
                        if (vr < BM) stage4<VEC>(w_dst + off + (uint32_t)(WR * kLd) * 4u, x_src + cn * kKC, x_len - cn * kKC, p.x);
                    } else if (!push && x_in) {
                        // a chunk lies in one CTA's slice (fpc is a multiple of 32); features past I (never written) are zero
                        const int owner = (cn * kKC) / fpc, k = cn * kKC + vk;
                        v = *reinterpret_cast<const float4*>(cluster.map_shared_rank(hs, owner) + vr * hld + (k - owner * fpc));
                        if (k + 4 > I) {
                            if (k >= I) v.x = 0.f;
                            if (k + 1 >= I) v.y = 0.f;
                            if (k + 2 >= I) v.z = 0.f;
                            if (k + 3 >= I) v.w = 0.f;
                        }
                    }
                }
                cp_commit();
                if (c >= 0) {
                    const float* ws = smem + st_out * kStage;
                    const float* xs = x_local ? hs + c * kKC : ws + WR * kLd;
                    const int x_pitch = x_local ? hld : kLd;
                    mac_chunk<TM, NW>(ws + (wf * 8 * NW + lf) * kLd, xs + (wr * 4 * TM + lr) * x_pitch, x_pitch, wk, nk, acc);
                    if (++st_out == S) st_out = 0;
                }
                if (cn < nc && phase == 1 && !push && vr < BM)
                    *reinterpret_cast<float4*>(smem + st_in * kStage + (WR + vr) * kLd + vk) = v;
                if (++st_in == S) st_in = 0;
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
            if (phase == 0) {
                if (!started) {
                    cluster.barrier_wait();
                    started = true;
                }
                if (wk == 0)
#pragma unroll
                    for (int r = 0; r < TM; ++r)
#pragma unroll
                        for (int q = 0; q < NW / 2; ++q) {
                            const int f = f0 + wf * 4 * NW + q * 8 + lf, row = (wr * TM + r) * 4 + lr;
                            const float g = acc[r][q], u = acc[r][q + NW / 2];
                            const float h = (g / (1.0f + expf(-g))) * u;
                            if (row >= p.tile_rows) continue;
                            if (!push) {
                                if (f < lo + fpc) hs[row * hld + f - lo] = h;
                            } else if (f < hi) {
#pragma unroll
                                for (int c = 0; c < kCl; ++c) cluster.map_shared_rank(hs, c)[row * hld + f] = h;
                            }
                        }
            } else if (wk == 0) {
#pragma unroll
                for (int r = 0; r < TM; ++r) {
                    const int row = (wr * TM + r) * 4 + lr;
                    if (row >= rows) continue;
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
    if (!push) cluster.sync();  // no CTA leaves while another may still read its slice of H
}

constexpr size_t kSmemLimit = 227 * 1024 - 1024;
constexpr size_t kPushBytes = 32 * 1024;
int features_per_cta(int I) { return ((I + kCl - 1) / kCl + kKC - 1) / kKC * kKC; }
bool push_h(int tile_rows, int I) { return (size_t)std::max(8, tile_rows) * I * sizeof(float) <= kPushBytes; }
int h_pitch(int tile_rows, int I) {  // whole chunks + 4: 16-byte aligned, the four rows of a warp's read in distinct banks
    return (push_h(tile_rows, I) ? (I + kKC - 1) / kKC * kKC : features_per_cta(I)) + 4;
}
size_t smem_bytes(int tile_rows, int I) {  // 128 weight rows and the form's token rows per stage, then H
    const int form_rows = std::max(8, tile_rows);  // all of which are read from a push tile (and not used past tile_rows)
    const int h_rows = push_h(tile_rows, I) ? form_rows : tile_rows;
    return ((size_t)stages_of(form_rows) * (128 + form_rows) * kLd + (size_t)h_rows * h_pitch(tile_rows, I)) * sizeof(float);
}

template <int TM, int NW, int RW, bool VEC>
cudaError_t launch_t(const FfnF32Params& p, int64_t tiles, cudaStream_t s) {
    const size_t smem = smem_bytes(p.tile_rows, p.I);
    cudaError_t err = cudaFuncSetAttribute(ffn_f32_kernel<TM, NW, RW, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)smem);
    if (err != cudaSuccess) return err;
    return launch_pdl_cluster(ffn_f32_kernel<TM, NW, RW, VEC>, (unsigned)(tiles * kCl), kThreads, smem, kCl, s, p);
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

// Rows per tile: a tile computes all of its rows, so short groups want short tiles (and more of them to fill the SMs); a
// tile's weights are read once per tile, so long groups want long ones. Measured, 16 / 32-row tiles: 17 experts of
// 768 x 1024 with 25 rows each 154 / 220 us; 20 of 512 x 384 with ~40 rows 109 / 123 us. Halved while the tile's slice of H
// does not fit the shared memory (8 rows: I above ~40 000 features).
int ffn_f32_tile_rows(int64_t rows, int G, int I) {
    int tile_rows = rows > (int64_t)48 * G ? 32 : rows > (int64_t)8 * G ? 16 : 8;
    while (tile_rows > 1 && smem_bytes(tile_rows, I) > kSmemLimit) tile_rows /= 2;
    return tile_rows;
}

cudaError_t launch_ffn_f32(FfnF32Params p, int64_t rows, cudaStream_t s) {
    if (rows == 0) return cudaSuccess;
    p.fpc = features_per_cta(p.I);
    p.push = push_h(p.tile_rows, p.I) ? 1 : 0;
    p.hld = h_pitch(p.tile_rows, p.I);
    const int64_t tiles = std::min<int64_t>(rows, rows / p.tile_rows + p.G);
    auto a16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    const bool vec = p.d % 4 == 0 && p.I % 4 == 0 && a16(p.x) && a16(p.wg) && a16(p.wu) && a16(p.wd);
    if (p.tile_rows == 32) return vec ? launch_t<4, 4, 2, true>(p, tiles, s) : launch_t<4, 4, 2, false>(p, tiles, s);
    if (p.tile_rows == 16) return vec ? launch_t<4, 2, 1, true>(p, tiles, s) : launch_t<4, 2, 1, false>(p, tiles, s);
    return vec ? launch_t<2, 2, 1, true>(p, tiles, s) : launch_t<2, 2, 1, false>(p, tiles, s);
}

cudaError_t launch_combine_f32(const float* out, const int32_t* inv_pos, const float* row_w, int64_t T, int Kr, int d,
                               int n_shared, const int32_t* shared0_dev, float* y, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    return launch_pdl(combine_f32_kernel, (unsigned)T, 128, 0, s, out, inv_pos, row_w, T, Kr, d, n_shared, shared0_dev, y);
}

}  // namespace exfold
