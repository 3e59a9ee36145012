// CUDA-core kernels around the expert GEMMs of bf16 layers: the per-token sum of the experts' rows (Eq. 3 / Eq. 4) and
// the router scores of fp32 layers and small bf16 batches.
#include <algorithm>

#include "common.cuh"

namespace exfold {

namespace {

// Eq. 4's weighted sum for the tensor-core path: GEMM-2 stored w~ * E(x) per route in bf16, sorted by
// expert; a token's routes are found through the inverse permutation and summed in fp32, slot order
// (a decode step with a K split: the `parts` planes of a row, in order, inside that).
// The row indices first, then up to eight row loads in flight together (the chain index -> row -> next index is all
// there is to a decode step's few blocks: 10 -> 3 us for 64 tokens).
__global__ void __launch_bounds__(256) combine_rows_kernel(const __nv_bfloat16* __restrict__ O,
                                                           const int32_t* __restrict__ inv_pos, int64_t Tn, int Kr, int d,
                                                           int n_shared, const int32_t* __restrict__ shared0_dev,
                                                           int parts, int64_t part_rows, __nv_bfloat16* __restrict__ y) {
    const int64_t i = blockIdx.x;
    grid_dep_launch();
    grid_dep_wait();
    const int64_t shared0 = shared0_dev != nullptr ? (int64_t)*shared0_dev : Tn * Kr;
    const int n_src = Kr + (n_shared ? 1 : 0);
    for (int c = threadIdx.x * 8; c < d; c += blockDim.x * 8) {
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        auto add = [&](const uint4& v) {
            const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(h2[q]);
                acc[2 * q] += f.x;
                acc[2 * q + 1] += f.y;
            }
        };
        for (int j0 = 0; j0 < n_src; j0 += 8) {
            int64_t row[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = j0 + u;
                row[u] = j < Kr ? (int64_t)inv_pos[i * Kr + j] : (j < n_src ? shared0 + i : -1);
            }
            for (int part = 0; part < parts; ++part) {
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (row[u] >= 0) v[u] = *reinterpret_cast<const uint4*>(O + (part * part_rows + row[u]) * d + c);
#pragma unroll
                for (int u = 0; u < 8; ++u)  // slot order; a row < 0 is a slot merged into an earlier one
                    if (row[u] >= 0) add(v[u]);
            }
        }
        uint4 o;
        __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
        for (int u = 0; u < 4; ++u) o2[u] = __floats2bfloat162_rn(acc[2 * u], acc[2 * u + 1]);
        *reinterpret_cast<uint4*>(y + i * d + c) = o;
    }
}

// The same for prefill, where every slot has a row of its own, with NS rows per token known at compile time: a thread owns
// eight columns and has all NS row loads in flight, and no registers for what decode needs (8192 tokens x 4 rows x 2048:
// 35 us with one load at a time and many blocks per SM, 65 with the kernel above, 24 now = 7 TB/s). Rows are read once: not
// kept in L1.
template <int NS>
__global__ void __launch_bounds__(512) combine_rows_exact_kernel(const __nv_bfloat16* __restrict__ O,
                                                                 const int32_t* __restrict__ inv_pos, int64_t Tn, int Kr, int d,
                                                                 __nv_bfloat16* __restrict__ y) {
    const int64_t i = blockIdx.x;
    grid_dep_launch();
    grid_dep_wait();
    int64_t row[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) row[j] = j < Kr ? (int64_t)inv_pos[i * Kr + j] : Tn * Kr + i;
    for (int c = threadIdx.x * 8; c < d; c += blockDim.x * 8) {
        uint4 v[NS];
#pragma unroll
        for (int j = 0; j < NS; ++j) v[j] = __ldcs(reinterpret_cast<const uint4*>(O + row[j] * d + c));
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < NS; ++j) {
            const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&v[j]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(h2[q]);
                acc[2 * q] += f.x;
                acc[2 * q + 1] += f.y;
            }
        }
        uint4 o;
        __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
        for (int u = 0; u < 4; ++u) o2[u] = __floats2bfloat162_rn(acc[2 * u], acc[2 * u + 1]);
        *reinterpret_cast<uint4*>(y + i * d + c) = o;
    }
}

// r[i][e] = <W_r[e], x_i>, fp32 accumulation in a fixed order: fp32 layers, and bf16 batches too small for the tensor-core
// kernel. A warp takes EW experts x TW tokens: 1 x 1 spreads a small batch over the most warps; 4 x 4 reads a quarter of
// the bytes through L2 and converts a quarter as often. The order of a score's sum is the same (lane partition, fused
// multiply-adds, shuffle tree).
template <typename T, int EW, int TW>
__global__ void __launch_bounds__(256) router_simt_kernel(const T* __restrict__ x, const T* __restrict__ wr, int64_t Tn,
                                                          int N, int d, float* __restrict__ out, DeviceStatus* status) {
    const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    grid_dep_launch();
    grid_dep_wait();  // x may be the output of the previous layer's last kernel
    if (status != nullptr && blockIdx.x == 0 && threadIdx.x < 4) reinterpret_cast<int*>(status)[threadIdx.x] = 0;
    const int eg = (N + EW - 1) / EW;
    const int64_t i0 = w / eg * TW;
    if (i0 >= Tn) return;
    const int e0 = (int)(w % eg) * EW;
    const T* xi[TW];
    const T* we[EW];
#pragma unroll
    for (int t = 0; t < TW; ++t) xi[t] = x + (i0 + t < Tn ? i0 + t : Tn - 1) * d;
#pragma unroll
    for (int u = 0; u < EW; ++u) we[u] = wr + (size_t)min(e0 + u, N - 1) * d;
    float acc[EW][TW];
#pragma unroll
    for (int u = 0; u < EW; ++u)
#pragma unroll
        for (int t = 0; t < TW; ++t) acc[u][t] = 0.f;
    if constexpr (sizeof(T) == 2) {  // bf16: 8 elements (16 bytes) per lane and step; d is a multiple of 64
#pragma unroll 2
        for (int c = lane * 8; c < d; c += 256) {
            uint4 a[EW], b[TW];
#pragma unroll
            for (int u = 0; u < EW; ++u) a[u] = *reinterpret_cast<const uint4*>(we[u] + c);
#pragma unroll
            for (int t = 0; t < TW; ++t) b[t] = *reinterpret_cast<const uint4*>(xi[t] + c);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 fa[EW];
#pragma unroll
                for (int u = 0; u < EW; ++u) fa[u] = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&a[u])[j]);
#pragma unroll
                for (int t = 0; t < TW; ++t) {
                    const float2 fb = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&b[t])[j]);
#pragma unroll
                    for (int u = 0; u < EW; ++u) {
                        acc[u][t] = fmaf(fa[u].x, fb.x, acc[u][t]);
                        acc[u][t] = fmaf(fa[u].y, fb.y, acc[u][t]);
                    }
                }
            }
        }
    } else {
        for (int c = lane; c < d; c += 32) {
            float fa[EW];
#pragma unroll
            for (int u = 0; u < EW; ++u) fa[u] = (float)we[u][c];
#pragma unroll
            for (int t = 0; t < TW; ++t) {
                const float fb = (float)xi[t][c];
#pragma unroll
                for (int u = 0; u < EW; ++u) acc[u][t] = fmaf(fa[u], fb, acc[u][t]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < EW; ++u)
#pragma unroll
        for (int t = 0; t < TW; ++t) {
            float v = acc[u][t];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane == 0 && e0 + u < N && i0 + t < Tn) out[(i0 + t) * N + e0 + u] = v;
        }
}

// bf16: 4 x 4 scores per warp once that leaves two warps per SM (Qwen3-shaped prefill of 100 tokens 205.7 -> 202.6 us); fp32 rows
// are too short for it (150 tokens x 64 experts x 512: 86.0 us, 89.8 with the tile)
constexpr int kRouterTileWarps = 296;
}  // namespace

cudaError_t launch_router_simt(const void* x, const void* wr, int dtype, int64_t T, int N, int d, float* out,
                               DeviceStatus* status, cudaStream_t s) {
    if (T * N == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((T * N + 7) / 8);
    if (dtype != EXFOLD_BF16)
        return launch_pdl(router_simt_kernel<float, 1, 1>, grid, 256, 0, s, reinterpret_cast<const float*>(x),
                          reinterpret_cast<const float*>(wr), T, N, d, out, status);
    const __nv_bfloat16* xb = reinterpret_cast<const __nv_bfloat16*>(x);
    const __nv_bfloat16* wb = reinterpret_cast<const __nv_bfloat16*>(wr);
    const int64_t tiles = (T + 3) / 4 * ((N + 3) / 4);
    if (tiles >= kRouterTileWarps)
        return launch_pdl(router_simt_kernel<__nv_bfloat16, 4, 4>, (unsigned)((tiles + 7) / 8), 256, 0, s, xb, wb, T, N, d, out, status);
    return launch_pdl(router_simt_kernel<__nv_bfloat16, 1, 1>, grid, 256, 0, s, xb, wb, T, N, d, out, status);
}

cudaError_t launch_combine_rows(const __nv_bfloat16* O, const int32_t* inv_pos, int64_t T, int Kr, int d,
                                int n_shared, const int32_t* shared0_dev, int parts, int64_t part_rows,
                                __nv_bfloat16* y, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    if (parts == 1 && shared0_dev == nullptr) {
        const int threads = std::min(512, (d / 8 + 31) / 32 * 32);
        switch (Kr + (n_shared ? 1 : 0)) {
#define EXFOLD_COMBINE(NS) \
    case NS: return launch_pdl(combine_rows_exact_kernel<NS>, (unsigned)T, threads, 0, s, O, inv_pos, T, Kr, d, y);
            EXFOLD_COMBINE(2) EXFOLD_COMBINE(3) EXFOLD_COMBINE(4) EXFOLD_COMBINE(5) EXFOLD_COMBINE(6) EXFOLD_COMBINE(7)
            EXFOLD_COMBINE(8) EXFOLD_COMBINE(9)
#undef EXFOLD_COMBINE
        }
    }
    return launch_pdl(combine_rows_kernel, (unsigned)T, 256, 0, s, O, inv_pos, T, Kr, d, n_shared, shared0_dev, parts, part_rows, y);
}

}  // namespace exfold
