// Prefill routing: Top-K gate (Eq. 2), retained-set selection (Eq. 10), minimum-loss
// assignment (Eq. 12), weight folding (Eq. 13) and the expert-sorted permutation.
//
//   route kernel   one warp per token; lane l holds logits l, l+32, ...; after the Top-K
//                  rounds lane k (k < K) owns route k. Writes ids/w/omitted pairs and a
//                  per-block histogram of retained experts.
//   scatter kernel same token->block map as the route kernel. Each block first derives its own
//                  bases: the route kernel left one histogram row per block and, added up with
//                  integer atomics (order-independent), one per super-block of 64 blocks; a block
//                  sums the super-block rows (all of them: group sizes; those before its own:
//                  earlier routes) and the at most 63 block rows before it inside its super-block,
//                  then takes a prefix over experts (block 0 also publishes offsets and the
//                  row-tile prefix for the GEMM work list). It then ranks its routes in (token,
//                  slot) order, so the permutation is the stable sort by expert and is
//                  bit-reproducible; it also gathers the token rows into sorted order.
#include <algorithm>

#include "common.cuh"
#include "route_token.cuh"

namespace exfold {

namespace {

template <int NPL>  // logits per lane = ceil(N / 32)
__global__ void __launch_bounds__(kRouteMaxThreads) prefill_route_kernel(PrefillRouteParams p) {
    __shared__ int hist[kMaxExperts];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int kWarps = blockDim.x >> 5;
    grid_dep_launch();
    for (int e = threadIdx.x; e < p.N; e += blockDim.x) hist[e] = 0;
    __syncthreads();
    grid_dep_wait();
    if (p.status != nullptr && blockIdx.x == 0 && threadIdx.x < 4) reinterpret_cast<int*>(p.status)[threadIdx.x] = 0;
    if (p.queue != nullptr && blockIdx.x == 0 && threadIdx.x < 2) p.queue[threadIdx.x] = 0;

    const int N = p.N, Kp = p.Kp, Ko = p.K - p.Kp;
    const int64_t tok0 = (int64_t)blockIdx.x * kRouteTokensPerBlock;
    // the next token's logits are fetched while the current token is processed
    float vn[NPL];
    {
        const int64_t i0 = tok0 + warp;
#pragma unroll
        for (int q = 0; q < NPL; ++q) {
            const int e = lane + 32 * q;
            vn[q] = (i0 < p.T && warp < kRouteTokensPerBlock && e < N) ? p.logits[i0 * N + e] : -INFINITY;
        }
    }
    for (int tl = warp; tl < kRouteTokensPerBlock; tl += kWarps) {
        const int64_t i = tok0 + tl;
        if (i >= p.T) break;
        float v[NPL];
#pragma unroll
        for (int q = 0; q < NPL; ++q) v[q] = vn[q];
        {
            const int64_t in = i + kWarps;
            const bool more = tl + kWarps < kRouteTokensPerBlock && in < p.T;
#pragma unroll
            for (int q = 0; q < NPL; ++q) {
                const int e = lane + 32 * q;
                vn[q] = (more && e < N) ? p.logits[in * N + e] : -INFINITY;
            }
        }
        const TokenRoute r = route_token<NPL>(p, v, lane);
        if (r.kept) {
            p.ids[i * Kp + r.rank] = r.id;
            p.w[i * Kp + r.rank] = r.w;
            atomicAdd(&hist[r.id], 1);
        } else if (r.omitted) {
            if (p.omit_src) p.omit_src[i * Ko + (r.rank - Kp)] = r.id;
            if (p.omit_tgt) p.omit_tgt[i * Ko + (r.rank - Kp)] = r.tgt;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < N; e += blockDim.x) {
        const int h = hist[e];
        p.block_hist[(size_t)blockIdx.x * N + e] = h;
        if (h != 0 && p.sb_hist != nullptr) atomicAdd(&p.sb_hist[(size_t)(blockIdx.x / kRouteSuperBlock) * N + e], h);
    }
}

// Exclusive prefix over N <= 256 counters held one per thread (threads e < N), all threads of the block call it;
// *total receives the sum. `warp_tot` is shared scratch of kMaxExperts / 32 words.
__device__ __forceinline__ int block_prefix(int v, int N, int* warp_tot, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = 0;
    if (warp * 32 < N) {
        incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) warp_tot[warp] = incl;
    }
    __syncthreads();
    int before = 0, all = 0;
    for (int w = 0; w * 32 < N; ++w) {
        if (w < warp) before += warp_tot[w];
        all += warp_tot[w];
    }
    __syncthreads();
    *total = all;
    return before + incl - v;
}

// `split` blocks share a block of tokens: each derives the same bases and positions, the first writes the metadata, and the
// rows to gather are dealt over them (few tokens would otherwise leave most SMs without rows to copy).
__global__ void __launch_bounds__(kRouteThreads) prefill_scatter_kernel(PrefillScatterParams p) {
    __shared__ int cnt[kMaxExperts];
    __shared__ int pos[kRouteTokensPerBlock * kMaxTopK];
    __shared__ int pre[kMaxExperts];  // routes of expert e in earlier blocks
    __shared__ int tot[kMaxExperts];  // routes of expert e in all blocks
    __shared__ int warp_tot[kMaxExperts / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int N = p.N, Kp = p.Kp;
    const int blk = (int)blockIdx.x / p.split, part = (int)blockIdx.x - blk * p.split;
    const int64_t tok0 = (int64_t)blk * kRouteTokensPerBlock;
    const int ntok = (int)min((int64_t)kRouteTokensPerBlock, p.T - tok0);
    const int n = ntok * Kp;
    const int64_t r0 = tok0 * Kp;
    for (int e = threadIdx.x; e < N; e += blockDim.x) pre[e] = tot[e] = 0;
    __syncthreads();
    grid_dep_launch();
    grid_dep_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.zero_words; i += gridDim.x * blockDim.x) p.zero[i] = 0;
    // Bases of this block: first sorted position of expert e = (rows of experts < e) + (rows of e in
    // earlier blocks). Super-block rows first (nsb of them), then the block rows before this one inside
    // its super-block: nsb + 63 rows of N counters at most, whatever the token count. With a single
    // super-block the block rows serve both sums.
    {
        const int sb = blk / kRouteSuperBlock, nsb = (p.nblk + kRouteSuperBlock - 1) / kRouteSuperBlock;
        const bool one = nsb == 1;
        const int b0 = sb * kRouteSuperBlock;
        const int n_rows = one ? p.nblk : nsb + blk - b0;
        for (int idx = threadIdx.x; idx < n_rows * N; idx += blockDim.x) {
            const int row = idx / N, e = idx - row * N;
            if (one) {
                const int v = p.block_hist[idx];
                if (v != 0) {
                    atomicAdd(&tot[e], v);
                    if (row < blk) atomicAdd(&pre[e], v);
                }
            } else if (row < nsb) {
                const int v = p.sb_hist[(size_t)row * N + e];
                if (v != 0) {
                    atomicAdd(&tot[e], v);
                    if (row < sb) atomicAdd(&pre[e], v);
                }
            } else {
                const int v = p.block_hist[(size_t)(b0 + row - nsb) * N + e];
                if (v != 0) atomicAdd(&pre[e], v);
            }
        }
    }
    __syncthreads();
    {
        const int e = threadIdx.x;  // N <= 256 <= the block
        const int rows = e < N ? tot[e] : 0;
        int all_rows, all_tiles;
        const int off = block_prefix(rows, N, warp_tot, &all_rows);
        if (e < N) cnt[e] = off + pre[e];
        if (blockIdx.x == 0) {  // group offsets and the row-tile prefix for the GEMM work list
            const int tiles = row_tiles(rows, p.tile_rows);
            const int tile0 = block_prefix(tiles, N, warp_tot, &all_tiles);
            if (e < N) {
                p.offsets[e] = off;
                p.work_start[e] = tile0;
            }
            if (e == 0) {
                p.offsets[N] = all_rows;
                p.work_start[N] = all_tiles;
                if (p.n_shared) {
                    p.offsets[N + 1] = all_rows + (int)p.T;
                    p.work_start[N + 1] = all_tiles + row_tiles((int)p.T, p.tile_rows);
                }
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        // routes of this block in (token, slot) order, 32 at a time
        for (int c0 = 0; c0 < n; c0 += 32) {
            int r = c0 + lane;
            int e = r < n ? p.ids[r0 + r] : -1 - lane;
            unsigned m = __match_any_sync(0xffffffffu, e);
            int before = __popc(m & ((1u << lane) - 1u));
            int base = r < n ? cnt[e] : 0;
            __syncwarp();
            if (r < n) {
                pos[r] = base + before;
                if (before == __popc(m) - 1) cnt[e] = base + __popc(m);  // last lane of the group updates
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int r = threadIdx.x; part == 0 && r < n; r += blockDim.x) {
        int q = pos[r];
        int64_t route = r0 + r;
        p.perm[q] = (int32_t)route;
        if (p.inv_pos != nullptr) p.inv_pos[route] = q;
        p.row_tok[q] = (int32_t)(route / Kp);
        p.row_w[q] = p.w[route];
    }
    if (p.n_shared && part == 0) {  // shared-expert rows follow the routed rows, identity order, weight 1
        const int64_t R = p.T * Kp;
        for (int t = threadIdx.x; t < ntok; t += blockDim.x) {
            p.row_tok[R + tok0 + t] = (int32_t)(tok0 + t);
            p.row_w[R + tok0 + t] = 1.0f;
        }
    }
    if (p.xs != nullptr && p.d_bytes > 0) {
        // gather: sorted row pos[r] <- token row; one warp per route, 16-byte chunks
        const int chunks = p.d_bytes >> 4;
        const int nwarps = blockDim.x >> 5;
        for (int r = part * nwarps + warp; r < n; r += p.split * nwarps) {
            const uint4* src = reinterpret_cast<const uint4*>(
                reinterpret_cast<const char*>(p.x) + (size_t)((r0 + r) / Kp) * p.d_bytes);
            uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<char*>(p.xs) + (size_t)pos[r] * p.d_bytes);
            for (int c = lane; c < chunks; c += 32) dst[c] = __ldg(src + c);
        }
    }
}

}  // namespace

cudaError_t launch_prefill_route(PrefillRouteParams p, cudaStream_t s) {
    const int nblk = (int)((p.T + kRouteTokensPerBlock - 1) / kRouteTokensPerBlock);
    const int npl = (p.N + 31) / 32;
    // No more blocks than SMs: a warp per token, the time is one token's chain of loads and reductions (777 tokens of 128
    // experts 9.6 -> 7.9 us). More blocks fill the SMs either way (8192 tokens 17.2 us, with a warp per token 17.7).
    const int threads = nblk <= kRouteFewBlocks ? kRouteMaxThreads : kRouteThreads;
    if (nblk <= kRouteSuperBlock) {
        p.sb_hist = nullptr;  // one super-block: the scatter kernel adds up the block rows itself
    } else {  // the super-block histograms are added up with atomics: they start at zero
        const size_t nsb = (size_t)(nblk + kRouteSuperBlock - 1) / kRouteSuperBlock;
        cudaError_t e = cudaMemsetAsync(p.sb_hist, 0, nsb * p.N * sizeof(int32_t), s);
        if (e != cudaSuccess) return e;
    }
    switch (npl) {
        case 1: return launch_pdl(prefill_route_kernel<1>, nblk, threads, 0, s, p);
        case 2: return launch_pdl(prefill_route_kernel<2>, nblk, threads, 0, s, p);
        case 3: case 4: return launch_pdl(prefill_route_kernel<4>, nblk, threads, 0, s, p);
        default: return launch_pdl(prefill_route_kernel<8>, nblk, threads, 0, s, p);
    }
}

cudaError_t launch_prefill_scatter(PrefillScatterParams p, cudaStream_t s) {
    const int nblk = (int)((p.T + kRouteTokensPerBlock - 1) / kRouteTokensPerBlock);
    // a warp copies a row at a time: as many blocks per token block as leave every warp a row or two, on ~2 blocks per SM
    // (777 tokens x 6 rows of 4 KB: 25 blocks 22.2 us, 275 blocks 12.1)
    const int64_t rows_per_block = (int64_t)kRouteTokensPerBlock * p.Kp;
    p.split = 1;
    if (p.xs != nullptr && p.d_bytes > 0)
        p.split = (int)std::max<int64_t>(1, std::min<int64_t>(2 * kRouteFewBlocks / nblk, rows_per_block / (kRouteThreads / 32)));
    return launch_pdl(prefill_scatter_kernel, nblk * p.split, kRouteThreads, 0, s, p);
}

}  // namespace exfold
