// Router scores of bf16 prompts (Eq. 2: r = W_r x) on the tensor cores, K split over a cluster.
//
// One output tile is 128 tokens x all N experts, so a prompt of T tokens has only T / 128 of them: with one CTA per tile a
// 777-token prompt walked all of K = 2048 on 7 SMs (17 us, of which the arithmetic is 12 one-SM microseconds). Here a cluster of
// `split` CTAs shares a tile, each multiplying its part of K into its own tensor memory; the fp32 partial tiles meet in
// shared memory, and every CTA sums a share of the rows over the cluster through distributed shared memory, in rank order
// (deterministic), and writes them. What bounds it then is latency: launch, first TMA loads, the exchange. Measured with the
// one-CTA-per-tile kernel before it: 777 tokens x 128 experts x 2048 17.2 (+ 3.7 for a memset of the status record) -> 9.2 us;
// whole Qwen3-shaped prefill with the router 200 tokens 230 -> 221 us, 777 258 -> 250, 8192 514 -> 508.
//
// The first kernel of a call: CTA 0 clears the status record. The waits here therefore do not look at the record (an
// earlier call's code may still stand in it); a wait that runs out reports two seconds later, long after the clearing.
#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"

#include <cooperative_groups.h>

namespace exfold {

namespace {

namespace cg = cooperative_groups;

constexpr int kRThreads = 192;  // warp 0: TMA producer, warp 1: MMA issuer, warps 2-5: accumulator rows
constexpr int kRMaxStages = 6;
constexpr int kRBK = 64;

// Bounded wait that looks at the CTA's own abort flag only
__device__ __forceinline__ bool wait_local(uint64_t* bar, uint32_t parity, volatile int* abort_flag, DeviceStatus* st, int where) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = ptx::globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 0u) {
            if (*abort_flag) return false;
            if (ptx::globaltimer_ns() - t0 > ptx::kWaitLimitNs) {
                *abort_flag = 1;
                report_timeout(st, where);
                return false;
            }
        }
    }
}

__global__ void __launch_bounds__(kRThreads, 1) router_gemm_kernel(const __grid_constant__ RouterGemmParams p) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kRMaxStages];
    __shared__ __align__(8) uint64_t empty_bar[kRMaxStages];
    __shared__ __align__(8) uint64_t done_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    unsigned char* tiles =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    cg::cluster_group cluster = cg::this_cluster();
    const int split = p.split, rank = (int)cluster.block_rank();
    const int row0 = (int)blockIdx.x / split * 128;
    if (threadIdx.x == 0) {
        ptx::prefetch_tmap(&p.tm_x);
        ptx::prefetch_tmap(&p.tm_wr);
        for (int s = 0; s < kRMaxStages; ++s) {
            ptx::mbar_init(&full_bar[s], 1);
            ptx::mbar_init(&empty_bar[s], 1);
        }
        ptx::mbar_init(&done_bar, 1);
        abort_s = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(&tmem_base_s, p.tmem_cols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    grid_dep_wait();
    if (p.clear_status && blockIdx.x == 0 && threadIdx.x < 4) reinterpret_cast<int*>(p.status)[threadIdx.x] = 0;
    const uint32_t tmem_base = tmem_base_s;
    volatile int* abort_flag = &abort_s;
    const int kb0 = rank * p.nkb / split, kb1 = (rank + 1) * p.nkb / split;  // never empty: split <= nkb
    const int a_bytes = 128 * kRBK * 2, stage_bytes = a_bytes + p.npad * kRBK * 2;

    if (warp == 0) {
        if (ptx::elect_one()) {
            int stage = 0, phase = 0;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!wait_local(&empty_bar[stage], phase ^ 1, abort_flag, p.status, 1)) break;
                unsigned char* dst = tiles + stage * stage_bytes;
                ptx::mbar_expect_tx(&full_bar[stage], stage_bytes);
                ptx::tma_load_2d(dst, &p.tm_x, &full_bar[stage], kb * kRBK, row0);
                ptx::tma_load_2d(dst + a_bytes, &p.tm_wr, &full_bar[stage], kb * kRBK, 0);
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (ptx::elect_one()) {
            const uint32_t idesc = ptx::make_idesc_bf16(128, p.npad);
            const uint32_t lo0 = (ptx::smem_u32(tiles) & 0x3FFFFu) >> 4;
            const uint32_t hi = (uint32_t)(ptx::make_kmajor_sw128_desc(0) >> 32);
            int stage = 0, phase = 0;
            bool ok = true, ready = false;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!ready && !wait_local(&full_bar[stage], phase, abort_flag, p.status, 3)) {
                    ok = false;
                    break;
                }
                const int ns = stage + 1 == p.stages ? 0 : stage + 1, nphase = ns == 0 ? phase ^ 1 : phase;
                const uint32_t a_lo = lo0 + (uint32_t)(stage * stage_bytes >> 4);
                ready = ptx::umma_kblock_bf16(tmem_base, a_lo, a_lo + (a_bytes >> 4), hi, idesc, kb > kb0 ? 1u : 0u,
                                              &empty_bar[stage], &full_bar[ns], nphase);
                stage = ns;
                phase = nphase;
            }
            if (ok) ptx::umma_commit(&done_bar);
        }
        __syncwarp();
    } else {
        // partial tile -> shared memory (the ring is free once every MMA has completed)
        const int q = warp & 3;
        int ok = 1;
        if (lane == 0) ok = wait_local(&done_bar, 0, abort_flag, p.status, 4) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (ok) {
            ptx::tc_fence_after();
            float* dst = reinterpret_cast<float*>(tiles) + (size_t)(q * 32 + lane) * p.part_ld;
            for (int c = 0; c < p.npad; c += 32) {
                uint32_t v[32];
                ptx::tmem_ld32(tmem_base + c + ((uint32_t)(q * 32) << 16), v);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<uint4*>(dst + c + 4 * j) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (abort_s) __nanosleep(100000);  // let any copy still in flight land before shared memory is released
    cluster.sync();                    // every part of the tile is in place
    {
        const int rows = 128 / split, r_lo = rank * rows;
        const int vec = p.N % 4 == 0 ? p.N / 4 : 0;  // whole float4 columns, or element by element
        const int cols = vec ? vec : p.N;
        for (int i = threadIdx.x; i < rows * cols; i += kRThreads) {
            const int r = r_lo + i / cols, c = i % cols;
            if (row0 + r >= p.T) continue;
            const size_t at = (size_t)r * p.part_ld + (vec ? 4 * c : c);
            float* out = p.logits + (size_t)(row0 + r) * p.N + (vec ? 4 * c : c);
            if (vec) {
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int k = 0; k < split; ++k) {
                    const float4 v = *reinterpret_cast<const float4*>(cluster.map_shared_rank(reinterpret_cast<float*>(tiles), k) + at);
                    s.x += v.x;
                    s.y += v.y;
                    s.z += v.z;
                    s.w += v.w;
                }
                *reinterpret_cast<float4*>(out) = s;
            } else {
                float s = 0.f;
                for (int k = 0; k < split; ++k) s += cluster.map_shared_rank(reinterpret_cast<float*>(tiles), k)[at];
                *out = s;
            }
        }
    }
    grid_dep_launch();
    cluster.sync();  // no CTA leaves while its part may still be read
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, p.tmem_cols);
    }
}

}  // namespace

int router_npad(int N) { return (N + 31) / 32 * 32; }

// K split: as many CTAs per tile as fill the chip (a power of two up to 8), each with four k-blocks at least
cudaError_t launch_router_gemm(RouterGemmParams p, int sms, cudaStream_t s) {
    const int tiles = (p.T + 127) / 128;
    p.split = 1;
    while (p.split < 8 && tiles * p.split * 2 <= sms && p.nkb >= 8 * p.split) p.split *= 2;
    p.npad = router_npad(p.N);
    p.part_ld = p.npad + 4;  // floats: 16-byte aligned rows, the rows of a quarter warp in distinct banks
    p.tmem_cols = 32;
    while ((int)p.tmem_cols < p.npad) p.tmem_cols *= 2;
    const int stage_bytes = (128 + p.npad) * kRBK * 2;
    const int per = (p.nkb + p.split - 1) / p.split;
    p.stages = std::max(2, std::min(std::min(kRMaxStages, per), 200 * 1024 / stage_bytes));
    const size_t smem = std::max((size_t)p.stages * stage_bytes, (size_t)128 * p.part_ld * sizeof(float)) + 1024;
    cudaError_t err = ensure_smem(router_gemm_kernel, smem);
    if (err != cudaSuccess) return err;
    return launch_pdl_cluster(router_gemm_kernel, (unsigned)(tiles * p.split), kRThreads, smem, p.split, s, p);
}

}  // namespace exfold
