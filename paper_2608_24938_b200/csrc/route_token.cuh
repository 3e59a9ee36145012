// Routing of one prefill token by one warp: Top-K gate (Eq. 2), retained set (Eq. 10), minimum-loss targets (Eq. 12) and the
// folded weights (Eq. 13). Used by the route kernel and by the two kernels that route in their prologue
// (fp32 FFN, few-token gate/up).
#pragma once
#include "common.cuh"

namespace exfold {

struct TokenRoute {  // of lane k: the token's route k in router order
    int id;          // expert, -1: no such route
    int rank;        // place among the token's routes by score and norm
    bool kept, omitted;
    float w;   // kept: the folded weight
    int tgt;   // omitted: the chosen target (-1: dropped, no admissible target)
};

// v[q]: score of expert lane + 32 q. Whole warp.
template <int NPL>
__device__ __forceinline__ TokenRoute route_token(const PrefillRouteParams& p, const float (&v)[NPL], int lane) {
    const int N = p.N, K = p.K, Kp = p.Kp;
    uint32_t key_q[NPL];
    uint32_t used = 0;
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
        key_q[q] = float_order_key(v[q]);
        if (lane + 32 * q >= N) used |= 1u << q;
    }
    // ---- Eq. 2: K rounds of warp arg-max (hardware reductions); ties -> lower expert id
    int my_id = -1;
    float my_r = 0.f;
    for (int k = 0; k < K; ++k) {
        uint32_t bk = 0;
        int be = 0x7fffffff;
#pragma unroll
        for (int q = 0; q < NPL; ++q) {
            const bool free_q = !((used >> q) & 1u);
            if (free_q && (be == 0x7fffffff || key_q[q] > bk)) {
                bk = key_q[q];
                be = lane + 32 * q;
            }
        }
        uint32_t mk;
        be = warp_argmax(be != 0x7fffffff, bk, be, &mk);
        if ((be & 31) == lane) used |= 1u << (be >> 5);
        if (lane == k) {
            my_id = be;
            my_r = float_from_order_key(mk);
        }
    }
    const bool has = lane < K;
    // softmax restricted to the Top-K set (slot 0 holds the largest logit)
    const float rmax = __shfl_sync(0xffffffffu, my_r, 0);
    float ex = has ? expf(my_r - rmax) : 0.f;
    float sum = ex;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    const float w = ex / sum;
    // ---- Eq. 10 on log scale: key = logit + ln h (one fp32 add); rank by (key desc, id asc). Ranked by the integer images, of
    // which any two compare also where a score or a norm is NaN: the ranks are places in arrays, no two the same, none left out.
    const uint32_t key = has ? float_order_key(__fadd_rn(my_r, p.lnh != nullptr ? p.lnh[my_id] : 0.f)) : 0u;
    int rank = 0;
    for (int j = 0; j < K; ++j) {
        const uint32_t kj = __shfl_sync(0xffffffffu, key, j);
        int ij = __shfl_sync(0xffffffffu, my_id, j);
        if (has && j != lane && (kj > key || (kj == key && ij < my_id))) rank++;
    }
    if (!has) rank = 0x7fff;
    const bool kept = has && rank < Kp;
    const bool omitted = has && rank >= Kp;
    // ---- Eq. 12 + 13, omitted routes in rank order, four at a time. For an omitted source s every
    // retained lane t loads L[s][t] and S[s][t] itself (independent loads, all in flight together);
    // a warp arg-min over (loss, id) picks the target, which then adds w_s * S[s][t] to its weight.
    float wt = w;
    int my_tgt = -1;  // for omitted lanes: the chosen target (-1: dropped, no admissible target)
    float kept_sum = 0.f;  // sum of the retained routes' original weights (confidence split only)
    if (p.confidence) {
        kept_sum = kept ? w : 0.f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) kept_sum += __shfl_xor_sync(0xffffffffu, kept_sum, off);
    }
    for (int rr0 = Kp; rr0 < K; rr0 += 4) {
        int src_lane[4], src_id[4];
        float lv[4], sv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int rr = rr0 + u;
            const unsigned m = __ballot_sync(0xffffffffu, rank == rr);
            src_lane[u] = m ? __ffs(m) - 1 : 0;
            src_id[u] = __shfl_sync(0xffffffffu, my_id, src_lane[u]);
            const bool act = kept && rr < K;
            lv[u] = act ? __ldg(p.L + (size_t)src_id[u] * N + my_id) : INFINITY;
            sv[u] = act ? __ldg(p.S + (size_t)src_id[u] * N + my_id) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (rr0 + u >= K) break;  // warp-uniform
            const bool adm = kept && !(lv[u] > p.loss_thr);  // loss-threshold safeguard
            const int bt = warp_argmin(adm, float_order_key(lv[u]), my_id);
            const float ws = __shfl_sync(0xffffffffu, w, src_lane[u]);
            if (bt != 0x7fffffff) {  // warp-uniform: a target exists
                const bool is_t = kept && my_id == bt;
                float c = 1.0f;
                if (p.confidence) {
                    const unsigned tm = __ballot_sync(0xffffffffu, is_t);
                    const float lt = __shfl_sync(0xffffffffu, lv[u], __ffs(tm) - 1);
                    c = fminf(fmaxf(1.0f - lt, 0.0f), 1.0f);
                    if (kept) wt = __fadd_rn(wt, ws * (1.0f - c) * (w / kept_sum));
                }
                if (is_t) wt = __fadd_rn(wt, __fmul_rn(ws * c, sv[u]));
            }
            if (lane == src_lane[u]) my_tgt = bt == 0x7fffffff ? -1 : bt;
        }
    }
    if (p.rescale) {  // keep the original routed-weight sum
        float fs = kept ? wt : 0.f, as = has ? w : 0.f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            fs += __shfl_xor_sync(0xffffffffu, fs, off);
            as += __shfl_xor_sync(0xffffffffu, as, off);
        }
        if (fs > 0.f) wt *= as / fs;
    }
    TokenRoute r;
    r.id = my_id;
    r.rank = rank;
    r.kept = kept;
    r.omitted = omitted;
    r.w = wt;
    r.tgt = my_tgt;
    return r;
}

}  // namespace exfold
