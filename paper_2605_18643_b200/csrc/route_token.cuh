// Top-K of one token, shared by the routing pass and the expert kernels of the smallest batches.
#pragma once

#include "expert_scan.cuh"

namespace zeda {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// ---------------------------------------------------------------------------------------------
// Softmax, top-K and routing weights: one warp per token, logits held in registers (candidate
// j lives in lane j % 32, register j / 32).  K rounds of warp arg-max; equal logits go to the
// lower candidate id.
// ---------------------------------------------------------------------------------------------
// Top-K and routing weights of one token by one warp.  On return lane k < K holds slot k, and v, m, den
// the logits (-inf beyond n_cand), their maximum and the softmax denominator.
// RPL = logits per lane (32 * RPL >= n_cand).
// The row may arrive as n_parts partial sums, part_stride floats apart; they are added in order, PB slices
// requested at a time (one slice after another is a chain of L2 round trips).
template <int RPL, int PB = (RPL <= 8 ? 7 : 3)>
__device__ __forceinline__ void topk_gate_token(const float *__restrict__ row, int n_parts, size_t part_stride,
                                                int n_real, int n_cand, int K, int gate_mode, int lane,
                                                float (&v)[RPL], float &m, float &den, int &my_idx, float &my_w) {
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
        const int j = r * 32 + lane;
        const float a = __ldcg(row + min(j, n_cand - 1));
        v[r] = j < n_cand ? a : -INFINITY;
    }
    for (int p = 1; p < n_parts; p += PB) {
        float a[PB][RPL];
#pragma unroll
        for (int q = 0; q < PB; ++q)
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
                const int j = r * 32 + lane;
                a[q][r] = ldcg_if(p + q < n_parts && j < n_cand, row + (p + q) * part_stride + j, 0.f);
            }
#pragma unroll
        for (int q = 0; q < PB; ++q)
#pragma unroll
            for (int r = 0; r < RPL; ++r)
                if (p + q < n_parts) v[r] += a[q][r];
    }
    // row maximum and softmax denominator over all candidates
    m = v[0];
#pragma unroll
    for (int r = 1; r < RPL; ++r) m = fmaxf(m, v[r]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    den = 0.f;
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
        const int j = r * 32 + lane;
        if (j < n_cand) den += expf(v[r] - m);
    }
    den = warp_sum(den);

    // Selection on order-preserving integer keys (0 = not available), so that one warp-wide integer
    // maximum finds the best logit and one integer minimum the lowest candidate id that holds it.
    unsigned key[RPL];
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
        unsigned u = __float_as_uint(v[r]);
        if (u == 0x80000000u) u = 0u;  // -0 and +0 are equal logits: the lower id decides between them
        // (a candidate's key is never 0, not even for the NaN whose key would be: no candidate is taken twice)
        key[r] = (r * 32 + lane < n_cand) ? max((u & 0x80000000u) ? ~u : (u | 0x80000000u), 1u) : 0u;
    }
    unsigned my_key = 0u;
    my_idx = -1;
    for (int k = 0; k < K; ++k) {
        unsigned lm = key[0];
#pragma unroll
        for (int r = 1; r < RPL; ++r) lm = max(lm, key[r]);
        const unsigned gm = __reduce_max_sync(kFull, lm);
        int cand = 0x7fffffff;
#pragma unroll
        for (int r = RPL - 1; r >= 0; --r)
            if (key[r] == gm) cand = r * 32 + lane;  // ends on this lane's lowest id with that logit
        const int bj = __reduce_min_sync(kFull, cand);
#pragma unroll
        for (int r = 0; r < RPL; ++r)
            if (r * 32 + lane == bj) key[r] = 0u;
        if (lane == k) { my_idx = bj; my_key = gm; }
    }
    // lane k < K holds slot k: its softmax probability, then the sums over the selected slots
    float my_p = 0.f;
    if (lane < K) {
        const float bv = __uint_as_float((my_key & 0x80000000u) ? (my_key & 0x7fffffffu) : ~my_key);
        my_p = expf(bv - m) / den;
    }
    const float sum_sel = warp_sum(my_p);
    const float sum_real = warp_sum(my_idx >= 0 && my_idx < n_real ? my_p : 0.f);
    my_w = my_p;
    if (gate_mode == ZEDA_GATE_TOPK_NORM) my_w = my_p / sum_sel;
    else if (gate_mode == ZEDA_GATE_RENORM_REAL) my_w = (my_idx < n_real && sum_real > 0.f) ? my_p / sum_real : 0.f;
}

// CALL(logits per lane) for n_cand candidates
#define ZEDA_RPL_DISPATCH(CALL)              \
    do {                                     \
        if (n_cand <= 64) { CALL(2); }       \
        else if (n_cand <= 128) { CALL(4); } \
        else if (n_cand <= 192) { CALL(6); } \
        else if (n_cand <= 256) { CALL(8); } \
        else { CALL(16); }                   \
    } while (0)

}  // namespace zeda
