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
// Top-K and routing weights of N tokens by one warp, from their logits v (-inf beyond n_cand).  On return lane
// k < K holds slot k of each, m the logits' maxima and, where DEN asks for them, den the softmax denominators.
// RPL = logits per lane (32 * RPL >= n_cand).
//
// What bounds it is the chain of dependent instructions (a token's 8 rounds over 192 candidates took 3.2 us on an
// SM of 16 warps), so each lane sorts its logits first: a round is then one warp maximum over the lanes' best, a
// ballot, and a shift in the lane that held it; and where a warp has several tokens it takes two at a time.  The
// largest logit is the first round's, and the denominator, which normalised weights do not need (it cancels), is
// summed for the raw softmax and the statistics only.
// Two logits a lane (up to 64 candidates) are not sorted: a maximum over them and a second warp reduction, for the
// lowest id, are less work than the ballot and the shuffle (routing pass of 64 candidates, us, sorted and not: K 8, 1500
// tokens 18.2, 15.0; 2048 tokens 20.2, 16.6; K 16, 2048 tokens 25.1, 19.0), and more than eight would take longer to
// sort than the rounds.
template <int RPL>
constexpr bool kSortedLogits = RPL > 2 && RPL <= 8;

template <int RPL, int N, bool DEN = false>
__device__ __forceinline__ void topk_gate_select(const float (&v)[N][RPL], int n_real, int n_cand, int K, int gate_mode, int lane,
                                                 float (&m)[N], float (&den)[N], int (&my_idx)[N], float (&my_w)[N]) {
    // Selection on order-preserving integer keys (0 = not available), so that one warp-wide integer
    // maximum finds the best logit.
    unsigned key[N][RPL], my_key[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            unsigned u = __float_as_uint(v[n][r]);
            if (u == 0x80000000u) u = 0u;  // -0 and +0 are equal logits: the lower id decides between them
            // (a candidate's key is never 0, not even for the NaN whose key would be: no candidate is taken twice)
            key[n][r] = (r * 32 + lane < n_cand) ? max((u & 0x80000000u) ? ~u : (u | 0x80000000u), 1u) : 0u;
        }
        my_key[n] = 0u;
        my_idx[n] = -1;
        m[n] = 0.f;
    }
    auto logit_of = [](unsigned k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k); };
    if constexpr (kSortedLogits<RPL>) {
        // the lane's keys in falling order (equal ones by rising id: neighbours change places only where the second is
        // larger), and which of its registers they came from, four bits each
        unsigned from[N];
#pragma unroll
        for (int n = 0; n < N; ++n) {
            unsigned reg[RPL];
#pragma unroll
            for (int r = 0; r < RPL; ++r) reg[r] = r;
#pragma unroll
            for (int pass = 0; pass < RPL; ++pass)
#pragma unroll
                for (int r = pass & 1; r + 1 < RPL; r += 2) {
                    const bool swap = key[n][r + 1] > key[n][r];
                    const unsigned hi = max(key[n][r], key[n][r + 1]), lo = min(key[n][r], key[n][r + 1]);
                    const unsigned a = swap ? reg[r + 1] : reg[r], b = swap ? reg[r] : reg[r + 1];
                    key[n][r] = hi;
                    key[n][r + 1] = lo;
                    reg[r] = a;
                    reg[r + 1] = b;
                }
            from[n] = 0u;
#pragma unroll
            for (int r = 0; r < RPL; ++r) from[n] |= reg[r] << (4 * r);
        }
        for (int k = 0; k < K; ++k) {
            unsigned gm[N], held[N];
#pragma unroll
            for (int n = 0; n < N; ++n) gm[n] = __reduce_max_sync(kFull, key[n][0]);
#pragma unroll
            for (int n = 0; n < N; ++n) held[n] = __ballot_sync(kFull, key[n][0] == gm[n]);
#pragma unroll
            for (int n = 0; n < N; ++n) {
                int winner = __ffs(held[n]) - 1;
                if (held[n] & (held[n] - 1u))  // equal logits in several lanes: the lowest id
                    winner = __reduce_min_sync(kFull, key[n][0] == gm[n] ? (from[n] & 15u) * 32 + lane : 0x7fffffffu) & 31;
                const int id = (__shfl_sync(kFull, from[n], winner) & 15u) * 32 + winner;
                if (lane == k) { my_idx[n] = id; my_key[n] = gm[n]; }
                if (k == 0) m[n] = logit_of(gm[n]);
                if (lane == winner) {
#pragma unroll
                    for (int r = 0; r + 1 < RPL; ++r) key[n][r] = key[n][r + 1];
                    key[n][RPL - 1] = 0u;
                    from[n] >>= 4;
                }
            }
        }
    } else {
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int n = 0; n < N; ++n) {
                unsigned lm = key[n][0];
#pragma unroll
                for (int r = 1; r < RPL; ++r) lm = max(lm, key[n][r]);
                const unsigned gm = __reduce_max_sync(kFull, lm);
                int cand = 0x7fffffff;
#pragma unroll
                for (int r = RPL - 1; r >= 0; --r)
                    if (key[n][r] == gm) cand = r * 32 + lane;  // ends on this lane's lowest id with that logit
                const int bj = __reduce_min_sync(kFull, cand);
#pragma unroll
                for (int r = 0; r < RPL; ++r)
                    if (r * 32 + lane == bj) key[n][r] = 0u;
                if (lane == k) { my_idx[n] = bj; my_key[n] = gm; }
                if (k == 0) m[n] = logit_of(gm);
            }
    }
    // a NaN among the logits, selected or not, is one in every weight (in Eq. 7's, whose sum is then not above 0, a zero)
#pragma unroll
    for (int n = 0; n < N; ++n) {
        bool bad = false;
#pragma unroll
        for (int r = 0; r < RPL; ++r) bad |= v[n][r] != v[n][r];
        if (__any_sync(kFull, bad)) m[n] = __int_as_float(0x7fffffff);
    }
    if (DEN || gate_mode == ZEDA_GATE_SOFTMAX_RAW) {
#pragma unroll
        for (int n = 0; n < N; ++n) {
            den[n] = 0.f;
#pragma unroll
            for (int r = 0; r < RPL; ++r)
                if (r * 32 + lane < n_cand) den[n] += expf(v[n][r] - m[n]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int n = 0; n < N; ++n) den[n] += __shfl_xor_sync(kFull, den[n], o);
    }
    // lane k < K holds slot k: e^(logit - m), over the sum that the gate mode asks for (K <= 16: the lanes above hold
    // zeros)
    static_assert(kMaxTopK <= 16, "the sums run over sixteen lanes");
    float e[N], sum[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        e[n] = lane < K ? expf(logit_of(my_key[n]) - m[n]) : 0.f;
        sum[n] = gate_mode != ZEDA_GATE_RENORM_REAL || (unsigned)my_idx[n] < (unsigned)n_real ? e[n] : 0.f;
    }
    if (gate_mode == ZEDA_GATE_SOFTMAX_RAW) {
#pragma unroll
        for (int n = 0; n < N; ++n) my_w[n] = e[n] / den[n];
        return;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
        for (int n = 0; n < N; ++n) sum[n] += __shfl_xor_sync(kFull, sum[n], o);
#pragma unroll
    for (int n = 0; n < N; ++n) {
        if (gate_mode == ZEDA_GATE_TOPK_NORM) my_w[n] = e[n] / sum[n];
        else my_w[n] = (my_idx[n] < n_real && sum[n] > 0.f) ? e[n] / sum[n] : 0.f;
    }
}

// The same with the token's logits read from memory (and returned in v), one token.
// The row may arrive as n_parts partial sums, part_stride floats apart; they are added in order, PB slices
// requested at a time (one slice after another is a chain of L2 round trips).
template <int RPL, int PB = (RPL <= 8 ? 7 : 3), bool DEN = false>
__device__ __forceinline__ void topk_gate_token(const float *__restrict__ row, int n_parts, size_t part_stride,
                                                int n_real, int n_cand, int K, int gate_mode, int lane,
                                                float (&v)[RPL], float &m, float &den, int &my_idx, float &my_w) {
    float u[1][RPL], mm[1], dd[1], w[1];
    int idx[1];
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
        const int j = r * 32 + lane;
        const float a = __ldcg(row + min(j, n_cand - 1));
        u[0][r] = j < n_cand ? a : -INFINITY;
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
                if (p + q < n_parts) u[0][r] += a[q][r];
    }
    topk_gate_select<RPL, 1, DEN>(u, n_real, n_cand, K, gate_mode, lane, mm, dd, idx, w);
#pragma unroll
    for (int r = 0; r < RPL; ++r) v[r] = u[0][r];
    m = mm[0];
    if (DEN) den = dd[0];
    my_idx = idx[0];
    my_w = w[0];
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
