// Weighted combine back to token order: the sum of Eq. 1,
//   y[t] = sum over the slots k of token t that hold a normal expert of g~[t,k] * O[inv[t,k]],
// taken in slot order in fp32 and rounded once to bf16.  It is a gather, not a scatter with
// atomics, so the result is the same bits on every run, and a token with no surviving slot gets
// +0 in every element.  The copy-expert variant (Appendix B) adds (sum of zero-slot weights) * x[t].
#include "zeda_internal.h"

namespace zeda {

namespace {

__device__ __forceinline__ void fma_bf16x8(float (&acc)[8], float w, const uint4 &v) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        acc[2 * i] = fmaf(w, __uint_as_float(u[i] << 16), acc[2 * i]);
        acc[2 * i + 1] = fmaf(w, __uint_as_float(u[i] & 0xffff0000u), acc[2 * i + 1]);
    }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&b);
}

__device__ __forceinline__ uint4 pack_bf16x8(const float (&a)[8]) {
    return make_uint4(pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]), pack_bf16(a[4], a[5]), pack_bf16(a[6], a[7]));
}

// A warp's share of a token's row: P * 32 16-byte chunks from chunk c0 on, chunk c0 + 32 p + lane in acc[p] (those beyond the
// row stay zero).  Lane k holds slot k: its position in the expert outputs (-1 for a zero slot) and its weight.  Only the
// surviving slots are walked, in slot order, ROWS at a time: P * ROWS loads of 16 bytes per lane in flight.
template <int P, int ROWS>
__device__ __forceinline__ void combine_chunks(float (&acc)[P][8], const __nv_bfloat16 *__restrict__ obuf, const int32_t *__restrict__ inv,
                                               const float *__restrict__ topk_w, const __nv_bfloat16 *__restrict__ x, int t, int c0, int K,
                                               int d, int copy_experts, int lane) {
    const int my_pos = lane < K ? __ldcg(inv + (size_t)t * K + lane) : -1;
    const float my_w = lane < K ? __ldcg(topk_w + (size_t)t * K + lane) : 0.f;
    const unsigned real = __ballot_sync(0xffffffffu, my_pos >= 0);
    const int c = c0 + lane, chunks = d / 8;
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[p][i] = 0.f;
    for (unsigned left = real; left;) {  // (uniform over the warp)
        uint4 v[ROWS][P];
        float w[ROWS];
        const int n = __popc(left);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int k = r < n ? __ffs(left) - 1 : 0;
            left &= left - 1u;
            w[r] = __shfl_sync(0xffffffffu, my_w, k);
            const int pos = __shfl_sync(0xffffffffu, my_pos, k);
            const uint4 *row = reinterpret_cast<const uint4 *>(obuf + (size_t)pos * d) + c;
#pragma unroll
            for (int p = 0; p < P; ++p)
                if (r < n && c + 32 * p < chunks) v[r][p] = __ldcg(row + 32 * p);
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int p = 0; p < P; ++p)
                if (r < n && c + 32 * p < chunks) fma_bf16x8(acc[p], w[r], v[r][p]);
    }
    if (!copy_experts) return;
    float zero_mass = 0.f;  // the summed weight of the zero slots
    for (int k = 0; k < K; ++k) {
        const float w = __shfl_sync(0xffffffffu, my_w, k);
        if (!(real >> k & 1u)) zero_mass += w;
    }
    if (zero_mass == 0.f) return;
#pragma unroll
    for (int p = 0; p < P; ++p)
        if (c + 32 * p < chunks) fma_bf16x8(acc[p], zero_mass, __ldcg(reinterpret_cast<const uint4 *>(x + (size_t)t * d) + c + 32 * p));
}

// A warp per CHUNKS * 32 chunks of a token.  Bound by the reads in flight: with every thread holding the
// slot table itself and eight loads predicated by slot, of which the zero slots' were none, 64 threads had a token's chunks
// one after the other.  Combine stage, us, before and now (two chunks per lane, four warps per CTA): 777 tokens of the
// Qwen-shaped layer 10.1 -> 8.3, 2048 tokens 14.3 -> 11.9, 8192 tokens of Zipf load 42.8 -> 37.3, of the static layer
// 60.4 -> 58.3; 5003 tokens of the GLM-shaped layer 24.5 -> 16.6.  (One chunk per lane: 10.0, 14.4, 46, 60.5, 27; four:
// 10.2, 19.3, 52.7, 95, 23.5.)
// Where the warps are few, one chunk per lane and eight slots at a time: twice the warps, half the round trips, and CTAs of
// two warps (40 tokens of the GLM-shaped layer, us a call: 164.1 before, 163.3 so, 1.2 longer in CTAs of four).  A call of
// the Qwen-shaped layer, us, so and with two chunks: 300 tokens 208.4, 209.1; 400 tokens 209.2, 210.3; 500 tokens 210.2,
// 212.1; 600 tokens 212.4, 213.4; 777 tokens 218.3, 218.4; 1000 tokens 225.4, 224.8.  With experts of H_e 128 600 tokens
// 74.5, 75.6; 1000 tokens 78.4, 77.7; at d 1024 (H_e 256) 600 tokens 64.5, 66.0; 1200 tokens 68.1, 69.3.
// At d 4096 (GLM-shaped) 300 tokens 95.7, 95.4; 368 tokens 96.4, 95.5; rows of up to 256 elements are one warp's either way.
constexpr int kFewWarps = 16;  // of two chunks per lane, per SM: the line lies at 592 tokens of d 2048

template <int CHUNKS, int ROWS, int THREADS>
__global__ void __launch_bounds__(THREADS, 896 / THREADS)
combine_kernel(const __nv_bfloat16 *__restrict__ obuf, const int32_t *__restrict__ inv,
               const float *__restrict__ topk_w, const __nv_bfloat16 *__restrict__ x, int T, int K, int d, int pieces,
               int copy_experts, __nv_bfloat16 *__restrict__ y) {
    pdl_launch_dependents();
    pdl_wait();
    const int id = blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int t = id / pieces, c0 = (id - t * pieces) * 32 * CHUNKS;
    if (t >= T) return;
    float acc[CHUNKS][8];
    combine_chunks<CHUNKS, ROWS>(acc, obuf, inv, topk_w, x, t, c0, K, d, copy_experts, lane);
#pragma unroll
    for (int p = 0; p < CHUNKS; ++p) {
        const int c = c0 + 32 * p + lane;
        if (c < d / 8) reinterpret_cast<uint4 *>(y + (size_t)t * d)[c] = pack_bf16x8(acc[p]);
    }
}

// The combine fused with the glue between stacked layers: instead of storing y the CTA forms
// r <- bf16(r + bf16(y)) and h = r / sqrt(mean(r^2) + eps) -- the bits a combine followed by the
// residual + norm kernel produces, without the round trip of y through memory and without the
// second launch.  One CTA per token, one chunk per thread: rows of up to 256 * 8 = 2048 elements.  Bound by
// the reads in flight: each warp loads the slot table once (lane k holds slot k) and only the surviving
// slots are walked, four rows requested at a time, so that the registers leave five CTAs per SM; the
// residual is requested first.  (Before: 64 threads with four chunks one after the other and registers for
// eight rows.  Four stacked layers, 100 tokens: 819 -> 794 us, 700: 918 -> 896, 4096: 1180 -> 1166.)
//
// Same bits: the residual + norm kernel gives chunk c to thread c as well, reduces the squares over the
// 32 lanes of a warp by xor shuffles and adds the warp sums in order.
constexpr int kGlueMaxChunks = 256;
constexpr int kRowsInFlight = 4;

__global__ void __launch_bounds__(kGlueMaxChunks, 5)
combine_glue_kernel(const __nv_bfloat16 *__restrict__ obuf, const int32_t *__restrict__ inv,
                    const float *__restrict__ topk_w, const __nv_bfloat16 *__restrict__ x, int K, int d,
                    int copy_experts, __nv_bfloat16 *__restrict__ resid, __nv_bfloat16 *__restrict__ h_next, float eps) {
    pdl_launch_dependents();
    pdl_wait();
    const int t = blockIdx.x, c = threadIdx.x, lane = threadIdx.x & 31;
    const bool in = c < d / 8;
    uint4 *rp = reinterpret_cast<uint4 *>(resid + (size_t)t * d) + c;
    const uint4 rv = in ? __ldcg(rp) : make_uint4(0u, 0u, 0u, 0u);
    const int my_pos = lane < K ? __ldcg(inv + (size_t)t * K + lane) : -1;
    const float my_w = lane < K ? __ldcg(topk_w + (size_t)t * K + lane) : 0.f;
    const unsigned real = __ballot_sync(0xffffffffu, my_pos >= 0);
    float acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
    for (unsigned left = real; left;) {  // slots in order; (uniform over the warp)
        uint4 v[kRowsInFlight];
        float w[kRowsInFlight];
        const int n = __popc(left);
#pragma unroll
        for (int r = 0; r < kRowsInFlight; ++r) {
            const int k = r < n ? __ffs(left) - 1 : 0;
            left &= left - 1u;
            w[r] = __shfl_sync(0xffffffffu, my_w, k);
            const int pos = __shfl_sync(0xffffffffu, my_pos, k);
            if (r < n && in) v[r] = __ldcg(reinterpret_cast<const uint4 *>(obuf + (size_t)pos * d) + c);
        }
#pragma unroll
        for (int r = 0; r < kRowsInFlight; ++r)
            if (r < n && in) fma_bf16x8(acc, w[r], v[r]);
    }
    if (copy_experts) {
        float zero_mass = 0.f;  // the summed weight of the zero slots
        for (int k = 0; k < K; ++k) {
            const float w = __shfl_sync(0xffffffffu, my_w, k);
            if (!(real >> k & 1u)) zero_mass += w;
        }
        if (zero_mass != 0.f && in) fma_bf16x8(acc, zero_mass, __ldcg(reinterpret_cast<const uint4 *>(x + (size_t)t * d) + c));
    }
    const uint32_t ru[4] = {rv.x, rv.y, rv.z, rv.w};
    uint32_t keep[4];  // the updated residual (bf16 pairs)
    float ss = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t yb = pack_bf16(acc[2 * j], acc[2 * j + 1]);  // y as it would be stored
        keep[j] = pack_bf16(__uint_as_float(ru[j] << 16) + __uint_as_float(yb << 16),
                            __uint_as_float(ru[j] & 0xffff0000u) + __uint_as_float(yb & 0xffff0000u));
        const float r0 = __uint_as_float(keep[j] << 16), r1 = __uint_as_float(keep[j] & 0xffff0000u);  // the stored residual
        ss = fmaf(r0, r0, ss);
        ss = fmaf(r1, r1, ss);
    }
    if (in) *rp = make_uint4(keep[0], keep[1], keep[2], keep[3]);
    else ss = 0.f;
    __shared__ float warp_ss[kGlueMaxChunks / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) warp_ss[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) tot += warp_ss[w];
    const float scale = rsqrtf(tot / (float)d + eps);
    if (in) {
        uint32_t o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            o[j] = pack_bf16(__uint_as_float(keep[j] << 16) * scale, __uint_as_float(keep[j] & 0xffff0000u) * scale);
        reinterpret_cast<uint4 *>(h_next + (size_t)t * d)[c] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

}  // namespace

int launch_combine(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y, cudaStream_t s) {
    return launch_combine_rows(h, h->ws.obuf, x, T, y, s);
}

// rows: the expert outputs of the call's surviving pairs in (expert, token) order
int launch_combine_rows(const zeda_moe *h, const __nv_bfloat16 *rows, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y,
                        cudaStream_t s) {
    const zeda_moe_config_t &c = h->cfg;
    auto go = [&](auto kernel, int per_warp, int threads) {
        const int pieces = (c.d_model / 8 + per_warp - 1) / per_warp, per_cta = threads / 32;
        return launch_kernel(h->pdl, kernel, dim3(((long long)T * pieces + per_cta - 1) / per_cta), dim3(threads), 0, s, rows,
                             (const int32_t *)h->ws.inv, (const float *)h->ws.topk_w, x, T, c.top_k, c.d_model, pieces,
                             (int)(c.expert_kind == ZEDA_EXPERT_COPY), y);
    };
    const bool few = (long long)T * ((c.d_model / 8 + 63) / 64) < (long long)kFewWarps * h->sm_count;
    const cudaError_t e = few ? go(combine_kernel<1, 8, 64>, 32, 64) : go(combine_kernel<2, 4, 128>, 64, 128);
    return e == cudaSuccess ? 1 : -1;
}

bool combine_glue_supported(const zeda_moe *h) { return h->cfg.d_model <= kGlueMaxChunks * 8; }

// resid <- bf16(resid + y), h_next = RMSNorm(resid) with y never stored; h_next must not overlap x
// (the copy-expert variant reads x[t] while other CTAs already write their h_next rows).
int launch_combine_glue(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *resid, __nv_bfloat16 *h_next, float eps,
                        cudaStream_t s) {
    const zeda_moe_config_t &c = h->cfg;
    const cudaError_t e = launch_kernel(h->pdl, combine_glue_kernel, dim3(T), dim3((c.d_model / 8 + 31) / 32 * 32), 0, s,
                                        (const __nv_bfloat16 *)h->ws.obuf, (const int32_t *)h->ws.inv, (const float *)h->ws.topk_w,
                                        x, c.top_k, c.d_model, (int)(c.expert_kind == ZEDA_EXPERT_COPY), resid, h_next, eps);
    return e == cudaSuccess ? 1 : -1;
}

}  // namespace zeda
