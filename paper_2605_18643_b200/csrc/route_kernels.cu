// Routing stage: router logits over the N + N_Z candidates, softmax / top-K / routing weights
// (Section 2.1), then the compaction that drops zero-expert slots and counting-sorts the surviving
// (token, normal expert) pairs by expert in a stable order.
#include <cooperative_groups.h>

#include <atomic>

#include "expert_scan.cuh"
#include "route_token.cuh"

namespace zeda {

namespace {

// ---------------------------------------------------------------------------------------------
// Router logits on the CUDA cores, up to 255 tokens: l[t, j] = <x_t, W_r[j]> + b[j] in fp32.
// ---------------------------------------------------------------------------------------------
// Few tokens: one candidate row per CTA, so that the rows (1.5 MB for 192 candidates of 2048) are read by
// 192 SM-wide bursts instead of 24; the reduction axis is split over four warps.  NT tokens per CTA, all
// of their loads in flight at once.  The row is asked into L2 before the wait for the kernel in front (a
// prefetch only: its values are read after the wait).
// From kTileRouterTokens on the tensor-core routers.  Their accumulators are fp32 too, but against 64 bits its logits
// are off by 2.1e-6 of their root mean square at d 2048 (1.0e-6 at 1024, 9e-6 at 8192), these kernels' by 1.1e-7:
// below, the CUDA cores keep them.
constexpr int kFewTokens = 32;  // calls of at most this many tokens
constexpr int kFewThreads = 128;
constexpr int kFewUnroll = 4;

template <int NT>
__global__ void __launch_bounds__(kFewThreads)
router_logits_few_kernel(const __nv_bfloat16 *__restrict__ x, const float *__restrict__ router_w,
                         const float *__restrict__ router_bias, int T, int d, int n_cand, float *__restrict__ logits,
                         int32_t *__restrict__ hist, int n_hist, int32_t *__restrict__ meta) {
    pdl_launch_dependents();
    const int j = blockIdx.x, t0 = blockIdx.y * NT;
    const float *wrow = router_w + (size_t)j * d;
    for (int i = threadIdx.x; i < d / 32; i += kFewThreads) asm volatile("prefetch.global.L2 [%0];" ::"l"(wrow + 32 * i));
    pdl_wait();
    clear_hist(hist, n_hist);
    if (j == 0 && t0 == 0 && threadIdx.x == 0) meta[kMetaRouted] = 0;
    float acc[NT];
#pragma unroll
    for (int r = 0; r < NT; ++r) acc[r] = 0.f;
    for (int c0 = threadIdx.x; c0 < d / 4; c0 += kFewThreads * kFewUnroll) {
        float4 w[kFewUnroll];
        uint2 xv[NT][kFewUnroll];
#pragma unroll
        for (int u = 0; u < kFewUnroll; ++u) {
            const int c = c0 + kFewThreads * u;
            const bool in = c < d / 4;
            w[u] = in ? __ldg(reinterpret_cast<const float4 *>(wrow) + c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int r = 0; r < NT; ++r)
                xv[r][u] = in && t0 + r < T ? __ldcg(reinterpret_cast<const uint2 *>(x + (size_t)(t0 + r) * d) + c) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int r = 0; r < NT; ++r) {
#pragma unroll
            for (int u = 0; u < kFewUnroll; ++u) {
                acc[r] = fmaf(w[u].x, __uint_as_float(xv[r][u].x << 16), acc[r]);
                acc[r] = fmaf(w[u].y, __uint_as_float(xv[r][u].x & 0xffff0000u), acc[r]);
                acc[r] = fmaf(w[u].z, __uint_as_float(xv[r][u].y << 16), acc[r]);
                acc[r] = fmaf(w[u].w, __uint_as_float(xv[r][u].y & 0xffff0000u), acc[r]);
            }
        }
    }
    __shared__ float red[kFewThreads / 32][NT];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < NT; ++r) {
        const float s = warp_sum(acc[r]);
        if (lane == 0) red[warp][r] = s;
    }
    __syncthreads();
    if (threadIdx.x < NT && t0 + (int)threadIdx.x < T) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < kFewThreads / 32; ++q) s += red[q][threadIdx.x];
        logits[(size_t)(t0 + threadIdx.x) * n_cand + j] = s + (router_bias ? __ldg(router_bias + j) : 0.f);
    }
}

// Router of 33 to 255 tokens: 4 TL x kTileCand logits per cluster of CTAS CTAs, TL x 4 logits per lane.
// The sum of a logit is the same additions in every form, so that a token's logits do not depend on its batch: 32 chains
// (chain c: elements 4 c to 4 c + 3 of every 128), each in runs of kRunSteps x 4 products that are added up one behind the
// other, then the chains pairwise, neighbours first, then the bias.  A warp takes a chain, a CTA kWarps of them; it sends
// the sum of its chains, through distributed shared memory, to the CTA of the cluster that finishes the token.
// What bounds it is shared memory and the fused multiply-adds alike (TL + 4 loads per 16 TL of them), on an SM's 8 or 4
// warps, behind one wait for memory: a CTA asks for the first two stages of its operands at once, its router rows (the
// caller's constants) in front of the wait for the kernel before.  The loop is short because a call meets its instructions
// cold (unrolled by four, 64 tokens 0.9 us longer).
//
// Which form takes a call: that of the least work per SM.  CTAs have an SM each (where two of a cluster share one while
// others have none, a call of 160 tokens takes 4 us longer), so the clusters that run at a time are few (33 of four CTAs, 15
// of eight), and a second wave of them costs as much as the first: tiles are as tall as one wave needs, eight CTAs where
// those fit.  A wave takes TL times 2 (eight CTAs) or 3 (four: twice the chains per SM, on twice the warps).  A layer with
// small experts (weights beyond L2), us, by the forms <8,8>, <8,10>, <4,8>, <4,10>, <4,12>, <4,14>, <4,16>, and by one that
// had a warp per candidate row and 8 tokens:
//   d 2048, 192 candidates   T=33   55.3  56.0  56.8  57.7  60.1  61.1  61.1,  59.1
//                            T=80   70.8  66.1  67.3  68.1  69.8  70.7  71.9,  67.4
//                            T=160  73.2  74.2  69.8  71.1  72.8  73.7  74.5,  76.5
//                            T=193  79.1  74.4  77.6  70.8  72.7  74.1  74.9,  76.6
//                            T=240  84.9  80.5  77.4  79.5  72.8  74.2  75.0,  84.1
//                            T=255  84.9  80.8  77.5  79.3  82.6  74.4  74.7,  84.1
//   d 2048, 512              T=64  111.8 113.7 102.4 103.4 105.2 106.2 107.1, 107.9
//                            T=255 187.7 187.4 169.0 171.7 170.3 171.5 163.1, 178.3
//   d 8192, 300              T=33  190.8 177.7 183.6 186.6 192.9 196.4 199.5, 187.8
//   d 512, 64                T=33   41.9  42.6  42.2  42.9  43.5  43.8  44.2,  43.0
// (Eight CTAs and taller tiles never cost less than four and 32 tokens.)
constexpr int kChains = 32, kRunSteps = 4;

// Two fp32 numbers side by side, and the same operation on both at once: each as by itself, bit for bit.
using F32x2 = unsigned long long;
__device__ __forceinline__ F32x2 f32x2(uint32_t lo, uint32_t hi) { return (F32x2)hi << 32 | lo; }
__device__ __forceinline__ void fma_f32x2(F32x2 &acc, float a, F32x2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(f32x2(__float_as_uint(a), __float_as_uint(a))), "l"(b));
}
__device__ __forceinline__ void add_f32x2(F32x2 &acc, F32x2 a) { asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(a)); }

template <int CTAS, int TL>
struct RouterCluster {
    static constexpr int kCtas = CTAS, kTileTokens = 4 * TL, kTileCand = 32;
    static constexpr int kWarps = kChains / CTAS, kThreads = 32 * kWarps;
    static constexpr int kSteps = 8, kStage = 128 * kSteps;  // of a chain per stage; elements of a row
    // bytes between rows: odd multiples of 16, so that rows next to one another lie in different banks
    static constexpr int kXLd = 8 * kWarps * kSteps + 16, kWLd = 16 * kWarps * kSteps + 16;
    static constexpr int kBuffer = kTileTokens * kXLd + kTileCand * kWLd;
    static constexpr int kRedLd = 40;                // floats between the tokens of a chain's sums: the lanes of a store hit all banks
    static constexpr int kOwn = kTileTokens / CTAS;  // tokens that a CTA finishes
    static constexpr int kUsed = 2 * kBuffer + kTileTokens * kTileCand * (int)sizeof(float);
    // more than half of an SM's shared memory: CTAs of a cluster that share an SM, while others have none, take twice as long
    static constexpr int kSmem = kUsed > 120 * 1024 ? kUsed : 120 * 1024;
    static_assert(kSteps % kRunSteps == 0, "no run of products crosses a stage");
    static_assert(kWarps * kTileTokens * kRedLd * 4 <= 2 * kBuffer, "the sums take the operands' room");
};

template <int CTAS, int TL>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(RouterCluster<CTAS, TL>::kThreads, 1)
router_logits_cluster_kernel(const __nv_bfloat16 *__restrict__ x, const float *__restrict__ router_w, const float *__restrict__ router_bias,
                             int T, int d, int n_cand, float *__restrict__ logits, int32_t *__restrict__ hist, int n_hist) {
    using C = RouterCluster<CTAS, TL>;
    pdl_launch_dependents();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    extern __shared__ __align__(16) unsigned char smem_raw[];  // two stages of tokens and router rows, then the sums received
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = blockIdx.x % CTAS;
    const int j0 = blockIdx.x / CTAS * C::kTileCand, t0 = blockIdx.y * C::kTileTokens;
    const int rows_w = min(C::kTileCand, n_cand - j0), rows_x = min(C::kTileTokens, T - t0);
    const int n_stages = (d + C::kStage - 1) / C::kStage;
    auto copy16 = [](void *dst, const void *src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    // Of every 128 elements of a row the CTA takes its chains' 4 x kWarps.  (Rows beyond the call's and elements beyond the
    // row are not copied: the former's sums are not stored, the latter are not multiplied.)
    auto copy_w = [&](int stage) {
        unsigned char *dst = smem_raw + (stage & 1) * C::kBuffer + C::kTileTokens * C::kXLd;
        constexpr int kPieces = C::kSteps * C::kWarps;  // of 16 bytes, of a row
        const int piece = threadIdx.x % kPieces;
        const int col = stage * C::kStage + 128 * (piece / C::kWarps) + 4 * (rank * C::kWarps + piece % C::kWarps);
        if (col < d)
#pragma unroll
            for (int r = threadIdx.x / kPieces; r < C::kTileCand; r += C::kThreads / kPieces)
                if (r < rows_w) copy16(dst + r * C::kWLd + 16 * piece, router_w + (size_t)(j0 + r) * d + col);
    };
    auto copy_x = [&](int stage) {  // (two chains to a piece: d is a multiple of 64, so both are in the row or neither)
        unsigned char *dst = smem_raw + (stage & 1) * C::kBuffer;
        constexpr int kPairs = C::kWarps / 2, kPieces = C::kSteps * kPairs;
        const int piece = threadIdx.x % kPieces;
        const int col = stage * C::kStage + 128 * (piece / kPairs) + 4 * rank * C::kWarps + 8 * (piece % kPairs);
        if (col < d)
#pragma unroll
            for (int r = threadIdx.x / kPieces; r < C::kTileTokens; r += C::kThreads / kPieces)
                if (r < rows_x) copy16(dst + r * C::kXLd + 16 * piece, x + (size_t)(t0 + r) * d + col);
    };
    copy_w(0);
    if (n_stages > 1) copy_w(1);
    commit();
    pdl_wait();
    clear_hist(hist, n_hist);
    copy_x(0);
    commit();
    if (n_stages > 1) copy_x(1);
    commit();
    // lane: tokens tg + 4 i, candidates cg + 8 j
    const int tg = lane >> 3, cg = lane & 7;
    F32x2 acc[TL / 2][4], tot[TL / 2][4];  // of tokens tg + 4 i and tg + 4 (i + TL / 2)
#pragma unroll
    for (int i = 0; i < TL / 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = tot[i][j] = 0;
    for (int stage = 0; stage < n_stages; ++stage) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");  // all but the next stage's
        __syncthreads();
        const unsigned char *xb = smem_raw + (stage & 1) * C::kBuffer + 8 * warp;
        const unsigned char *wb = smem_raw + (stage & 1) * C::kBuffer + C::kTileTokens * C::kXLd + 16 * warp;
        const int left = d - stage * C::kStage - 4 * (rank * C::kWarps + warp);  // of the row, from the chain's next element on
        const int steps = min(C::kSteps, (left + 127) / 128);
#pragma unroll 1  // (a short loop: a call meets its instructions cold)
        for (int u = 0; u < steps; ++u) {
            uint2 xv[TL];
            float4 w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4 *>(wb + (cg + 8 * j) * C::kWLd + 16 * C::kWarps * u);
#pragma unroll
            for (int i = 0; i < TL; ++i) xv[i] = *reinterpret_cast<const uint2 *>(xb + (tg + 4 * i) * C::kXLd + 8 * C::kWarps * u);
#pragma unroll
            for (int i = 0; i < TL / 2; ++i) {
                const uint2 a = xv[i], b = xv[i + TL / 2];
                const F32x2 x0 = f32x2(a.x << 16, b.x << 16), x1 = f32x2(a.x & 0xffff0000u, b.x & 0xffff0000u);
                const F32x2 x2 = f32x2(a.y << 16, b.y << 16), x3 = f32x2(a.y & 0xffff0000u, b.y & 0xffff0000u);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    fma_f32x2(acc[i][j], w[j].x, x0);
                    fma_f32x2(acc[i][j], w[j].y, x1);
                    fma_f32x2(acc[i][j], w[j].z, x2);
                    fma_f32x2(acc[i][j], w[j].w, x3);
                }
            }
            if ((u + 1) % kRunSteps == 0 || u + 1 == steps) {  // (uniform over the warp)
#pragma unroll
                for (int i = 0; i < TL / 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) { add_f32x2(tot[i][j], acc[i][j]); acc[i][j] = 0; }
            }
        }
        __syncthreads();  // the stage has been read: its room takes another, or the sums
        if (stage + 2 < n_stages) {
            copy_w(stage + 2);
            copy_x(stage + 2);
        }
        commit();
    }
    float *red = reinterpret_cast<float *>(smem_raw);  // [kWarps][kTileTokens][kRedLd]
#pragma unroll
    for (int i = 0; i < TL; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            red[(warp * C::kTileTokens + tg + 4 * i) * C::kRedLd + cg + 8 * j] = __uint_as_float((uint32_t)(tot[i % (TL / 2)][j] >> (i < TL / 2 ? 0 : 32)));
    __syncthreads();
    auto cluster = cooperative_groups::this_cluster();
    float *got = reinterpret_cast<float *>(smem_raw + 2 * C::kBuffer);  // [CTAS][kOwn][kTileCand]
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // (every CTA of the cluster has started)
    for (int i = threadIdx.x; i < C::kTileTokens * C::kTileCand / 4; i += C::kThreads) {  // four candidates of a token
        const int t = i / (C::kTileCand / 4), c = i % (C::kTileCand / 4) * 4;
        float4 v[C::kWarps];
#pragma unroll
        for (int q = 0; q < C::kWarps; ++q) v[q] = *reinterpret_cast<const float4 *>(red + (q * C::kTileTokens + t) * C::kRedLd + c);
#pragma unroll
        for (int o = 1; o < C::kWarps; o *= 2)
#pragma unroll
            for (int q = 0; q < C::kWarps; q += 2 * o) v[q] = make_float4(v[q].x + v[q + o].x, v[q].y + v[q + o].y, v[q].z + v[q + o].z, v[q].w + v[q + o].w);
        *reinterpret_cast<float4 *>(cluster.map_shared_rank(got, t / C::kOwn) + (rank * C::kOwn + t % C::kOwn) * C::kTileCand + c) = v[0];
    }
    cluster.sync();
    for (int own = warp; own < C::kOwn; own += C::kWarps) {  // a token per warp, a candidate per lane
        const int r = rank * C::kOwn + own;
        float v[CTAS];
#pragma unroll
        for (int q = 0; q < CTAS; ++q) v[q] = got[(q * C::kOwn + own) * C::kTileCand + lane];
#pragma unroll
        for (int o = 1; o < CTAS; o *= 2)
#pragma unroll
            for (int q = 0; q < CTAS; q += 2 * o) v[q] += v[q + o];
        if (r < rows_x && lane < rows_w) logits[(size_t)(t0 + r) * n_cand + j0 + lane] = v[0] + (router_bias ? __ldg(router_bias + j0 + lane) : 0.f);
    }
}

// The forms; of equal cost the later one takes a call.
template <typename F>
void each_router_form(F f) {
    f(RouterCluster<8, 8>(), router_logits_cluster_kernel<8, 8>);
    f(RouterCluster<8, 10>(), router_logits_cluster_kernel<8, 10>);
    f(RouterCluster<4, 8>(), router_logits_cluster_kernel<4, 8>);
    f(RouterCluster<4, 10>(), router_logits_cluster_kernel<4, 10>);
    f(RouterCluster<4, 12>(), router_logits_cluster_kernel<4, 12>);
    f(RouterCluster<4, 14>(), router_logits_cluster_kernel<4, 14>);
    f(RouterCluster<4, 16>(), router_logits_cluster_kernel<4, 16>);
}

// block_hist (optional): pass 1 of the counting sort done here.  Every slot on a normal expert adds 1
// to its entry of the histogram of its block of kSortTokens tokens (integer adds: the counts do not
// depend on their order).  The histograms must be zero on entry: the call's router kernel clears them.
template <int RPL>
__global__ void __launch_bounds__(256)
topk_gate_kernel(const float *__restrict__ logits, int n_parts, int T, int n_real, int n_cand, int K, int gate_mode,
                 int32_t *__restrict__ topk_idx, float *__restrict__ topk_w, int32_t *__restrict__ block_hist) {
    pdl_launch_dependents();
    pdl_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + warp;
    if (t >= T) return;
    int my_idx;
    float my_w, v[RPL], m, den;
    topk_gate_token<RPL>(logits + (size_t)t * n_cand, n_parts, (size_t)T * n_cand, n_real, n_cand, K, gate_mode, lane,
                         v, m, den, my_idx, my_w);
    if (lane < K) {
        topk_idx[(size_t)t * K + lane] = my_idx;
        topk_w[(size_t)t * K + lane] = my_w;
        if (block_hist && (unsigned)my_idx < (unsigned)n_real)
            atomicAdd(block_hist + (size_t)(t / kSortTokens) * n_real + my_idx, 1);
    }
}

// ---------------------------------------------------------------------------------------------
// Counting sort, pass 1 as a kernel of its own (the paths that do not take it in the top-K kernel):
// per-CTA histogram of the normal-expert slots of kSortTokens tokens.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
slot_hist_kernel(const int32_t *__restrict__ topk_idx, int T, int K, int n_real,
                 int32_t *__restrict__ block_hist) {
    pdl_launch_dependents();
    pdl_wait();
    extern __shared__ int32_t hist[];  // [n_real]
    for (int e = threadIdx.x; e < n_real; e += blockDim.x) hist[e] = 0;
    __syncthreads();
    const int s0 = blockIdx.x * kSortTokens * K;
    const int s1 = min(T * K, s0 + kSortTokens * K);
    for (int s = s0 + threadIdx.x; s < s1; s += blockDim.x) {
        const int e = __ldcg(topk_idx + s);
        if ((unsigned)e < (unsigned)n_real) atomicAdd(&hist[e], 1);  // zero experts and ids < 0 are dropped
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n_real; e += blockDim.x) block_hist[(size_t)blockIdx.x * n_real + e] = hist[e];
}

// ---------------------------------------------------------------------------------------------
// Counting sort, pass 2 (one CTA): column-wise exclusive scan over the CTA histograms, expert
// counts, exclusive offsets, P, U, and the work lists of the expert kernels.
// ---------------------------------------------------------------------------------------------
constexpr int kScanSlabInts = 8192;  // 32 KB of CTA histograms per slab of the expert scan

__global__ void __launch_bounds__(512)
expert_scan_kernel(int32_t *__restrict__ block_hist, int nblk, int n_real, int total_slots,
                   int32_t *__restrict__ counts, int32_t *__restrict__ offsets,
                   int32_t *__restrict__ n_pairs_out, int32_t *__restrict__ meta, const WorkLists wl, int tile_rows) {
    __shared__ ScanShared sh;
    // Exclusive scan of every expert column over the CTA histograms.  The histograms are staged in
    // shared memory slab by slab with independent coalesced loads (a load-scan-store loop straight
    // on global memory is a chain of dependent L2 round trips), scanned by one thread per expert,
    // and written back coalesced.
    __shared__ int32_t slab[kScanSlabInts];
    const int slab_blocks = max(1, kScanSlabInts / n_real);
    const int e = threadIdx.x;
    int run = 0;
    for (int b0 = 0; b0 < nblk; b0 += slab_blocks) {
        const int nb = min(slab_blocks, nblk - b0);
        int32_t *g = block_hist + (size_t)b0 * n_real;
        for (int i = threadIdx.x; i < nb * n_real; i += blockDim.x) slab[i] = g[i];
        __syncthreads();
        if (e < n_real) {
            for (int b = 0; b < nb; ++b) {
                const int c = slab[b * n_real + e];
                slab[b * n_real + e] = run;  // pairs of expert e in earlier CTAs
                run += c;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nb * n_real; i += blockDim.x) g[i] = slab[i];
        __syncthreads();
    }
    if (e < n_real) sh.cnt[e] = run;
    __syncthreads();
    finish_expert_scan(sh, n_real, total_slots, counts, offsets, n_pairs_out, meta, wl, true, 0, 1, tile_rows);
}

// ---------------------------------------------------------------------------------------------
// Small batches (T <= 128, decode): top-K, routing weights and the whole counting sort in ONE
// launch of a thread-block cluster.  Each CTA of the cluster takes 16 tokens (one warp per token)
// and records "token t selected expert e" as bit t of a T-bit mask that lives in CTA 0's shared
// memory (distributed shared memory, atomicOr).  A token selects an expert at most once, so an
// expert's count is a popcount and the stable rank of a pair is the popcount of the lower token
// bits: the (expert, token) order needs no atomics on positions and no second pass.  After the
// cluster barrier CTA 0 scans the experts and places the pairs.
// ---------------------------------------------------------------------------------------------
constexpr int kSmallTokens = 128;
constexpr int kSmallCluster = 8;
constexpr int kSmallThreads = 32 * (kSmallTokens / kSmallCluster);  // one warp per token

// CLUSTER = 1: up to 16 tokens fit one CTA, which saves the cluster's launch and barriers.
template <int RPL, int CLUSTER>
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(kSmallThreads)
route_small_kernel(const float *__restrict__ logits, int n_parts, int T, int n_real, int n_cand, int K, int gate_mode,
                   int32_t *__restrict__ topk_idx, float *__restrict__ topk_w, int32_t *__restrict__ counts,
                   int32_t *__restrict__ offsets, int32_t *__restrict__ n_pairs_out, int32_t *__restrict__ meta,
                   const WorkLists wl, int tile_rows, int32_t *__restrict__ perm,
                   int32_t *__restrict__ perm_user, int32_t *__restrict__ inv, int32_t *__restrict__ pair_token) {
    pdl_launch_dependents();
    pdl_wait();
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ ScanShared sh;
    __shared__ uint32_t sel[kMaxCand][kSmallTokens / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned rank = CLUSTER > 1 ? cluster.block_rank() : 0u;
    if (rank == 0)
        for (int i = threadIdx.x; i < n_real * (kSmallTokens / 32); i += blockDim.x) (&sel[0][0])[i] = 0u;
    if (CLUSTER > 1) cluster.sync(); else __syncthreads();
    uint32_t *sel0 = CLUSTER > 1 ? cluster.map_shared_rank(&sel[0][0], 0) : &sel[0][0];
    const int t = rank * (kSmallThreads / 32) + warp;
    if (t < T) {
        int my_idx;
        float my_w, v[RPL], m, den;
        topk_gate_token<RPL>(logits + (size_t)t * n_cand, n_parts, (size_t)T * n_cand, n_real, n_cand, K, gate_mode, lane, v, m, den, my_idx, my_w);
        if (lane < K) {
            topk_idx[(size_t)t * K + lane] = my_idx;
            topk_w[(size_t)t * K + lane] = my_w;
            if (my_idx < n_real) atomicOr(sel0 + my_idx * (kSmallTokens / 32) + (t >> 5), 1u << (t & 31));
        }
    }
    // release/acquire at cluster (CTA) scope: masks and topk_idx of every CTA are visible
    if (CLUSTER > 1) cluster.sync(); else __syncthreads();
    if (rank != 0) return;
    if ((int)threadIdx.x < n_real) {
        int c = 0;
#pragma unroll
        for (int i = 0; i < kSmallTokens / 32; ++i) c += __popc(sel[threadIdx.x][i]);
        sh.cnt[threadIdx.x] = c;
    }
    __syncthreads();
    finish_expert_scan(sh, n_real, T * K, counts, offsets, n_pairs_out, meta, wl, true, 0, 1, tile_rows);
    for (int s = threadIdx.x; s < T * K; s += blockDim.x) {
        const int e = topk_idx[s], tk = s / K;
        int p = -1;
        if (e < n_real) {
            int r = __popc(sel[e][tk >> 5] & ((1u << (tk & 31)) - 1u));
            for (int i = 0; i < (tk >> 5); ++i) r += __popc(sel[e][i]);
            p = sh.off[e] + r;
            perm[p] = s;
            if (perm_user) perm_user[p] = s;
            pair_token[p] = tk;
        }
        inv[s] = p;
    }
}

// ---------------------------------------------------------------------------------------------
// Counting sort, pass 3: stable placement.  Each CTA re-walks its kSortTokens*K slots in slot
// order; each warp owns a contiguous run of slots, ranks equal experts inside a 32-slot step with
// match.any / popc (a warp-level prefix count) and carries per-expert running positions in shared
// memory.  No atomics decide a position, so the order is (expert, token) ascending every run.
// ---------------------------------------------------------------------------------------------
constexpr int kPlaceWarps = 8;

__global__ void __launch_bounds__(kPlaceWarps * 32)
slot_place_kernel(const int32_t *__restrict__ topk_idx, int T, int K, int n_real,
                  const int32_t *__restrict__ block_base, const int32_t *__restrict__ offsets,
                  int32_t *__restrict__ perm, int32_t *__restrict__ perm_user,
                  int32_t *__restrict__ inv, int32_t *__restrict__ pair_token) {
    extern __shared__ int32_t pos[];  // [kPlaceWarps][n_real]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < kPlaceWarps * n_real; i += blockDim.x) pos[i] = 0;
    __syncthreads();
    const int s0 = blockIdx.x * kSortTokens * K;
    const int s1 = min(T * K, s0 + kSortTokens * K);
    const int per_warp = ((kSortTokens * K + kPlaceWarps - 1) / kPlaceWarps + 31) / 32 * 32;
    const int w0 = s0 + warp * per_warp;
    const int w1 = min(s1, w0 + per_warp);
    int32_t *mine = pos + warp * n_real;
    const unsigned lt = (1u << lane) - 1u;
    // count this warp's slots per expert
    for (int s = w0 + lane; s - lane < w1; s += 32) {
        int e = (s < w1) ? topk_idx[s] : -1;
        if ((unsigned)e >= (unsigned)n_real) e = -1;  // zero experts; ids < 0 are dropped the same way
        const unsigned grp = __match_any_sync(kFull, e);
        if (e >= 0 && (grp & lt) == 0) mine[e] += __popc(grp);
        __syncwarp();
    }
    __syncthreads();
    // turn counts into start positions: global offset + earlier CTAs + earlier warps
    for (int e = threadIdx.x; e < n_real; e += blockDim.x) {
        int run = offsets[e] + block_base[(size_t)blockIdx.x * n_real + e];
        for (int w = 0; w < kPlaceWarps; ++w) {
            const int c = pos[w * n_real + e];
            pos[w * n_real + e] = run;
            run += c;
        }
    }
    __syncthreads();
    for (int s = w0 + lane; s - lane < w1; s += 32) {
        int e = (s < w1) ? topk_idx[s] : -1;
        const bool in_range = s < w1;
        if ((unsigned)e >= (unsigned)n_real) e = -1;  // zero experts; ids < 0 are dropped the same way
        const unsigned grp = __match_any_sync(kFull, e);
        int p = -1;
        if (e >= 0) p = mine[e] + __popc(grp & lt);
        __syncwarp();
        if (e >= 0 && (grp & lt) == 0) mine[e] += __popc(grp);
        __syncwarp();
        if (in_range) {
            inv[s] = p;
            if (p >= 0) {
                perm[p] = s;
                if (perm_user) perm_user[p] = s;
                pair_token[p] = s / K;
            }
        }
    }
}

// Routing statistics, final sums by one CTA: adds up what the CTAs of the top-K pass have left in `part` (per CTA n_cand
// selection counts, then n_cand sums of probabilities) in a fixed order.  A group of neighbouring columns (four where the
// rows allow 16-byte loads) is shared by as many threads as fit, each adding every n-th row, 32 requested at a time (8 in the
// kernel of its own) and added up pairwise (8192 tokens of 192 candidates: 45.3 us a call with the sums behind the placement, 43.5 beside it with
// sixteen rows at a time, 36.8 with 32), then the threads of a group pairwise (one after the other, 8192 tokens of 12
// candidates took 15.0 us, so 13.7).
struct StatsJob {
    const float *part;
    int rows;  // of part
    float *f, *p_mean, *out;
};

__device__ __forceinline__ float4 add_columns(const float4 &a, const float4 &b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float2 add_columns(const float2 &a, const float2 &b) { return make_float2(a.x + b.x, a.y + b.y); }

constexpr int kStatFinalThreads = 256, kStatFinalDeep = 32;        // beside the placement
constexpr int kStatManyRowsThreads = 1024, kStatManyRowsDeep = 8;  // as a kernel of its own, for more rows

template <int THREADS>
struct StatsShared {
    float col[2 * kMaxCand];
    float4 share[THREADS];
    float red[5][THREADS / 32];
};

template <typename V, int THREADS, int kDeep>
__device__ __forceinline__ void sum_stat_columns(const StatsJob &job, int cols, float *col, float4 *share) {
    const int groups = cols / (int)(sizeof(V) / sizeof(float)), segs = max(1, THREADS / groups), seg = threadIdx.x / groups;
    for (int c0 = 0; c0 < groups; c0 += THREADS) {  // (more than one turn only where each group has one thread)
        const int c = segs > 1 ? threadIdx.x - seg * groups : c0 + threadIdx.x;
        const bool on = segs > 1 ? seg < segs : c < groups;
        V a = {};
        if (on)
            for (int b0 = segs > 1 ? seg : 0; b0 < job.rows; b0 += kDeep * segs) {
                V v[kDeep];
#pragma unroll
                for (int q = 0; q < kDeep; ++q)
                    v[q] = b0 + q * segs < job.rows ? __ldcg(reinterpret_cast<const V *>(job.part + (size_t)(b0 + q * segs) * cols) + c) : V{};
#pragma unroll
                for (int o = kDeep / 2; o > 0; o >>= 1)
#pragma unroll
                    for (int q = 0; q < o; ++q) v[q] = add_columns(v[q], v[q + o]);
                a = add_columns(a, v[0]);
            }
        // the shares of a group, those of the upper half of its threads onto the lower half's
        V *mine = reinterpret_cast<V *>(share) + threadIdx.x;
        for (int n = segs; n > 1;) {
            const int half = (n + 1) / 2;
            if (on && seg >= half && seg < n) *mine = a;
            __syncthreads();
            if (on && seg + half < n) a = add_columns(a, mine[half * groups]);
            n = half;
        }
        if (on && (segs == 1 || seg == 0)) reinterpret_cast<V *>(col)[c] = a;
        __syncthreads();
    }
}

template <int THREADS, int DEEP>
__device__ __forceinline__ void stats_final(const StatsJob &job, int T, int K, int n_real, int n_cand, StatsShared<THREADS> &sh) {
    if (n_cand % 2 == 0) sum_stat_columns<float4, THREADS, DEEP>(job, 2 * n_cand, sh.col, sh.share);
    else sum_stat_columns<float2, THREADS, DEEP>(job, 2 * n_cand, sh.col, sh.share);
    float sums[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    for (int j = threadIdx.x; j < n_cand; j += THREADS) {
        const float fj = sh.col[j] / T, pj = sh.col[n_cand + j] / T;
        if (job.f) job.f[j] = fj;
        if (job.p_mean) job.p_mean[j] = pj;
        const bool real = j < n_real;
        const float add[5] = {fj * pj, real ? fj : 0.f, real ? pj : 0.f, real ? 0.f : fj, real ? 0.f : pj};
#pragma unroll
        for (int i = 0; i < 5; ++i) sums[i] += add[i];
    }
    if (!job.out) return;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float s = warp_sum(sums[i]);
        if ((threadIdx.x & 31) == 0) sh.red[i][threadIdx.x >> 5] = s;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        float tot[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) tot[i] = warp_sum(threadIdx.x < THREADS / 32 ? sh.red[i][threadIdx.x] : 0.f);
        if (threadIdx.x == 0) {
            job.out[0] = tot[3] / K;
            job.out[1] = tot[0];
            job.out[2] = tot[1] * tot[2];
            job.out[3] = tot[3] * tot[4];
        }
    }
}

// As a kernel of its own, where the placement is no single kernel (more than kFoldMaxBlocks blocks of the counting sort): more
// than 512 rows, for which 32 warps take less time than eight with four times the requests (a call of 33,000 tokens of 192
// candidates 142.5 us with eight, 138.9 so; 65,536 tokens of 512 candidates 587, 559).
__global__ void __launch_bounds__(kStatManyRowsThreads)
stats_final_kernel(const StatsJob job, int T, int K, int n_real, int n_cand) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ __align__(16) StatsShared<kStatManyRowsThreads> sh;
    stats_final<kStatManyRowsThreads, kStatManyRowsDeep>(job, T, K, n_real, n_cand, sh);
}

// ---------------------------------------------------------------------------------------------
// Counting sort, passes 2 + 3 in one launch (used while the CTA histograms are few): every CTA
// sums the histogram columns itself (pairs of each expert in earlier CTAs, and in all CTAs), scans
// the expert totals, and places the slots of its kSortTokens tokens.  A token selects an expert at most
// once, so a slot's rank among its CTA's pairs of the expert is a popcount over a bit mask of the CTA's
// tokens (one shared-memory atomicOr per slot instead of two passes of match.any over them).  CTA 0
// also publishes counts, offsets and the counters; the tile list is filled by all CTAs, a share each.
// What bounds it is the chain of dependent steps, not the data: of the 5.5 us that a CTA took, 1.4 (2 blocks)
// to 3.2 (64) went to staging and summing the histograms in shared memory and 1 to the fence of a ticket by
// which the last CTA cleared them.
// A statistics call (STATS) adds one CTA, which takes the final sums beside the placement instead of behind it.
// ---------------------------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kMaskWords = kSortTokens / 32;

template <bool STATS>
__global__ void __launch_bounds__(kScanThreads)
slot_scan_place_kernel(const int32_t *__restrict__ topk_idx, int T, int K, int n_real, int nblk,
                       const int32_t *__restrict__ block_hist, int32_t *__restrict__ counts,
                       int32_t *__restrict__ offsets, int32_t *__restrict__ n_pairs_out, int32_t *__restrict__ meta,
                       const WorkLists wl, int tile_rows, int32_t *__restrict__ perm, int32_t *__restrict__ perm_user,
                       int32_t *__restrict__ inv, int32_t *__restrict__ pair_token, const StatsJob job, int n_cand) {
    static_assert(kStatFinalThreads == kScanThreads, "one CTA size for both");
    if (STATS && (int)blockIdx.x == nblk) {
        __shared__ __align__(16) StatsShared<kStatFinalThreads> stats;
        pdl_launch_dependents();
        pdl_wait();
        stats_final<kStatFinalThreads, kStatFinalDeep>(job, T, K, n_real, n_cand, stats);
        return;
    }
    __shared__ ScanShared sh;
    extern __shared__ __align__(16) uint32_t place_smem[];  // token masks [n_real][kMaskWords], then base[n_real]
    uint32_t *mask = place_smem;
    int32_t *base = reinterpret_cast<int32_t *>(mask + kMaskWords * n_real);
    pdl_launch_dependents();
    for (int i = threadIdx.x; i < n_real * kMaskWords; i += blockDim.x) mask[i] = 0u;
    for (int e = threadIdx.x; e < n_real; e += blockDim.x) { base[e] = 0; sh.cnt[e] = 0; }
    const uint32_t inv_k = (65536u + K - 1) / K;  // i / K = i * inv_k >> 16 for i < kSortTokens * kMaxTopK
    __syncthreads();
    pdl_wait();
    // slot s0 + threadIdx.x + kScanThreads * u in e_reg[u], -1 for zero-expert slots and beyond the end
    constexpr int kSlotRegs = kSortTokens * kMaxTopK / kScanThreads;
    const int s0 = blockIdx.x * kSortTokens * K, n_slots = min(T * K - s0, kSortTokens * K);
    int e_reg[kSlotRegs];
#pragma unroll
    for (int u = 0; u < kSlotRegs; ++u) {
        const int i = threadIdx.x + kScanThreads * u;
        const int e = i < n_slots ? __ldcg(topk_idx + s0 + i) : -1;
        e_reg[u] = (unsigned)e >= (unsigned)n_real ? -1 : e;
    }
    // Column sums of the CTA histograms, straight from global memory, sixteen blocks requested at a time;
    // with fewer experts than threads, several threads share a column.
    const int col_parts = max(1, kScanThreads / n_real);
    const int part0 = threadIdx.x / n_real;
    for (int e = threadIdx.x - part0 * n_real; e < n_real && part0 < col_parts; e += kScanThreads) {
        int before = 0, total = 0;
        for (int b0 = part0; b0 < nblk; b0 += 16 * col_parts) {
            int c[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) c[q] = b0 + q * col_parts < nblk ? __ldcg(block_hist + (size_t)(b0 + q * col_parts) * n_real + e) : 0;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                total += c[q];
                if (b0 + q * col_parts < (int)blockIdx.x) before += c[q];
            }
        }
        atomicAdd(&base[e], before);
        atomicAdd(&sh.cnt[e], total);
    }
#pragma unroll
    for (int u = 0; u < kSlotRegs; ++u) {
        const uint32_t tok = (threadIdx.x + kScanThreads * u) * inv_k >> 16;
        if (e_reg[u] >= 0) atomicOr(mask + e_reg[u] * kMaskWords + (tok >> 5), 1u << (tok & 31));
    }
    __syncthreads();
    finish_expert_scan(sh, n_real, T * K, counts, offsets, n_pairs_out, meta, wl, blockIdx.x == 0, blockIdx.x, nblk, tile_rows);
#pragma unroll
    for (int u = 0; u < kSlotRegs; ++u) {
        const int i = threadIdx.x + kScanThreads * u;
        if (i >= n_slots) break;
        const int e = e_reg[u], s = s0 + i, tok = i * inv_k >> 16;
        int p = -1;
        if (e >= 0) {
            const uint4 m = *reinterpret_cast<const uint4 *>(mask + e * kMaskWords);
            const uint32_t w[kMaskWords] = {m.x, m.y, m.z, m.w};
            p = sh.off[e] + base[e];
#pragma unroll
            for (int q = 0; q < kMaskWords; ++q)
                p += __popc(q < (tok >> 5) ? w[q] : q == (tok >> 5) ? w[q] & ((1u << (tok & 31)) - 1u) : 0u);
            perm[p] = s;
            if (perm_user) perm_user[p] = s;
            pair_token[p] = blockIdx.x * kSortTokens + tok;
        }
        inv[s] = p;
    }
}

// ---------------------------------------------------------------------------------------------
// Routing statistics (Eq. 4-6 forward values), two deterministic passes.  The top-K pass of a statistics
// call has each token's logits, softmax maximum and denominator in registers already, so it also adds
// up its CTA's selection counts (integers) and softmax probabilities: every warp in registers over its
// tokens, then the warps in order.  The final pass adds the CTAs' sums in a fixed order.  (As a kernel
// of its own, one thread per candidate walking 64 tokens, the first pass took 49 us for 8192 tokens of
// 192 candidates and the final pass, a chain of loads per candidate, 19 us.)
// ---------------------------------------------------------------------------------------------
constexpr int kStatTokens = 64;
// Warps of a CTA by the logits per lane: sixteen logits a lane do not fit the 64 registers of a thread of 32 warps
// (8192 tokens of 372 candidates: 96.4 us a call with 32 warps, 93.5 with 16).
// The CTA's probabilities, a row of candidates per warp, and its counts need no more shared memory than every launch may have.
template <int RPL>
constexpr int kStatWarps = RPL <= 8 ? 32 : 16;
static_assert((kStatWarps<8> + 1) * 256 <= 12288 && (kStatWarps<16> + 1) * kMaxCand <= 12288, "no opt-in to more than 48 KB is made for the kernel");

template <int RPL>
__global__ void __launch_bounds__(32 * kStatWarps<RPL>)
topk_stats_kernel(const float *__restrict__ logits, int n_parts, int T, int n_real, int n_cand, int K, int gate_mode,
                  int32_t *__restrict__ topk_idx, float *__restrict__ topk_w, int32_t *__restrict__ block_hist, float *__restrict__ part) {
    pdl_launch_dependents();
    constexpr int kWarps = kStatWarps<RPL>;
    extern __shared__ float sm[];  // [kWarps][n_cand] probabilities, then [n_cand] counts
    int32_t *cnt = reinterpret_cast<int32_t *>(sm + kWarps * n_cand);
    for (int i = threadIdx.x; i < n_cand; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    pdl_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = blockIdx.x * kStatTokens, t1 = min(T, t0 + kStatTokens);
    float acc[RPL];
#pragma unroll
    for (int r = 0; r < RPL; ++r) acc[r] = 0.f;
    for (int t = t0 + warp; t < t1; t += kWarps) {
        int my_idx;
        float my_w, v[RPL], m, den;
        topk_gate_token<RPL, 3, true>(logits + (size_t)t * n_cand, n_parts, (size_t)T * n_cand, n_real, n_cand, K, gate_mode, lane,
                             v, m, den, my_idx, my_w);
        if (lane < K) {
            topk_idx[(size_t)t * K + lane] = my_idx;
            topk_w[(size_t)t * K + lane] = my_w;
            atomicAdd(cnt + my_idx, 1);
        }
#pragma unroll
        for (int r = 0; r < RPL; ++r)
            if (r * 32 + lane < n_cand) acc[r] += expf(v[r] - m) / den;
    }
#pragma unroll
    for (int r = 0; r < RPL; ++r)
        if (r * 32 + lane < n_cand) sm[warp * n_cand + r * 32 + lane] = acc[r];
    __syncthreads();
    for (int j = threadIdx.x; j < n_cand; j += blockDim.x) {
        float p = 0.f;
#pragma unroll 8
        for (int w = 0; w < kWarps; ++w) p += sm[w * n_cand + j];
        part[(size_t)blockIdx.x * 2 * n_cand + j] = (float)cnt[j];
        part[(size_t)blockIdx.x * 2 * n_cand + n_cand + j] = p;
        // pass 1 of the counting sort, as in the top-K kernel above
        if (block_hist && j < n_real && cnt[j]) atomicAdd(block_hist + (size_t)(t0 / kSortTokens) * n_real + j, cnt[j]);
    }
}

// Per-token zero-expert ratio (Section 2.2, looked at per token in Section 4.1): the share of the
// token's K slots that selected a zero expert.
__global__ void __launch_bounds__(256)
token_zero_share_kernel(const int32_t *__restrict__ topk_idx, int T, int K, int n_real, float *__restrict__ out) {
    pdl_launch_dependents();
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    int zero = 0;
    for (int k0 = 0; k0 < K; k0 += 8) {  // eight loads in flight
        int e[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) e[u] = __ldcg(topk_idx + (size_t)t * K + min(k0 + u, K - 1));
#pragma unroll
        for (int u = 0; u < 8; ++u) zero += k0 + u < K && e[u] >= n_real ? 1 : 0;
    }
    out[t] = (float)zero / (float)K;
}

}  // namespace

int launch_token_zero_share(const zeda_moe *h, int T, float *out, cudaStream_t s) {
    const cudaError_t e = launch_kernel(h->pdl, token_zero_share_kernel, dim3((T + 255) / 256), dim3(256), 0, s,
                                        (const int32_t *)h->ws.topk_idx, T, (int)h->cfg.top_k, (int)h->cfg.n_real, out);
    return e == cudaSuccess ? 1 : -1;
}

int init_route_kernels(zeda_moe *h) {
    cudaError_t e = cudaSuccess;
    each_router_form([&](auto form, auto kernel) {
        using C = decltype(form);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmem);
        if (e != cudaSuccess) return;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(C::kCtas);
        cfg.blockDim = dim3(C::kThreads);
        cfg.dynamicSmemBytes = C::kSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C::kCtas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int &clusters = C::kCtas == 8 ? h->router_clusters8 : h->router_clusters4;
        if (!clusters) e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg);
        if (e == cudaSuccess && clusters < 1) clusters = 1;
    });
    if (e != cudaSuccess) return -1;
    return 0;
}

int launch_router_logits(const zeda_moe *h, const __nv_bfloat16 *x, int T, float *logits, cudaStream_t s, int *n_parts, int split_T,
                         float *stat_part) {
    if (n_parts) *n_parts = 1;
    if (n_parts && pair_router_path(h, split_T > T ? split_T : T)) {
        *n_parts = 0;
        return launch_router_topk_pair(h, x, T, split_T, hist_ints(h, T) ? h->ws.block_hist : nullptr, stat_part, s);
    }
    // large batches: the GEMM goes to the tensor cores (exact three-way bf16 split of the weights)
    if (T >= kTileRouterTokens) {
        const int split = n_parts ? router_split_factor(h, split_T > T ? split_T : T) : 1;
        if (n_parts) *n_parts = split;
        return launch_router_logits_tile(h, x, T, logits, split, s);
    }
    const int d = h->cfg.d_model, n_cand = h->cfg.n_real + h->cfg.n_zero;
    if (T <= kFewTokens) {
        auto go = [&](auto kernel, int per_cta) {
            return launch_kernel(h->pdl, kernel, dim3(n_cand, (T + per_cta - 1) / per_cta), dim3(kFewThreads), 0, s, x, h->router_w,
                                 h->router_bias, T, d, n_cand, logits, h->ws.block_hist, hist_ints(h, T), h->ws.meta);
        };
        const cudaError_t e = T == 1   ? go(router_logits_few_kernel<1>, 1)
                              : T == 2 ? go(router_logits_few_kernel<2>, 2)
                              : T <= 4 ? go(router_logits_few_kernel<4>, 4)
                                       : go(router_logits_few_kernel<8>, 8);
        return e == cudaSuccess ? 1 : -1;
    }
    // the form of the least work per SM (at the kernel)
    int best = 0, of_best = 0, at = 0;
    auto tiles = [](int n, int per) { return (n + per - 1) / per; };
    each_router_form([&](auto form, auto) {
        using C = decltype(form);
        const int clusters = tiles(n_cand, C::kTileCand) * tiles(T, C::kTileTokens), wave = C::kCtas == 8 ? h->router_clusters8 : h->router_clusters4;
        const int cost = tiles(clusters, wave) * C::kTileTokens * (C::kCtas == 8 ? 2 : 3);
        if (at == 0 || cost <= of_best) { best = at; of_best = cost; }
        ++at;
    });
    cudaError_t e = cudaSuccess;
    at = 0;
    each_router_form([&](auto form, auto kernel) {
        using C = decltype(form);
        if (at++ == best)
            e = launch_kernel(h->pdl, kernel, dim3(tiles(n_cand, C::kTileCand) * C::kCtas, tiles(T, C::kTileTokens)), dim3(C::kThreads), C::kSmem, s, x,
                              h->router_w, h->router_bias, T, d, n_cand, logits, h->ws.block_hist, hist_ints(h, T));
    });
    return e == cudaSuccess ? 1 : -1;
}

// Top-K and routing weights of T tokens from n_parts >= 1 slices of their logits, and pass 1 of the counting sort where it
// counts there (hist_ints).
int launch_topk(const zeda_moe *h, const float *logits, int n_parts, int T, float *stat_part, cudaStream_t s) {
    const zeda_moe_config_t &c = h->cfg;
    const int n_cand = c.n_real + c.n_zero, K = c.top_k;
    const Workspace &ws = h->ws;
    const int topk_warps = T <= 8 * h->sm_count ? 2 : 8;  // the loads of a few tokens spread over all SMs
    int32_t *hist_in_topk = hist_ints(h, T) ? ws.block_hist : nullptr;
    cudaError_t e = cudaSuccess;
#define ZEDA_CALL_TOPK(R) \
    e = launch_kernel(h->pdl, topk_gate_kernel<R>, dim3((T + topk_warps - 1) / topk_warps), dim3(32 * topk_warps), 0, s, logits, n_parts, T, c.n_real, n_cand, K, \
              c.gate_mode, ws.topk_idx, ws.topk_w, hist_in_topk)
#define ZEDA_CALL_STATS(R) \
    e = launch_kernel(h->pdl, topk_stats_kernel<R>, dim3((T + kStatTokens - 1) / kStatTokens), dim3(32 * kStatWarps<R>), \
              sizeof(float) * (kStatWarps<R> + 1) * n_cand, s, logits, n_parts, T, c.n_real, n_cand, K, c.gate_mode, \
              ws.topk_idx, ws.topk_w, hist_in_topk, stat_part)
    if (stat_part) ZEDA_RPL_DISPATCH(ZEDA_CALL_STATS);
    else ZEDA_RPL_DISPATCH(ZEDA_CALL_TOPK);
#undef ZEDA_CALL_TOPK
#undef ZEDA_CALL_STATS
    return e == cudaSuccess ? 1 : -1;
}

int launch_route_from_logits(const zeda_moe *h, const float *logits, int T, const RouteOut &out, cudaStream_t s, int n_parts,
                             const StatsOut *stats) {
    const zeda_moe_config_t &c = h->cfg;
    const int n_cand = c.n_real + c.n_zero, K = c.top_k;
    const Workspace &ws = h->ws;
    const int nblk = (T + kSortTokens - 1) / kSortTokens;
    int launches = 4;
    cudaError_t e = cudaSuccess;  // of the latest launch: nothing is launched behind one that failed
    const WorkLists wl = {ws.ptile_expert, ws.ptile_row0};
    const int tile_rows = tile_rows_for(h, T);
    float *stat_part = stats ? ws.stat_part : nullptr;
    StatsJob job = {};
    if (stats) job = {stat_part, n_parts == 0 ? pair_router_stat_blocks(h, T) : (T + kStatTokens - 1) / kStatTokens, stats->f, stats->p_mean, stats->out};
    if (!stats && T <= kSmallTokens && c.n_real <= kSmallThreads) {
        const bool one_cta = T <= kSmallTokens / kSmallCluster;
#define ZEDA_CALL_SMALL(R)                                                                                         \
    e = launch_kernel(h->pdl, one_cta ? route_small_kernel<R, 1> : route_small_kernel<R, kSmallCluster>,            \
        dim3(one_cta ? 1 : kSmallCluster), dim3(kSmallThreads), 0, s, logits, n_parts, T, c.n_real, n_cand, K, c.gate_mode, ws.topk_idx, ws.topk_w, ws.counts, ws.offsets, out.n_pairs,   \
        ws.meta, wl, tile_rows, ws.perm, out.perm, ws.inv, ws.pair_token)
        ZEDA_RPL_DISPATCH(ZEDA_CALL_SMALL);
#undef ZEDA_CALL_SMALL
        launches = 1;
    } else {
        // up to kFoldMaxBlocks sort blocks the top-K kernel counts the slots itself and one more launch
        // scans and places; beyond, histogram, scan and placement are kernels of their own
        const bool fold = nblk <= kFoldMaxBlocks;
        // no router kernel has cleared the histograms in front of a caller's own logits
        if (fold && n_parts && logits != ws.logits) e = cudaMemsetAsync(ws.block_hist, 0, sizeof(int32_t) * nblk * c.n_real, s);
        if (e != cudaSuccess) return -1;
        if (n_parts == 0) launches = 3;  // the slots are chosen already
        else if (launch_topk(h, logits, n_parts, T, stat_part, s) < 0) return -1;
        if (fold) {
            e = launch_kernel(h->pdl, stats ? slot_scan_place_kernel<true> : slot_scan_place_kernel<false>, dim3(nblk + (stats ? 1 : 0)), dim3(kScanThreads),
                              sizeof(int32_t) * (kMaskWords + 1) * c.n_real, s, (const int32_t *)ws.topk_idx, T, K, c.n_real,
                              nblk, (const int32_t *)ws.block_hist, ws.counts, ws.offsets, out.n_pairs, ws.meta, wl, tile_rows, ws.perm,
                              out.perm, ws.inv, ws.pair_token, job, n_cand);
            launches -= 2;
        } else {
            e = launch_kernel(h->pdl, slot_hist_kernel, dim3(nblk), dim3(256), sizeof(int32_t) * c.n_real, s,
                              (const int32_t *)ws.topk_idx, T, K, c.n_real, ws.block_hist);
            if (e != cudaSuccess) return -1;
            e = launch_kernel(false, expert_scan_kernel, dim3(1), dim3(512), 0, s, ws.block_hist, nblk, c.n_real, T * K, ws.counts,
                              ws.offsets, out.n_pairs, ws.meta, wl, tile_rows);
            if (e != cudaSuccess) return -1;
            e = launch_kernel(false, slot_place_kernel, dim3(nblk), dim3(kPlaceWarps * 32), sizeof(int32_t) * kPlaceWarps * c.n_real, s,
                              (const int32_t *)ws.topk_idx, T, K, c.n_real, (const int32_t *)ws.block_hist, (const int32_t *)ws.offsets,
                              ws.perm, out.perm, ws.inv, ws.pair_token);
            if (stats && e == cudaSuccess) {
                e = launch_kernel(h->pdl, stats_final_kernel, dim3(1), dim3(kStatManyRowsThreads), 0, s, job, T, K, c.n_real, n_cand);
                ++launches;
            }
        }
    }
    if (e != cudaSuccess) return -1;
    // copies for a caller that asked for the routing itself
    auto copy = [&](void *dst, const void *src, size_t n) {
        if (dst && e == cudaSuccess) e = cudaMemcpyAsync(dst, src, 4 * n, cudaMemcpyDeviceToDevice, s);
    };
    copy(out.topk_idx, ws.topk_idx, (size_t)T * K);
    copy(out.topk_w, ws.topk_w, (size_t)T * K);
    copy(out.counts, ws.counts, c.n_real);
    copy(out.offsets, ws.offsets, c.n_real + 1);
    return e == cudaSuccess ? launches : -1;
}

}  // namespace zeda

// ---------------------------------------------------------------------------------------------
// zeda_compact_static: the counting sort above for callers that cannot allocate device memory.
// Its scratch (per-CTA histograms, slot -> position table, pair -> token table, work lists,
// counters) lives in the fixed array below instead of a caller-provided workspace.  Every GPU
// that loads this library holds the array until the process exits.
// ---------------------------------------------------------------------------------------------
namespace zeda {
namespace {

constexpr int kStaticMaxTokens = ZEDA_STATIC_MAX_TOKENS;
constexpr int kStaticMaxSlots = ZEDA_STATIC_MAX_SLOTS;
constexpr int kStaticBlocks = (kStaticMaxTokens + kSortTokens - 1) / kSortTokens;
constexpr int kStaticLists = kStaticMaxSlots / kPairTileM + kMaxCand + 1;

struct StaticScratch {
    int32_t block_hist[kStaticBlocks * kMaxCand];
    int32_t inv[kStaticMaxSlots];
    int32_t pair_token[kStaticMaxSlots];
    int32_t ptile_expert[kStaticLists];
    int32_t ptile_row0[kStaticLists];
    int32_t meta[kMetaCount];
};

static __device__ __align__(256) unsigned char g_static_scratch[sizeof(StaticScratch)];

constexpr int kMaxDevices = 64;
// device address of the array, per device; atomic so that host threads may race on the first call
std::atomic<StaticScratch *> g_static_ptr[kMaxDevices] = {};

}  // namespace
}  // namespace zeda

extern "C" zeda_status_t zeda_compact_static(const int32_t *topk_idx, int32_t T, int32_t top_k, int32_t n_real,
                                             int32_t *expert_counts, int32_t *expert_offsets, int32_t *perm,
                                             int32_t *n_pairs, void *stream) {
    using namespace zeda;
    if (T == 0) return ZEDA_OK;
    if (T < 0 || T > kStaticMaxTokens || top_k < 1 || top_k > kMaxTopK || (long long)T * top_k > kStaticMaxSlots) {
        set_error("zeda_compact_static handles at most %d tokens and %d slots (T * top_k); got T=%d, top_k=%d",
                  kStaticMaxTokens, kStaticMaxSlots, T, top_k);
        return ZEDA_ERR_UNSUPPORTED;
    }
    if (n_real < 1 || n_real > kMaxCand) { set_error("n_real must be in [1, %d]", kMaxCand); return ZEDA_ERR_UNSUPPORTED; }
    if (!topk_idx || !expert_counts || !expert_offsets || !perm || !n_pairs) {
        set_error("zeda_compact_static: every pointer is required");
        return ZEDA_ERR_INVALID_ARG;
    }
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) { set_error("cudaGetDevice: %s", cudaGetErrorString(e)); return ZEDA_ERR_CUDA; }
    if (dev < 0 || dev >= kMaxDevices) { set_error("device ordinal %d not supported", dev); return ZEDA_ERR_UNSUPPORTED; }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    StaticScratch *sc = g_static_ptr[dev].load(std::memory_order_acquire);
    if (!sc) {
        // One-time set-up for this device: in host code the array's name is only a stand-in, the
        // kernels need its device address.  The lookup is not a stream operation, so it must not
        // happen while the stream is being captured.
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        e = cudaStreamIsCapturing(s, &cap);
        if (e != cudaSuccess) { set_error("cudaStreamIsCapturing: %s", cudaGetErrorString(e)); return ZEDA_ERR_CUDA; }
        if (cap != cudaStreamCaptureStatusNone) {
            set_error("zeda_compact_static: the first call on a device must come before stream capture begins");
            return ZEDA_ERR_INVALID_ARG;
        }
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) { set_error("cudaGetSymbolAddress: %s", cudaGetErrorString(e)); return ZEDA_ERR_CUDA; }
        sc = static_cast<StaticScratch *>(p);
        g_static_ptr[dev].store(sc, std::memory_order_release);  // every thread would store the same address
    }
    // the array keeps the previous call's contents; the counters start from zero every call
    e = cudaMemsetAsync(sc->meta, 0, sizeof(sc->meta), s);
    if (e != cudaSuccess) { set_error("cudaMemsetAsync: %s", cudaGetErrorString(e)); return ZEDA_ERR_CUDA; }
    const int nblk = (T + kSortTokens - 1) / kSortTokens;
    slot_hist_kernel<<<nblk, 256, sizeof(int32_t) * n_real, s>>>(topk_idx, T, top_k, n_real, sc->block_hist);
    const WorkLists wl = {sc->ptile_expert, sc->ptile_row0};
    expert_scan_kernel<<<1, 512, 0, s>>>(sc->block_hist, nblk, n_real, T * top_k, expert_counts, expert_offsets,
                                         n_pairs, sc->meta, wl, kPairTileM);
    slot_place_kernel<<<nblk, kPlaceWarps * 32, sizeof(int32_t) * kPlaceWarps * n_real, s>>>(
        topk_idx, T, top_k, n_real, sc->block_hist, expert_offsets, perm, nullptr, sc->inv, sc->pair_token);
    e = cudaGetLastError();
    if (e != cudaSuccess) { set_error("zeda_compact_static launch: %s", cudaGetErrorString(e)); return ZEDA_ERR_CUDA; }
    return ZEDA_OK;
}

