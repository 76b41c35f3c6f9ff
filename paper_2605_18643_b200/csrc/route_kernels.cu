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
// Router logits, CUDA-core version: l[t, j] = <x_t, W_r[j]> + b[j] in fp32.
// One CTA = kTok tokens (bf16 rows staged in shared memory) x a slice of the candidates; one warp
// per candidate row, lanes striding the feature axis with 16-byte loads.
// ---------------------------------------------------------------------------------------------
constexpr int kTok = 8;
constexpr int kRouterUnroll = 8;  // 16-byte weight loads a lane keeps in flight

__global__ void __launch_bounds__(256)
router_logits_kernel(const __nv_bfloat16 *__restrict__ x, const float *__restrict__ router_w,
                     const float *__restrict__ router_bias, int T, int d, int n_cand,
                     int cand_per_cta, float *__restrict__ logits, int32_t *__restrict__ hist, int n_hist) {
    pdl_launch_dependents();
    pdl_wait();
    clear_hist(hist, n_hist);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __nv_bfloat16 *xs = reinterpret_cast<__nv_bfloat16 *>(smem_raw);  // [kTok][d]
    const int t0 = blockIdx.x * kTok;
    const int nt = min(kTok, T - t0);
    const int vec_per_row = d / 8;
    // eight 16-byte loads in flight per thread (a plain load-store loop waits for each load in turn)
    for (int i0 = threadIdx.x; i0 < kTok * vec_per_row; i0 += 8 * blockDim.x) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * blockDim.x;
            const int r = i / vec_per_row, c = i % vec_per_row;
            v[u] = make_uint4(0, 0, 0, 0);
            if (i < kTok * vec_per_row && r < nt) v[u] = __ldcg(reinterpret_cast<const uint4 *>(x + (size_t)(t0 + r) * d) + c);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i < kTok * vec_per_row) reinterpret_cast<uint4 *>(xs + (size_t)(i / vec_per_row) * d)[i % vec_per_row] = v[u];
        }
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j_begin = blockIdx.y * cand_per_cta;
    const int j_end = min(n_cand, j_begin + cand_per_cta);
    for (int j = j_begin + warp; j < j_end; j += 8) {
        float acc[kTok];
#pragma unroll
        for (int r = 0; r < kTok; ++r) acc[r] = 0.f;
        const float4 *wrow = reinterpret_cast<const float4 *>(router_w + (size_t)j * d);
        for (int c4 = lane; c4 < d / 4; c4 += 32 * kRouterUnroll) {
            float4 w[kRouterUnroll];
#pragma unroll
            for (int u = 0; u < kRouterUnroll; ++u)  // independent 16-byte loads in flight per lane
                w[u] = (c4 + 32 * u < d / 4) ? __ldg(wrow + c4 + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < kRouterUnroll; ++u) {
                if (c4 + 32 * u < d / 4) {
#pragma unroll
                    for (int r = 0; r < kTok; ++r) {
                        const uint2 xv = reinterpret_cast<const uint2 *>(xs + (size_t)r * d)[c4 + 32 * u];
                        const float x0 = __uint_as_float(xv.x << 16), x1 = __uint_as_float(xv.x & 0xffff0000u);
                        const float x2 = __uint_as_float(xv.y << 16), x3 = __uint_as_float(xv.y & 0xffff0000u);
                        acc[r] = fmaf(w[u].x, x0, acc[r]);
                        acc[r] = fmaf(w[u].y, x1, acc[r]);
                        acc[r] = fmaf(w[u].z, x2, acc[r]);
                        acc[r] = fmaf(w[u].w, x3, acc[r]);
                    }
                }
            }
        }
        const float b = router_bias ? __ldg(router_bias + j) : 0.f;
#pragma unroll
        for (int r = 0; r < kTok; ++r) {
            const float s = warp_sum(acc[r]);
            if (lane == 0 && r < nt) logits[(size_t)(t0 + r) * n_cand + j] = s + b;
        }
    }
}

// Few tokens: one candidate row per CTA, so that the rows (1.5 MB for 192 candidates of 2048) are read by
// 192 SM-wide bursts instead of 24; the reduction axis is split over four warps.  NT tokens per CTA, all
// of their loads in flight at once.  The row is asked into L2 before the wait for the kernel in front (a
// prefetch only: its values are read after the wait).
// From kTileRouterTokens on the tensor-core routers.  Their accumulators are fp32 too, but against 64 bits its logits
// are off by 2.1e-6 of their root mean square at d 2048 (1.0e-6 at 1024, 9e-6 at 8192), these kernels' by 1.6e-7:
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

// Sliced router of 33 to 255 tokens: kSliceTokens x kSliceCand logits per CTA over a slice of the reduction axis, each of its
// eight warps over an eighth of the slice, 8 x 4 logits per lane.  A warp copies what it needs into shared memory by itself,
// all of it at once (its router rows before the wait for the kernel in front: they are the caller's constants), so a CTA
// waits for memory once; the products then take 16 loads of 16 bytes per 256 fused multiply-adds.  (The kernel above, a warp
// per candidate row and 8 tokens, converts every x value once per candidate and waits for each row.)  Sums are fp32, of runs
// of 16 products, then of the runs, the warps and, in the top-K pass, the slices; the bias comes behind them.
constexpr int kSliceTokens = 32, kSliceCand = 32, kSliceWarps = 8;
constexpr int kSliceRedLd = 40;   // floats between the tokens of a warp's sums: the lanes of a store hit all banks
constexpr int kSliceRun = 2;      // octets of products added up before they go to the total
constexpr int kSliceMinPart = 256;  // elements of the reduction axis that make a slice worth it
constexpr int kSliceMaxParts = 7;   // with the bias as many as the top-K pass requests at a time (8 where they would not fit otherwise)
constexpr int kSliceMinModel = 1024, kSliceMinLogits = 4000;   // d, and T x candidates
constexpr long long kSliceMinProducts = 12600000;              // T x candidates x d
constexpr int kSliceMaxSmem = 200 * 1024;

// Bytes between the rows of a warp's operands of `octets` groups of eight elements: odd multiples of 16, so that rows next
// to one another lie in different banks.
__host__ __device__ constexpr int slice_x_stride(int octets) { return 16 * (octets | 1); }
__host__ __device__ constexpr int slice_w_stride(int octets) { return 32 * octets + 16; }
__host__ __device__ constexpr int slice_warp_octets(int d, int parts) { return ((d / 8 + parts - 1) / parts + kSliceWarps - 1) / kSliceWarps; }

size_t slice_smem(int d, int parts) {
    const int n = slice_warp_octets(d, parts);
    const size_t operands = (size_t)kSliceWarps * (kSliceTokens * slice_x_stride(n) + kSliceCand * slice_w_stride(n));
    const size_t sums = (size_t)kSliceWarps * kSliceTokens * kSliceRedLd * sizeof(float);
    return operands > sums ? operands : sums;
}

__global__ void __launch_bounds__(32 * kSliceWarps, 1)
router_logits_slice_kernel(const __nv_bfloat16 *__restrict__ x, const float *__restrict__ router_w, int T, int d, int n_cand,
                           float *__restrict__ logits, int32_t *__restrict__ hist, int n_hist) {
    pdl_launch_dependents();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j0 = blockIdx.x * kSliceCand, t0 = blockIdx.y * kSliceTokens, part = blockIdx.z, parts = gridDim.z;
    const int o0 = d / 8 * part / parts, o1 = d / 8 * (part + 1) / parts;
    const int q0 = o0 + (o1 - o0) * warp / kSliceWarps, n = o0 + (o1 - o0) * (warp + 1) / kSliceWarps - q0;  // this warp's octets, 4 to 16
    const int octets = slice_warp_octets(d, parts);
    const int xs = slice_x_stride(octets), ws = slice_w_stride(octets);
    unsigned char *xb = smem_raw + warp * (kSliceTokens * xs + kSliceCand * ws), *wb = xb + kSliceTokens * xs;
    auto copy16 = [](void *dst, const void *src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
    };
    const int rows_w = min(kSliceCand, n_cand - j0), rows_x = min(kSliceTokens, T - t0);
    {
        const uint32_t inv = (1u << 20) / (2 * n) + 1;  // i / (2 n) = i * inv >> 20 for the i below
        for (int i = lane; i < rows_w * 2 * n; i += 32) {
            const int r = i * inv >> 20, c = i - r * 2 * n;
            copy16(wb + r * ws + 16 * c, router_w + (size_t)(j0 + r) * d + 8 * q0 + 4 * c);
        }
    }
    pdl_wait();
    {
        const int cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        for (int i = cta * blockDim.x + threadIdx.x; i < n_hist; i += gridDim.x * gridDim.y * gridDim.z * blockDim.x) hist[i] = 0;
    }
    {
        const uint32_t inv = (1u << 20) / n + 1;
        for (int i = lane; i < rows_x * n; i += 32) {
            const int r = i * inv >> 20, c = i - r * n;
            copy16(xb + r * xs + 16 * c, x + (size_t)(t0 + r) * d + 8 * (q0 + c));
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    // lane: tokens tg + 4 i, candidates cg + 8 j (rows beyond the call's hold what was there: their sums are not stored)
    const int tg = lane >> 3, cg = lane & 7;
    float acc[8][4], tot[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = tot[i][j] = 0.f;
    for (int q = 0; q < n; ++q) {
        uint4 xv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) xv[i] = *reinterpret_cast<const uint4 *>(xb + (tg + 4 * i) * xs + 16 * q);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float4 w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4 *>(wb + (cg + 8 * j) * ws + 32 * q + 16 * h);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t lo = h ? xv[i].z : xv[i].x, hi = h ? xv[i].w : xv[i].y;
                const float x0 = __uint_as_float(lo << 16), x1 = __uint_as_float(lo & 0xffff0000u);
                const float x2 = __uint_as_float(hi << 16), x3 = __uint_as_float(hi & 0xffff0000u);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fmaf(w[j].x, x0, acc[i][j]);
                    acc[i][j] = fmaf(w[j].y, x1, acc[i][j]);
                    acc[i][j] = fmaf(w[j].z, x2, acc[i][j]);
                    acc[i][j] = fmaf(w[j].w, x3, acc[i][j]);
                }
            }
        }
        if ((q + 1) % kSliceRun == 0 || q + 1 == n) {  // (uniform)
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) { tot[i][j] += acc[i][j]; acc[i][j] = 0.f; }
        }
    }
    __syncthreads();  // the operands have been read: their room takes the warps' sums
    float *red = reinterpret_cast<float *>(smem_raw);  // [kSliceWarps][kSliceTokens][kSliceRedLd]
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) red[(warp * kSliceTokens + tg + 4 * i) * kSliceRedLd + cg + 8 * j] = tot[i][j];
    __syncthreads();
    const int r = threadIdx.x >> 3, c = (threadIdx.x & 7) * 4;  // four candidates of a token per thread
    float4 v[kSliceWarps];
#pragma unroll
    for (int q = 0; q < kSliceWarps; ++q) v[q] = *reinterpret_cast<const float4 *>(red + (q * kSliceTokens + r) * kSliceRedLd + c);
#pragma unroll
    for (int o = 1; o < kSliceWarps; o *= 2)
#pragma unroll
        for (int q = 0; q < kSliceWarps; q += 2 * o) v[q] = make_float4(v[q].x + v[q + o].x, v[q].y + v[q + o].y, v[q].z + v[q + o].z, v[q].w + v[q + o].w);
    if (r >= rows_x) return;
    float *out = logits + ((size_t)part * T + t0 + r) * n_cand + j0;
    const float s[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (c + j < rows_w) out[c + j] = s[j];
}

// Slices of the reduction axis for a call of T tokens by that kernel, 0 where the one above takes the call: as many as give
// every SM at most one CTA, but no fewer than fit its shared memory.  Routing pass, us, by the kernel above and by this:
//   d 2048, 192 candidates   T=33 13.8, 11.2    T=64 13.2, 11.4    T=128 15.7, 12.7   T=193 20.2, 15.9   T=255 27.0, 16.7
//   d 2048, 96               T=33 11.2, 11.9    T=64 11.9, 12.2    T=96 13.7, 12.1    T=193 15.3, 11.7   T=255 15.3, 12.3
//   d 1024, 96               T=33 9.3, 10.8     T=64 10.1, 11.0    T=128 11.2, 11.7   T=129 12.6, 11.5   T=255 13.2, 11.8
//   d 2048, 12               T=33 8.9, 9.7      T=128 9.3, 10.1    T=255 11.0, 10.4
//   d 8192, 400              T=33 39.2, 36.6    T=128 103.5, 51.5  T=255 171, 85
//   d 2048, 512              T=33 20.6, 19.3    T=128 34.6, 25.7   T=129 31.3, 35.1   T=160 40.2, 33.9
// So few logits stay there, and calls (the last row's 129 tokens) whose last wave here would be a handful of CTAs.  The
// weights' distance from 64 bits, 2-norms: d 1024 1.0e-7 and 9.3e-8, d 2048 1.6e-7 and 1.3e-7, d 8192 5e-7 and 2.6e-7.
int router_slices(const zeda_moe *h, int T) {
    const int d = h->cfg.d_model, n_cand = h->cfg.n_real + h->cfg.n_zero;
    if (T <= kFewTokens || T >= kTileRouterTokens || d < kSliceMinModel || T * n_cand < kSliceMinLogits ||
        (long long)T * n_cand * d < kSliceMinProducts)
        return 0;
    const int tiles = ((T + kSliceTokens - 1) / kSliceTokens) * ((n_cand + kSliceCand - 1) / kSliceCand);
    int parts = h->sm_count / tiles;
    if (parts > d / kSliceMinPart) parts = d / kSliceMinPart;
    parts = parts < 1 ? 1 : parts > kSliceMaxParts ? kSliceMaxParts : parts;
    while (parts < kRouterMaxSplit && slice_smem(d, parts) > kSliceMaxSmem) ++parts;
    const int ctas = tiles * parts;
    return ctas > h->sm_count && 10 * ctas <= 11 * h->sm_count ? 0 : parts;
}

// block_hist (optional): pass 1 of the counting sort done here.  Every slot on a normal expert adds 1
// to its entry of the histogram of its block of kSortTokens tokens (integer adds: the counts do not
// depend on their order).  The histograms must be zero on entry: the call's router kernel clears them.
template <int RPL, bool LATE>
__global__ void __launch_bounds__(256)
topk_gate_kernel(const float *__restrict__ logits, int n_parts, const float *__restrict__ late_bias, int T, int n_real, int n_cand, int K, int gate_mode,
                 int32_t *__restrict__ topk_idx, float *__restrict__ topk_w, int32_t *__restrict__ block_hist) {
    pdl_launch_dependents();
    pdl_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + warp;
    if (t >= T) return;
    int my_idx;
    float my_w, v[RPL], m, den;
    topk_gate_token<RPL, LATE>(logits + (size_t)t * n_cand, n_parts, (size_t)T * n_cand, late_bias, n_real, n_cand, K, gate_mode, lane,
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
template <int RPL, int CLUSTER, bool LATE>
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(kSmallThreads)
route_small_kernel(const float *__restrict__ logits, int n_parts, const float *__restrict__ late_bias, int T, int n_real, int n_cand, int K, int gate_mode,
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
        topk_gate_token<RPL, LATE>(logits + (size_t)t * n_cand, n_parts, (size_t)T * n_cand, late_bias, n_real, n_cand, K, gate_mode, lane, v, m, den, my_idx, my_w);
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
// rows allow 16-byte loads) is shared by as many threads as fit, each adding every n-th row, 32 requested at a time and
// added up pairwise (8192 tokens of 192 candidates: 45.3 us a call with the sums behind the placement, 43.5 beside it with
// sixteen rows at a time, 36.8 with 32).
struct StatsJob {
    const float *part;
    int rows;  // of part
    float *f, *p_mean, *out;
};

__device__ __forceinline__ float4 add_columns(const float4 &a, const float4 &b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float2 add_columns(const float2 &a, const float2 &b) { return make_float2(a.x + b.x, a.y + b.y); }

constexpr int kStatFinalThreads = 256;

struct StatsShared {
    float col[2 * kMaxCand];
    float red[5][kStatFinalThreads / 32];
};

template <typename V>
__device__ __forceinline__ void sum_stat_columns(const StatsJob &job, int cols, float *col) {
    constexpr int kDeep = 32;
    const int groups = cols / (int)(sizeof(V) / sizeof(float)), segs = max(1, kStatFinalThreads / groups), seg = threadIdx.x / groups;
    for (int c0 = 0; c0 < groups; c0 += kStatFinalThreads) {  // (more than one turn only where each group has one thread)
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
        for (int s = 0; s < segs; ++s) {  // the shares of a group in order
            if (on && (segs == 1 || seg == s)) {
                V *dst = reinterpret_cast<V *>(col) + c;
                *dst = s == 0 ? a : add_columns(*dst, a);
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ void stats_final(const StatsJob &job, int T, int K, int n_real, int n_cand, StatsShared &sh) {
    if (n_cand % 2 == 0) sum_stat_columns<float4>(job, 2 * n_cand, sh.col);
    else sum_stat_columns<float2>(job, 2 * n_cand, sh.col);
    float sums[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    for (int j = threadIdx.x; j < n_cand; j += kStatFinalThreads) {
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
        for (int i = 0; i < 5; ++i) tot[i] = warp_sum(threadIdx.x < kStatFinalThreads / 32 ? sh.red[i][threadIdx.x] : 0.f);
        if (threadIdx.x == 0) {
            job.out[0] = tot[3] / K;
            job.out[1] = tot[0];
            job.out[2] = tot[1] * tot[2];
            job.out[3] = tot[3] * tot[4];
        }
    }
}

// as a kernel of its own, where the placement is no single kernel (more than kFoldMaxBlocks blocks of the counting sort)
__global__ void __launch_bounds__(kStatFinalThreads)
stats_final_kernel(const StatsJob job, int T, int K, int n_real, int n_cand) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ __align__(16) StatsShared sh;
    stats_final(job, T, K, n_real, n_cand, sh);
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
        __shared__ __align__(16) StatsShared stats;
        pdl_launch_dependents();
        pdl_wait();
        stats_final(job, T, K, n_real, n_cand, stats);
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

template <int RPL, bool LATE>
__global__ void __launch_bounds__(32 * kStatWarps<RPL>)
topk_stats_kernel(const float *__restrict__ logits, int n_parts, const float *__restrict__ late_bias, int T, int n_real, int n_cand, int K, int gate_mode,
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
        topk_gate_token<RPL, LATE, 3, true>(logits + (size_t)t * n_cand, n_parts, (size_t)T * n_cand, late_bias, n_real, n_cand, K, gate_mode, lane,
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

int init_route_kernels(const zeda_moe *h) {
    const size_t smem = (size_t)kTok * h->cfg.d_model * sizeof(__nv_bfloat16);
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(router_logits_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    if (cudaFuncSetAttribute(router_logits_slice_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSliceMaxSmem) != cudaSuccess) return -1;
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
    if (T >= kTileRouterTokens && h->router_maps) {
        const int split = n_parts ? router_split_factor(h, split_T > T ? split_T : T) : 1;
        if (n_parts) *n_parts = split;
        return launch_router_logits_tile(h, x, T, logits, split, s);
    }
    const int d = h->cfg.d_model, n_cand = h->cfg.n_real + h->cfg.n_zero;
    const int tiles = (T + kTok - 1) / kTok;
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
    if (const int parts = n_parts ? router_slices(h, T) : 0) {
        *n_parts = parts;
        const cudaError_t e = launch_kernel(h->pdl, router_logits_slice_kernel, dim3((n_cand + kSliceCand - 1) / kSliceCand, (T + kSliceTokens - 1) / kSliceTokens, parts),
                                            dim3(32 * kSliceWarps), slice_smem(d, parts), s, x, h->router_w, T, d, n_cand, logits, h->ws.block_hist, hist_ints(h, T));
        return e == cudaSuccess ? 1 : -1;
    }
    // split the candidates over grid.y until the grid covers the SMs about twice
    int splits = 1;
    const int max_splits = (n_cand + 7) / 8;
    while (tiles * splits < 2 * h->sm_count && splits < max_splits) splits *= 2;
    if (splits > max_splits) splits = max_splits;
    const int per = (n_cand + splits - 1) / splits;
    const size_t smem = (size_t)kTok * d * sizeof(__nv_bfloat16);
    const cudaError_t e = launch_kernel(h->pdl, router_logits_kernel, dim3(tiles, (n_cand + per - 1) / per), dim3(256), smem, s,
                                        x, h->router_w, h->router_bias, T, d, n_cand, per, logits, h->ws.block_hist, hist_ints(h, T));
    return e == cudaSuccess ? 1 : -1;
}

namespace {
// what the top-K pass has to add to the sum of its slices: the bias, if they are the sliced router's
const float *bias_of_slices(const zeda_moe *h, const float *logits, int T) {
    return logits == h->ws.logits && router_slices(h, T) > 0 ? h->router_bias : nullptr;
}
}  // namespace

// Top-K and routing weights of T tokens from n_parts >= 1 slices of their logits, and pass 1 of the counting sort where it
// counts there (hist_ints).
int launch_topk(const zeda_moe *h, const float *logits, int n_parts, int T, float *stat_part, cudaStream_t s) {
    const zeda_moe_config_t &c = h->cfg;
    const int n_cand = c.n_real + c.n_zero, K = c.top_k;
    const Workspace &ws = h->ws;
    const int topk_warps = T <= 8 * h->sm_count ? 2 : 8;  // the loads of a few tokens spread over all SMs
    int32_t *hist_in_topk = hist_ints(h, T) ? ws.block_hist : nullptr;
    const float *late_bias = bias_of_slices(h, logits, T);
    cudaError_t e = cudaSuccess;
#define ZEDA_CALL_TOPK(R) \
    e = launch_kernel(h->pdl, late_bias ? topk_gate_kernel<R, true> : topk_gate_kernel<R, false>, dim3((T + topk_warps - 1) / topk_warps), dim3(32 * topk_warps), 0, s, logits, n_parts, late_bias, T, c.n_real, n_cand, K, \
              c.gate_mode, ws.topk_idx, ws.topk_w, hist_in_topk)
#define ZEDA_CALL_STATS(R) \
    e = launch_kernel(h->pdl, late_bias ? topk_stats_kernel<R, true> : topk_stats_kernel<R, false>, dim3((T + kStatTokens - 1) / kStatTokens), dim3(32 * kStatWarps<R>), \
              sizeof(float) * (kStatWarps<R> + 1) * n_cand, s, logits, n_parts, late_bias, T, c.n_real, n_cand, K, c.gate_mode, \
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
    const float *late_bias = bias_of_slices(h, logits, T);
    float *stat_part = stats ? ws.stat_part : nullptr;
    StatsJob job = {};
    if (stats) job = {stat_part, n_parts == 0 ? pair_router_stat_blocks(h, T) : (T + kStatTokens - 1) / kStatTokens, stats->f, stats->p_mean, stats->out};
    if (!stats && T <= kSmallTokens && c.n_real <= kSmallThreads) {
        const bool one_cta = T <= kSmallTokens / kSmallCluster;
#define ZEDA_CALL_SMALL(R)                                                                                         \
    e = launch_kernel(h->pdl, one_cta ? route_small_kernel<R, 1, false>                                             \
                              : late_bias ? route_small_kernel<R, kSmallCluster, true> : route_small_kernel<R, kSmallCluster, false>, \
        dim3(one_cta ? 1 : kSmallCluster), dim3(kSmallThreads), 0, s, logits, n_parts, late_bias, T, c.n_real, n_cand, K, c.gate_mode, ws.topk_idx, ws.topk_w, ws.counts, ws.offsets, out.n_pairs,   \
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
                e = launch_kernel(h->pdl, stats_final_kernel, dim3(1), dim3(kStatFinalThreads), 0, s, job, T, K, c.n_real, n_cand);
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

