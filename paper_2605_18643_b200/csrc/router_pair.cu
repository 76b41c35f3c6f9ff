// Router with top-K for large batches of up to 256 candidates (pair_router_path below says which): logits, softmax, selection and routing weights
// (Section 2.1) in one kernel, and the block histograms that the counting sort starts from.
//
// The fp32 router rows come as three bf16 pieces (exact, see router_tile.cu).  Tokens are the M operand of MMAs
// on CTA pairs (256 tokens, 128 per CTA) and all candidates are N, so nothing is computed for padding beyond a
// multiple of 32 candidates and a pair brings in the router rows once per 256 tokens, half of them in each CTA.
// The large products (hi) accumulate apart from the small ones (mid + lo).  Where the tiles of 256 tokens leave
// SMs idle, a cluster takes one tile in two or three pairs, each a slice of the reduction axis.  Every CTA leaves its
// partial logits in its shared memory and finishes 1/slices of its half's 128 tokens, a warp two at a time, fetching
// the other slices' rows from their CTAs (two tokens ahead).
//
// What bounds it, at 8192 tokens of 192 candidates (two slices): 2.7 us to the first operands, 16 k-steps of 0.69 us
// (twelve MMAs of 96 cycles each; every SM takes 52 KB from L2 meanwhile), 1.6 us to the last MMA's end, 1.6 us to
// lay the logits out and meet, then the top-K of 64 tokens per SM, whose instructions and shuffles take longer than
// the exchange.  26 us against 28.5 for the logits alone on the kernel of router_tile.cu and 8 for a top-K pass behind
// it: the routing statistics of 8192 tokens 51.9 -> 44.4 us a call.  Routing weights of 4096 tokens of d 2048 are 4.2e-7
// of their norm off 64 bits (6.4e-7 there), and of 409,600 tokens' top 8 of 192, 3 fall otherwise than in 64 bits (11).
#include "tc_common.cuh"

#include "route_token.cuh"

namespace zeda {

namespace {

using namespace tc;

constexpr int kBlockK = 64;
constexpr int kTokens = 128;                     // tokens of a CTA
constexpr int kXBytes = kTokens * kBlockK * 2;   // 16 KB
constexpr int kWarps = 16;
constexpr int kThreads = 32 * kWarps;
constexpr int kMaxStages = 8;
constexpr int kMaxSlices = 3;
constexpr int kTogether = 2;                     // tokens that a warp finishes together
constexpr int kRingBytes = 216 * 1024;           // most bytes of the ring; the logits take its place behind the last k-step
constexpr int kMidLoCol = 256, kHiOddCol = 128;  // TMEM columns of the accumulators (hi: 0)

struct PairRouterMaps {
    CUtensorMap w_split;  // [3][NC_pad][d] bf16, box {64, n_cols / 2, 3}
    int n_cols;           // candidates rounded up to 32
    int max_clusters[kMaxSlices + 1];  // of 2 * slices CTAs that fit the GPU at a time
};

__host__ __device__ constexpr int stage_bytes(int n_cols) { return kXBytes + 3 * (n_cols / 2) * kBlockK * 2; }
__host__ __device__ constexpr int ring_stages(int n_cols) {
    return kRingBytes / stage_bytes(n_cols) < kMaxStages ? kRingBytes / stage_bytes(n_cols) : kMaxStages;
}
// floats from row to row of the partial logits: a multiple of 16 bytes, four banks apart
__host__ __device__ constexpr int logit_stride(int n_cols) { return n_cols + 4; }

// 16 columns of fp32 from TMEM; the registers are valid after tmem_ld_wait()
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}

__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

// Arrive on the mbarrier at this shared-memory offset in both CTAs of the pair that starts at cluster rank `first`.
__device__ __forceinline__ void commit_pair_of(uint32_t bar, uint32_t first) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)(3u << first)) : "memory");
}

struct PairRouterArgs {
    const float *bias;
    int T, n_real, n_cand, n_cols, k_steps, slices, K, gate_mode;
    int32_t *topk_idx;
    float *topk_w;
    int32_t *block_hist;  // NULL: no histograms
    float *stat_part;     // STATS: per CTA selection counts and probabilities of all candidates
    int32_t *meta;
};

// A cluster of 2 * slices CTAs per tile of 256 tokens; CTA rank = 2 * slice + half of the tile.
template <int RPL, bool STATS>
__global__ void __launch_bounds__(kThreads, 1)
router_topk_pair_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const PairRouterArgs a) {
    pdl_launch_dependents();
    extern __shared__ __align__(1024) unsigned char pr_smem[];
    __shared__ __align__(8) unsigned long long bars[2 * kMaxStages + 1];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ int32_t s_cnt[STATS ? kPairRouterMaxCand : 1];
    const int stages = ring_stages(a.n_cols), stage_size = stage_bytes(a.n_cols);
    const uint32_t ring = (smem_u32(pr_smem) + 1023u) & ~1023u;
    float *logits = reinterpret_cast<float *>(pr_smem + (ring - smem_u32(pr_smem)));  // [128 tokens][stride]
    const uint32_t bar_full = smem_u32(&bars[0]);  // used in the pair's leader CTA only
    const uint32_t bar_empty = smem_u32(&bars[kMaxStages]);
    const uint32_t bar_done = smem_u32(&bars[2 * kMaxStages]);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int half = rank & 1, slice = rank >> 1, slices = a.slices;
    const bool leader = half == 0;
    const uint32_t first = rank & ~1u;  // the pair's leader
    const int tile = blockIdx.x / (2 * slices), tok0 = tile * 2 * kTokens + half * kTokens;
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int i = 0; i < stages; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1); }
        mbar_init(bar_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if constexpr (STATS)
        for (int i = threadIdx.x; i < kPairRouterMaxCand; i += kThreads) s_cnt[i] = 0;
    if (warp == 1) tmem_alloc_pair(smem_u32(&s_tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem = s_tmem_base;
    volatile int *abort_flag = &s_abort;
    const int ks0 = slice * a.k_steps / slices, n_steps = (slice + 1) * a.k_steps / slices - ks0;
    const bool two_hi = a.n_cols <= 128 && n_steps > 1;  // TMEM has room for two accumulators of the large products

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        const uint32_t full0 = mapa(bar_full, first);
        const int rows = a.n_cols / 2, w_row = half * rows;  // this CTA's router rows, three pieces of them
        const int ahead = min(n_steps, stages);
        // the router rows are constants: the first of them are asked for before the wait for the kernel in front
        for (int ks = 0; ks < ahead; ++ks)
            if (elect_one()) {
                if (leader) mbar_expect_tx(bar_full + 8 * ks, 2 * stage_size);  // the bytes of both CTAs
                tma_load_3d_pair(ring + ks * stage_size + kXBytes, &map_w, (ks0 + ks) * kBlockK, w_row, 0, full0 + 8 * ks);
            }
        pdl_wait();
        bool ok = true;
        uint32_t s = 0, ph = 1;
        int issued = 0;
        for (int ks = 0; ks < n_steps; ++ks, ++issued) {
            if (ks >= ahead) {
                ok = __all_sync(0xffffffffu, mbar_wait(bar_empty + 8 * s, ph, abort_flag));
                if (!ok) break;
            }
            if (elect_one()) {
                if (ks >= ahead) {
                    if (leader) mbar_expect_tx(bar_full + 8 * s, 2 * stage_size);
                    tma_load_3d_pair(ring + s * stage_size + kXBytes, &map_w, (ks0 + ks) * kBlockK, w_row, 0, full0 + 8 * s);
                }
                tma_load_2d_pair(ring + s * stage_size, &map_x, (ks0 + ks) * kBlockK, tok0, full0 + 8 * s);
            }
            __syncwarp();
            if (++s == (uint32_t)stages) { s = 0; ph ^= 1u; }
        }
        if (!ok) {
            if (lane == 0) {
                if (!*abort_flag) atomicExch(&a.meta[kMetaError], 4);
                s_abort = 1;
            }
            if (leader)  // the pair's copies in flight land before the CTAs may leave
                for (int i = max(0, issued - stages); i < issued; ++i) mbar_wait(bar_full + 8 * (i % stages), (i / stages) & 1u, abort_flag);
        }
    } else if (warp == 1 && leader) {
        // ---------------------------------------------------------------- MMA issuer
        const uint32_t idesc = instr_desc_pair(a.n_cols);
        const uint64_t a0 = smem_desc_sw128(ring), b0 = smem_desc_sw128(ring + kXBytes);
        const uint32_t piece = (uint32_t)(a.n_cols / 2) * kBlockK * 2 >> 4;  // from piece to piece (hi, mid, lo), in 16 bytes
        bool ok = true;
        uint32_t s = 0, ph = 0;
        for (int ks = 0; ks < n_steps; ++ks) {
            ok = __all_sync(0xffffffffu, mbar_wait(bar_full + 8 * s, ph, abort_flag));
            if (!ok) break;
            tc_fence_after();
            const uint64_t xa = a0 + (uint64_t)(s * (stage_size >> 4)), wb = b0 + (uint64_t)(s * (stage_size >> 4));
            const uint32_t hi = tmem + (two_hi && (ks & 1) ? kHiOddCol : 0);
            const uint32_t hi_more = ks >= (two_hi ? 2 : 1) ? 1u : 0u;
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < kBlockK / 16; ++k) {
                    umma_bf16_pair(tmem + kMidLoCol, xa + 2 * k, wb + 2 * piece + 2 * k, idesc, (ks | k) ? 1u : 0u);
                    umma_bf16_pair(tmem + kMidLoCol, xa + 2 * k, wb + piece + 2 * k, idesc, 1u);
                    umma_bf16_pair(hi, xa + 2 * k, wb + 2 * k, idesc, k ? 1u : hi_more);
                }
                commit_pair_of(bar_empty + 8 * s, first);
            }
            __syncwarp();
            if (++s == (uint32_t)stages) { s = 0; ph ^= 1u; }
        }
        if (ok) {
            if (elect_one()) commit_pair_of(bar_done, first);
            __syncwarp();
        } else if (lane == 0) {
            if (!*abort_flag) atomicExch(&a.meta[kMetaError], 5);
            s_abort = 1;
        }
    }
    // -------------------------------------------------------------------- all warps from here on
    pdl_wait();  // what is written below, calls in front may still read
    // this block's histogram: only this cluster's CTAs add to it, behind the cluster barrier
    if (a.block_hist && slice == 0 && tok0 < a.T)
        for (int e = threadIdx.x; e < a.n_real; e += kThreads) a.block_hist[(size_t)(tok0 / kSortTokens) * a.n_real + e] = 0;
    float b[RPL];
#pragma unroll
    for (int r = 0; r < RPL; ++r) b[r] = a.bias && r * 32 + lane < a.n_cand ? __ldg(a.bias + r * 32 + lane) : 0.f;
    bool ok = __all_sync(0xffffffffu, mbar_wait(bar_done, 0, abort_flag));
    if (!ok && lane == 0) {
        if (!*abort_flag) atomicExch(&a.meta[kMetaError], 6);
        s_abort = 1;
    }
    __syncwarp();
    tc_fence_after();
    // bar_done: the pair's MMAs have read their operands, so the ring may take this CTA's partial logits
    const int stride = logit_stride(a.n_cols), own_max = (kTokens + slices - 1) / slices;
    const int own0 = slice * own_max, own_n = min(own_max, kTokens - own0);  // tokens of the half tile that this CTA finishes
    if (ok) {
        // lane = token of the half tile; the four warps of a lane quarter share the columns
        const int q = warp & 3;
        float4 *dst = reinterpret_cast<float4 *>(logits + (32 * q + lane) * stride);
        const uint32_t t0 = tmem + ((uint32_t)(32 * q) << 16);
        for (int c = (warp >> 2) * 16; c < a.n_cols; c += 64) {
            uint32_t lo[16], odd[16], hi[16];
            tmem_ld16_nowait(t0 + kMidLoCol + c, lo);
            if (two_hi) tmem_ld16_nowait(t0 + kHiOddCol + c, odd);
            tmem_ld16_nowait(t0 + c, hi);
            tmem_ld_wait();
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                v[j] = __uint_as_float(lo[j]);
                if (two_hi) v[j] += __uint_as_float(odd[j]);
                v[j] += __uint_as_float(hi[j]);
            }
#pragma unroll
            for (int j = 0; j < 16; j += 4) dst[(c + j) / 4] = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
    }
    tc_fence_before();
    cluster_sync_all();  // all slices' logits are there, and the histogram's entries are cleared
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, 512);
    }
    // (where a wait gave up, the error word is set and the logits are whatever the ring held: the routing below is
    // that of other logits, but its ids, counts and positions belong together)
    float acc[RPL];
#pragma unroll
    for (int r = 0; r < RPL; ++r) acc[r] = 0.f;
    constexpr int N = kTogether;
    float part[kMaxSlices][N][RPL];  // the partial logits of the next tokens
    auto fetch = [&](int i0) {
#pragma unroll
        for (int q = 0; q < kMaxSlices; ++q) {
            if (q >= slices) break;
            const uint32_t rows = mapa(ring, 2 * q + half);
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const uint32_t row = rows + ((own0 + min(i0 + n * kWarps, own_n - 1)) * stride + lane) * 4;
#pragma unroll
                for (int r = 0; r < RPL; ++r)
                    if (r * 32 < a.n_cols) part[q][n][r] = ld_cluster_f32(row + r * 128);  // (rows have n_cols entries)
            }
        }
    };
    if (warp < own_n) fetch(warp);
    for (int i0 = warp; i0 < own_n && tok0 + own0 + i0 < a.T; i0 += N * kWarps) {
        float v[N][RPL], m[N], den[N], my_w[N];
        int my_idx[N];
#pragma unroll
        for (int n = 0; n < N; ++n)
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
                v[n][r] = b[r];
#pragma unroll
                for (int q = 0; q < kMaxSlices; ++q)
                    if (q < slices) v[n][r] += part[q][n][r];
                if (r * 32 + lane >= a.n_cand) v[n][r] = -INFINITY;
            }
        if (i0 + N * kWarps < own_n) fetch(i0 + N * kWarps);
        topk_gate_select<RPL, N, STATS>(v, a.n_real, a.n_cand, a.K, a.gate_mode, lane, m, den, my_idx, my_w);
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const int i = i0 + n * kWarps, t = tok0 + own0 + i;
            if (i >= own_n || t >= a.T) break;
            if (lane < a.K) {
                a.topk_idx[(size_t)t * a.K + lane] = my_idx[n];
                a.topk_w[(size_t)t * a.K + lane] = my_w[n];
                if (a.block_hist && (unsigned)my_idx[n] < (unsigned)a.n_real)
                    atomicAdd(a.block_hist + (size_t)(tok0 / kSortTokens) * a.n_real + my_idx[n], 1);
                if (STATS) atomicAdd(s_cnt + my_idx[n], 1);
            }
            if constexpr (STATS) {
#pragma unroll
                for (int r = 0; r < RPL; ++r)
                    if (r * 32 + lane < a.n_cand) acc[r] += expf(v[n][r] - m[n]) / den[n];
            }
        }
    }
    if constexpr (STATS) {
        // the warps' sums behind the logits in the ring, then added in warp order
        float *sums = logits + kTokens * stride;
#pragma unroll
        for (int r = 0; r < RPL; ++r)
            if (r * 32 + lane < a.n_cand) sums[warp * a.n_cand + r * 32 + lane] = acc[r];
        __syncthreads();
        float *cta_sums = a.stat_part + (size_t)((tile * 2 + half) * slices + slice) * 2 * a.n_cand;
        for (int j = threadIdx.x; j < a.n_cand; j += kThreads) {
            float p = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) p += sums[w * a.n_cand + j];
            cta_sums[j] = (float)s_cnt[j];
            cta_sums[a.n_cand + j] = p;
        }
    }
    __syncwarp();
    if (slices > 1) cluster_sync_all();  // no CTA leaves while another may still read its logits
}

constexpr int kSmemBytes = kRingBytes + 1024;
// the partial logits and the sums of the statistics fit the ring
constexpr bool logits_fit(int n_cols) {
    return (kTokens * logit_stride(n_cols) + kWarps * n_cols) * 4 <= ring_stages(n_cols) * stage_bytes(n_cols) && ring_stages(n_cols) >= 2;
}
static_assert(kTokens == kSortTokens, "a CTA's tokens are a block of the counting sort");
static_assert(logits_fit(32) && logits_fit(96) && logits_fit(128) && logits_fit(160) && logits_fit(192) && logits_fit(224) && logits_fit(256),
              "the ring is too small for the partial logits");

template <int RPL>
bool prepare_one() {
    for (auto k : {router_topk_pair_kernel<RPL, false>, router_topk_pair_kernel<RPL, true>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) return false;
    return true;
}

// cluster launch of `grid` CTAs in clusters of `cluster`; with max_clusters only how many of them fit the GPU
template <typename K>
cudaError_t launch_clusters(bool pdl, K kernel, int grid, int cluster, cudaStream_t s, const CUtensorMap &mw, const CUtensorMap &mx,
                            const PairRouterArgs &a, int *max_clusters = nullptr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 2 : 1;
    if (max_clusters) {
        cfg.numAttrs = 1;
        return cudaOccupancyMaxActiveClusters(max_clusters, kernel, &cfg);
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, mw, mx, a);
    if (e != cudaSuccess) note_launch_error(e);
    return e;
}

}  // namespace

int init_router_pair(zeda_moe *h) {
    const zeda_moe_config_t &c = h->cfg;
    const int n_cand = c.n_real + c.n_zero;
    if (n_cand > kPairRouterMaxCand || c.max_tokens < kPairRouterTokens) return 0;
    PairRouterMaps *rm = static_cast<PairRouterMaps *>(aligned_alloc(64, (sizeof(PairRouterMaps) + 63) / 64 * 64));
    if (!rm) { set_error("out of host memory"); return -1; }
    rm->n_cols = (n_cand + 31) / 32 * 32;
    const int nc_pad = router_split_pad(n_cand);
    const cuuint64_t dims[3] = {(cuuint64_t)c.d_model, (cuuint64_t)nc_pad, 3};
    const cuuint64_t strides[2] = {(cuuint64_t)c.d_model * 2, (cuuint64_t)nc_pad * c.d_model * 2};
    const cuuint32_t box[3] = {kBlockK, (cuuint32_t)rm->n_cols / 2, 3};
    bool ok = encode_bf16_map(&rm->w_split, h->ws.router_split, 3, dims, strides, box);
    ok = ok && prepare_one<2>() && prepare_one<4>() && prepare_one<6>() && prepare_one<8>();
    rm->max_clusters[0] = 0;
    for (int s = 1; s <= kMaxSlices && ok; ++s) {
        int n = 0;
        // (a cluster size that the GPU cannot place at all counts as none)
        if (launch_clusters(false, router_topk_pair_kernel<8, true>, 2 * s, 2 * s, nullptr, rm->w_split, rm->w_split, PairRouterArgs{}, &n) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        rm->max_clusters[s] = n;
    }
    if (!ok) { free(rm); return -1; }
    h->pair_router = rm;
    return 0;
}

// As many slices as the clusters of all tiles are resident with at a time.
int pair_router_slices(const zeda_moe *h, int T) {
    const PairRouterMaps *rm = static_cast<const PairRouterMaps *>(h->pair_router);
    const int tiles = (T + 2 * kTokens - 1) / (2 * kTokens), k_steps = h->cfg.d_model / kBlockK;
    int s = kMaxSlices;
    while (s > 1 && (s > k_steps || tiles > rm->max_clusters[s] || 2 * s * tiles > kPairRouterMaxSliced)) --s;
    return s;
}

// What this kernel saves over the candidate-major router with a top-K pass behind it, in us, from the shape of the
// call.  Both go in waves: there of (128 tokens x 128 candidates) items over the SMs, here of clusters.  Fitted to the
// routing pass both ways at 2,197 shapes (4096 to 65,536 tokens, d 256 to 8192, 16 to 256 candidates, K 2 to 16); us,
// there and here, d 2048 and K 8:
//    96 candidates   T=4096 22.2, 19.4   T=8448 30.9, 23.3   T=8449 31.0, 33.4 (one slice)   T=9473 37.4, 33.2
//   128              T=4096 22.6, 21.8   T=8448 32.3, 26.5   T=8449 32.3, 37.9   T=12288 42.6, 38.9   T=20000 71.7, 72.7
//   192              T=4096 27.4, 27.0   T=8448 39.2, 33.8   T=8449 39.2, 47.3   T=9473 55.9, 47.1    T=20000 93.2, 92.5
//   256              T=4096 29.4, 33.4   T=4737 36.3, 34.7   T=8449 43.7, 59.8   T=9473 61.7, 59.7    T=20000 102.9, 117.6
double pair_router_saves_us(const zeda_moe *h, int T) {
    const PairRouterMaps *rm = static_cast<const PairRouterMaps *>(h->pair_router);
    const int n_cand = h->cfg.n_real + h->cfg.n_zero;
    const double k_steps = h->cfg.d_model / kBlockK, K = h->cfg.top_k;
    const int items = (T + 127) / 128 * ((n_cand + 127) / 128), split = router_split_factor(h, T);
    const int waves_there = (items * split + h->sm_count - 1) / h->sm_count;
    const double topk_there = 0.001 * T * (0.12 + 0.029 * K) + 3.7;  // with its launch
    const double there = waves_there * (0.33 * k_steps / split + 7.2) + topk_there;
    const int slices = pair_router_slices(h, T), tiles = (T + 2 * kTokens - 1) / (2 * kTokens), fit = rm->max_clusters[slices];
    const int waves = fit > 0 ? (tiles + fit - 1) / fit : tiles;
    const int turns = ((kTokens + slices - 1) / slices + kTogether * kWarps - 1) / (kTogether * kWarps);  // of a warp's tokens
    const double topk = turns * (0.39 + 0.126 * K + 0.66 * ((n_cand + 63) / 64));
    return there - waves * (0.00167 * rm->n_cols * k_steps / slices + 5.9 + topk);
}

// Where it saves anything, and 2 us in two ranges where the fit is that far off.  Of the 1,568 shapes that this sends
// here 22 are more than 2 % slower than there (11 % at most, 5632 tokens of many candidates and short rows), of the others
// 93 would be more than 4 % faster here.
bool pair_router_path(const zeda_moe *h, int T) {
    if (!h->pair_router || T < kPairRouterTokens) return false;
    const int n_cand = h->cfg.n_real + h->cfg.n_zero;
    const bool margin = (pair_router_slices(h, T) == 1 && n_cand <= 64) || (h->cfg.d_model < 2048 && n_cand > 128);
    return pair_router_saves_us(h, T) > (margin ? 2.0 : 0.0);
}

int pair_router_stat_blocks(const zeda_moe *h, int T) { return (T + 2 * kTokens - 1) / (2 * kTokens) * 2 * pair_router_slices(h, T); }

int launch_router_topk_pair(const zeda_moe *h, const __nv_bfloat16 *x, int T, int split_T, int32_t *block_hist, float *stat_part,
                            cudaStream_t s) {
    const zeda_moe_config_t &c = h->cfg;
    const PairRouterMaps *rm = static_cast<const PairRouterMaps *>(h->pair_router);
    const int n_cand = c.n_real + c.n_zero, slices = pair_router_slices(h, split_T > T ? split_T : T);
    CUtensorMap map_x;
    const cuuint64_t dims[2] = {(cuuint64_t)c.d_model, (cuuint64_t)T};
    const cuuint64_t strides[1] = {(cuuint64_t)c.d_model * 2};
    const cuuint32_t box[2] = {kBlockK, kTokens};
    if (!encode_bf16_map(&map_x, x, 2, dims, strides, box)) return -1;
    const PairRouterArgs a = {h->router_bias, T, (int)c.n_real, n_cand, rm->n_cols, (int)c.d_model / kBlockK, slices, (int)c.top_k,
                              (int)c.gate_mode, h->ws.topk_idx, h->ws.topk_w, block_hist, stat_part, h->ws.meta};
    const int grid = (T + 2 * kTokens - 1) / (2 * kTokens) * 2 * slices;
    cudaError_t e = cudaSuccess;
    auto go = [&](auto plain, auto stats) {
        e = launch_clusters(h->pdl, stat_part ? stats : plain, grid, 2 * slices, s, rm->w_split, map_x, a);
    };
    if (n_cand <= 64) go(router_topk_pair_kernel<2, false>, router_topk_pair_kernel<2, true>);
    else if (n_cand <= 128) go(router_topk_pair_kernel<4, false>, router_topk_pair_kernel<4, true>);
    else if (n_cand <= 192) go(router_topk_pair_kernel<6, false>, router_topk_pair_kernel<6, true>);
    else go(router_topk_pair_kernel<8, false>, router_topk_pair_kernel<8, true>);
    return e == cudaSuccess ? 1 : -1;
}

}  // namespace zeda
