// Expert kernels for the smallest batches (a few decoding sequences): weight streams without a ring.
//
// With T tokens a call reads at most T * K experts, each for one or a few pair rows: 2 x 6.3 + 3.1 MB
// of weights per active expert at d = 2048, H_e = 768 and next to no arithmetic.  What bounds such a
// call is how evenly that read spreads over the SMs and how long the chain of dependent steps is.  The
// tensor-memory kernels of expert_pair.cu hand out work in items of 256 or 512 weight rows (one token:
// 12 items for 74 CTA pairs), so here the work is cut into blocks of 16 weight rows, the M of the
// warp-level MMA, and the weights go from global memory straight into its A fragments.
//
// Fragment trick: the sum over k may be taken in any order, so lane (g, t) of a warp reads 16
// consecutive bytes of weight row g (k = 32 b + 8 t ..) as the A operands of two m16n8k16 MMAs and the
// same 16 bytes of the pair row of column g as their B operands.  Every load is a full 16 bytes, four
// lanes cover 64 consecutive bytes of a row, and nothing goes through shared memory.
#include <algorithm>
#include <cmath>

#include "route_token.cuh"

namespace zeda {

namespace {

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 32 k of 16 weight rows (lo: row g, hi: row g + 8 of the fragment) times 8 pair rows
__device__ __forceinline__ void mma_block(float (&c)[4], const uint4 &lo, const uint4 &hi, const uint4 &b) {
    mma_bf16(c, lo.x, hi.x, lo.y, hi.y, b.x, b.y);
    mma_bf16(c, lo.z, hi.z, lo.w, hi.w, b.z, b.w);
}

// weights are read once per call: past L1
__device__ __forceinline__ uint4 ld_weights(const __nv_bfloat16 *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// activations come from the kernel before: straight from L2
__device__ __forceinline__ uint4 ld_rows(const __nv_bfloat16 *p) { return __ldcg(reinterpret_cast<const uint4 *>(p)); }

__device__ __forceinline__ float ld_value(const __nv_bfloat16 *p) {
    return __uint_as_float((uint32_t)__ldcg(reinterpret_cast<const unsigned short *>(p)) << 16);
}

constexpr uint4 kZero4 = {0u, 0u, 0u, 0u};
static_assert(kStreamTokens <= 16, "the kernels are instantiated for up to two column tiles of 8 pair rows");

// The routing results of the call in shared memory.  One tile of the tile list per active expert: an
// expert has at most one pair per token, and T <= kStreamTokens is below every tile height.
template <int SLOTS>
struct RouteTables {
    int32_t expert[SLOTS];  // active experts in id order
    int32_t off[kMaxCand + 1];
    int32_t inv[SLOTS], tok[SLOTS], idx[SLOTS];  // of the slot: position, candidate; of the position: token
    float w[SLOTS];
    int32_t n_tiles;
    uint32_t mask[kMaxCand];      // tokens that selected the expert
    int4 chunk[kMaxCand / 32];    // per 32 experts: pairs, active experts, most pairs of one expert
};

struct RouteArgs {  // the routing pass' buffers in the workspace
    const float *logits;
    int32_t *topk_idx;
    float *topk_w;
    int32_t *inv, *perm, *pair_token, *counts, *offsets, *tile_expert, *tile_row0, *meta;
    int T, K, n_real, n_cand, gate_mode;
};

// Loads what the routing pass left, by independent loads (one round trip).
template <int SLOTS>
__device__ __forceinline__ void load_route_tables(RouteTables<SLOTS> &rt, const RouteArgs &ra) {
    const int slots = ra.T * ra.K;
    for (int i = threadIdx.x; i < slots; i += blockDim.x) {
        if (i < ra.n_real) rt.expert[i] = __ldcg(ra.tile_expert + i);
        rt.inv[i] = __ldcg(ra.inv + i);
        rt.tok[i] = __ldcg(ra.pair_token + i);
        rt.w[i] = __ldcg(ra.topk_w + i);
    }
    for (int i = threadIdx.x; i <= ra.n_real; i += blockDim.x) rt.off[i] = __ldcg(ra.offsets + i);
    if (threadIdx.x == blockDim.x - 1) rt.n_tiles = __ldcg(ra.meta + kMetaPairTiles);
    __syncthreads();
}

// Up to kRouteHereTokens tokens every gate/up CTA routes them itself, from the logits: one warp per token (no loop: with
// sixteen logits a lane it spilled) and a scan over bit masks take no longer than a routing kernel in front, and the call
// has one kernel fewer in its chain (one token: 24.9 -> 15.7 us a call back to back, 8 tokens: 53.7 -> 52.7).  All CTAs
// arrive at the same tables.
constexpr int kRouteHereTokens = 8;

template <int RPL, int SLOTS>
__device__ __forceinline__ void route_here(RouteTables<SLOTS> &rt, const RouteArgs &ra) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    const int n_chunks = (ra.n_real + 31) / 32;
    if (const int t = warp; t < ra.T) {
        int my_idx;
        float my_w, v[RPL], m, den;
        topk_gate_token<RPL>(ra.logits + (size_t)t * ra.n_cand, 1, 0, ra.n_real, ra.n_cand, ra.K, ra.gate_mode, lane, v, m, den, my_idx, my_w);
        if (lane < ra.K) {
            rt.idx[t * ra.K + lane] = my_idx;
            rt.w[t * ra.K + lane] = my_w;
            if (my_idx < ra.n_real) atomicOr(rt.mask + my_idx, 1u << t);
        }
    }
    __syncthreads();
    for (int ch = warp; ch < n_chunks; ch += n_warps) {
        const int i = 32 * ch + lane, c = i < ra.n_real ? __popc(rt.mask[i]) : 0;
        int sum = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(kFull, sum, o);
            if (lane >= o) sum += a;
        }
        if (i < ra.n_real) rt.off[i] = sum - c;
        const unsigned act = __ballot_sync(kFull, c > 0);
        const int mx = __reduce_max_sync(kFull, c);
        if (lane == 31) rt.chunk[ch] = make_int4(sum, __popc(act), mx, 0);
    }
    __syncthreads();
    for (int ch = warp; ch <= n_chunks; ch += n_warps) {  // one turn more: the totals
        int off = 0, tiles = 0;
        for (int q = 0; q < ch; ++q) { off += rt.chunk[q].x; tiles += rt.chunk[q].y; }
        if (ch == n_chunks) {
            if (lane == 0) { rt.off[ra.n_real] = off; rt.n_tiles = tiles; }
            break;
        }
        const int i = 32 * ch + lane;
        const bool active = i < ra.n_real && rt.mask[i];
        const unsigned act = __ballot_sync(kFull, active);
        if (i < ra.n_real) rt.off[i] += off;
        if (active) rt.expert[tiles + __popc(act & ((1u << lane) - 1u))] = i;
    }
    __syncthreads();
    for (int s = threadIdx.x; s < ra.T * ra.K; s += blockDim.x) {
        const int e = rt.idx[s], t = s / ra.K;
        int p = -1;
        if (e < ra.n_real) {
            p = rt.off[e] + __popc(rt.mask[e] & ((1u << t) - 1u));
            rt.tok[p] = t;
        }
        rt.inv[s] = p;
    }
    __syncthreads();
}

// The same for one token, as far as gate/up reads it: the active experts, their positions and the token.  A warp has the
// whole choice in its lanes, so the scan over bit masks and all but one of the barriers drop out, and the weights, which
// only the down kernel needs, are left to the CTA that publishes the tables.
template <int RPL, int SLOTS>
__device__ __forceinline__ void route_one_token(RouteTables<SLOTS> &rt, const RouteArgs &ra) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int my_idx;
        float my_w, v[RPL], m, den;
        topk_gate_token<RPL>(ra.logits, 1, 0, ra.n_real, ra.n_cand, ra.K, ZEDA_GATE_TOPK_NORM, lane, v, m, den, my_idx, my_w);
        const bool real = lane < ra.K && my_idx < ra.n_real;
        const int id = real ? my_idx : kMaxCand;
        int pos = 0;
#pragma unroll
        for (int k = 0; k < kMaxTopK; ++k) pos += __shfl_sync(kFull, id, k) < id ? 1 : 0;  // (slots beyond K hold no expert)
        if (real) {
            rt.expert[pos] = id;
            rt.off[id] = pos;
            rt.off[id + 1] = pos + 1;  // (the next expert's too, if it is active)
            rt.tok[pos] = 0;
        }
        const int n = __popc(__ballot_sync(kFull, real));
        if (lane == 0) rt.n_tiles = n;
    }
    __syncthreads();
}

// What the routing pass leaves in the workspace, by one CTA; then the flag that says so.
template <int SLOTS>
__device__ __forceinline__ void publish_route(const RouteTables<SLOTS> &rt, const RouteArgs &ra) {
    const int slots = ra.T * ra.K;
    for (int s = threadIdx.x; s < slots; s += blockDim.x) {
        const int p = rt.inv[s];
        ra.topk_idx[s] = rt.idx[s];
        ra.topk_w[s] = rt.w[s];
        ra.inv[s] = p;
        if (p >= 0) {
            ra.perm[p] = s;
            ra.pair_token[p] = s / ra.K;
        }
    }
    for (int i = threadIdx.x; i <= ra.n_real; i += blockDim.x) {
        ra.offsets[i] = rt.off[i];
        if (i < ra.n_real) ra.counts[i] = rt.off[i + 1] - rt.off[i];
    }
    for (int i = threadIdx.x; i < rt.n_tiles; i += blockDim.x) {
        ra.tile_expert[i] = rt.expert[i];
        ra.tile_row0[i] = 0;
    }
    if (threadIdx.x == 0) {
        int mx = 0;
        for (int q = 0; q < (ra.n_real + 31) / 32; ++q) mx = max(mx, rt.chunk[q].z);
        const int pairs = rt.off[ra.n_real];
        ra.meta[kMetaPairs] = pairs;
        ra.meta[kMetaActive] = rt.n_tiles;
        ra.meta[kMetaZeroSlots] = slots - pairs;
        ra.meta[kMetaPairTiles] = rt.n_tiles;
        ra.meta[kMetaMaxRows] = mx;
    }
    __syncthreads();  // the CTA's stores come before the release that follows it
    if (threadIdx.x == 0) asm volatile("st.release.gpu.global.s32 [%0], 1;" ::"l"(ra.meta + kMetaRouted) : "memory");
}

// Whether the tables above are there, for one thread of a CTA to ask; the barrier behind it passes its acquire on to the
// others (each asking for itself takes 0.2 us longer).
__device__ __forceinline__ bool route_published(const RouteArgs &ra) {
    int32_t v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(ra.meta + kMetaRouted) : "memory");
    return v != 0;
}

// RPL > 0: route here, with that many logits per lane; RPL = 0: another kernel has.
template <int RPL>
constexpr int kTableSlots = RPL > 0 ? kRouteHereTokens * kMaxTopK : kStreamSlots;

// GEMM1 + SwiGLU.  Unit = (active expert, 8 features): rows g of the fragment are the 8 gate rows, rows
// g + 8 the 8 up rows, so a lane's accumulators hold gate and up of the same feature and pair and
// SwiGLU needs no exchange.  The eight warps of a CTA split the reduction axis; their partial sums meet
// in shared memory (double-buffered: one barrier per unit), added in warp order.  The next unit's
// weights are requested before the current one is reduced.
constexpr int kUpWarps = 8;
constexpr int kUpChunk = 4;  // 32-k blocks a warp keeps in flight: 4 x (2 x 512 B of weights)

template <int NT, int RPL>
__global__ void __launch_bounds__(32 * kUpWarps, NT == 1 ? 3 : 2)
stream_gate_up_kernel(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ w, const RouteArgs ra, int d, int He,
                      __nv_bfloat16 *__restrict__ hmid) {
    __shared__ RouteTables<kTableSlots<RPL>> rt;
    __shared__ float part[2][kUpWarps][NT][4][32];
    if constexpr (RPL > 0) {
        for (int i = threadIdx.x; i < ra.n_real; i += blockDim.x) rt.mask[i] = 0u;
        __syncthreads();
    }
    pdl_wait();
    pdl_launch_dependents();  // only now: the down kernel reads the logits or the routing results before its own wait
    if constexpr (RPL > 0) {
        const bool publish = blockIdx.x == gridDim.x - 1;  // the CTA with the fewest units
        if (ra.T == 1 && !publish) route_one_token<RPL>(rt, ra);
        else route_here<RPL>(rt, ra);
        if (publish) publish_route(rt, ra);
    } else {
        load_route_tables(rt, ra);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int groups = He / 8, units = rt.n_tiles * groups;
    const int kblocks = d / 32, batches = (kblocks + kUpWarps * kUpChunk - 1) / (kUpWarps * kUpChunk);
    uint4 wg[kUpChunk], wu[kUpChunk], xb[kUpChunk];
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[nt][c] = 0.f;
    auto row_of = [&](int pos0, int n, int col) -> const __nv_bfloat16 * {
        return col < n ? x + (size_t)rt.tok[pos0 + col] * d : nullptr;
    };
    auto fetch = [&](int u, int batch) {
        const int e = rt.expert[u / groups], f0 = (u % groups) * 8;
        const __nv_bfloat16 *gate = w + ((size_t)e * 2 * He + f0 + g) * d, *up = gate + (size_t)He * d;
        const __nv_bfloat16 *row = row_of(rt.off[e], rt.off[e + 1] - rt.off[e], g);
#pragma unroll
        for (int i = 0; i < kUpChunk; ++i) {
            const int b = (batch * kUpWarps + warp) * kUpChunk + i, k = b * 32 + t * 8;
            const bool in = b < kblocks;
            wg[i] = in ? ld_weights(gate + k) : kZero4;
            wu[i] = in ? ld_weights(up + k) : kZero4;
            xb[i] = in && row ? ld_rows(row + k) : kZero4;
        }
    };
    int u = blockIdx.x, batch = 0, buf = 0;
    if (u < units) fetch(u, 0);
    while (u < units) {
        const int e = rt.expert[u / groups], f0 = (u % groups) * 8, pos0 = rt.off[e], n = rt.off[e + 1] - pos0;
        const bool last = batch + 1 == batches;
#pragma unroll
        for (int i = 0; i < kUpChunk; ++i) mma_block(acc[0], wg[i], wu[i], xb[i]);
#pragma unroll
        for (int nt = 1; nt < NT; ++nt) {
            if (8 * nt >= n) break;  // (uniform over the CTA)
            const __nv_bfloat16 *row = row_of(pos0, n, 8 * nt + g);
            uint4 xc[kUpChunk];
#pragma unroll
            for (int i = 0; i < kUpChunk; ++i) {
                const int b = (batch * kUpWarps + warp) * kUpChunk + i;
                xc[i] = b < kblocks && row ? ld_rows(row + b * 32 + t * 8) : kZero4;
            }
#pragma unroll
            for (int i = 0; i < kUpChunk; ++i) mma_block(acc[nt], wg[i], wu[i], xc[i]);
        }
        const int nu = last ? u + gridDim.x : u, nb = last ? 0 : batch + 1;
        if (nu < units) fetch(nu, nb);
        if (last) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (8 * nt < n) part[buf][warp][nt][c][lane] = acc[nt][c];
                    acc[nt][c] = 0.f;
                }
            __syncthreads();
            if (threadIdx.x < 64 * NT) {
                const int nt = threadIdx.x >> 6, j = (threadIdx.x >> 5) & 1, col = 8 * nt + 2 * t + j;
                if (col < n) {
                    float gs = 0.f, us = 0.f;
#pragma unroll
                    for (int q = 0; q < kUpWarps; ++q) { gs += part[buf][q][nt][j][lane]; us += part[buf][q][nt][2 + j][lane]; }
                    hmid[(size_t)(pos0 + col) * He + f0 + g] = __float2bfloat16_rn(swiglu(gs, us));
                }
            }
            buf ^= 1;
        }
        u = nu;
        batch = nb;
    }
}

// GEMM2 with the weighted combine of Eq. 1: CTA b owns output features [16 b, 16 b + 16) of every token
// and walks all active experts, so the sum over a token's slots never leaves the CTA.  Sixteen warps:
// four experts at a time, four slices of the reduction axis; each warp keeps its partial sums of every
// pair in shared memory and no barrier stands in the stream.  W_down does not depend on GEMM1: the
// first weights are requested before the wait for it.  At the end the slices are added in order, each
// expert output is rounded to bf16 (as the other expert kernels store it) and the token's slots are
// summed in slot order in fp32.
// resid given: r <- bf16(r + bf16(y)) in place of storing y.
// Up to kRouteHereTokens tokens the routing is gate/up's: it has left its tables long before its last CTAs leave the SMs
// to these, and fetching them takes 1 us where routing takes 3 (us for four layers, routing here and fetching: 1 token
// 81.9, 77.0; 2 tokens 109.2, 104.1; 4 tokens 151.0, 146.3; 8 tokens 224.8, 220.3).  A CTA that is here before them does
// not wait: it routes for itself and arrives at the same tables.  That is nearly every CTA where gate/up's have little to
// do (no pair at all, or H_e 128), for the price of the look at the flag, at most 1 % of such a call.
constexpr int kDownWarps = 16, kDownSlices = 4, kDownExperts = kDownWarps / kDownSlices;
static_assert(kUpWarps >= kRouteHereTokens && kDownWarps >= kRouteHereTokens, "a warp per token");
constexpr int kDownChunk = 6;
constexpr int kDownStride = 20;  // floats per pair and slice: 16 features; 20 keeps the fragment stores free of bank conflicts

template <int NT, int RPL>
__global__ void __launch_bounds__(32 * kDownWarps, 1)
stream_down_combine_kernel(const __nv_bfloat16 *__restrict__ hmid, const __nv_bfloat16 *__restrict__ w, const RouteArgs ra,
                           const __nv_bfloat16 *__restrict__ x, int d, int He, int copy_experts, __nv_bfloat16 *__restrict__ y,
                           __nv_bfloat16 *__restrict__ resid) {
    __shared__ RouteTables<kTableSlots<RPL>> rt;
    extern __shared__ float part[];  // [kDownSlices][slots][kDownStride]
    pdl_launch_dependents();
    const int T = ra.T, K = ra.K, slots = T * K;
    if constexpr (RPL > 0) {
        for (int i = threadIdx.x; i < ra.n_real; i += blockDim.x) rt.mask[i] = 0u;
        if (__syncthreads_or(threadIdx.x == 0 && route_published(ra))) load_route_tables(rt, ra);
        else route_here<RPL>(rt, ra);
    } else {
        load_route_tables(rt, ra);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int slice = warp % kDownSlices, m0 = blockIdx.x * 16;
    const int kblocks = He / 32, batches = (kblocks + kDownSlices * kDownChunk - 1) / (kDownSlices * kDownChunk);
    const int n_tiles = rt.n_tiles;
    uint4 lo[kDownChunk], hi[kDownChunk], hb[kDownChunk];
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[nt][c] = 0.f;
    auto fetch_w = [&](int tile, int batch) {
        const __nv_bfloat16 *row = w + ((size_t)rt.expert[tile] * d + m0 + g) * He;
#pragma unroll
        for (int i = 0; i < kDownChunk; ++i) {
            const int b = (batch * kDownSlices + slice) * kDownChunk + i, k = b * 32 + t * 8;
            const bool in = b < kblocks;
            lo[i] = in ? ld_weights(row + k) : kZero4;
            hi[i] = in ? ld_weights(row + (size_t)8 * He + k) : kZero4;
        }
    };
    auto fetch_h = [&](uint4 (&v)[kDownChunk], int tile, int batch, int col) {
        const int e = rt.expert[tile], pos0 = rt.off[e];
        const bool has = pos0 + col < rt.off[e + 1];
        const __nv_bfloat16 *row = hmid + (size_t)(pos0 + col) * He;
#pragma unroll
        for (int i = 0; i < kDownChunk; ++i) {
            const int b = (batch * kDownSlices + slice) * kDownChunk + i;
            v[i] = has && b < kblocks ? ld_rows(row + b * 32 + t * 8) : kZero4;
        }
    };
    int tile = warp / kDownSlices, batch = 0;
    if (tile < n_tiles) fetch_w(tile, 0);
    pdl_wait();  // hmid is GEMM1's output
    if (tile < n_tiles) fetch_h(hb, tile, 0, g);
    while (tile < n_tiles) {
        const int e = rt.expert[tile], pos0 = rt.off[e], n = rt.off[e + 1] - pos0;
        const bool last = batch + 1 == batches;
#pragma unroll
        for (int i = 0; i < kDownChunk; ++i) mma_block(acc[0], lo[i], hi[i], hb[i]);
#pragma unroll
        for (int nt = 1; nt < NT; ++nt) {
            if (8 * nt >= n) break;  // (uniform over the warp)
            uint4 hc[kDownChunk];
            fetch_h(hc, tile, batch, 8 * nt + g);
#pragma unroll
            for (int i = 0; i < kDownChunk; ++i) mma_block(acc[nt], lo[i], hi[i], hc[i]);
        }
        const int ntile = last ? tile + kDownExperts : tile, nb = last ? 0 : batch + 1;
        if (ntile < n_tiles) { fetch_w(ntile, nb); fetch_h(hb, ntile, nb, g); }
        if (last) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float *p = part + ((size_t)slice * slots + pos0 + 8 * nt + 2 * t) * kDownStride;
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    if (8 * nt + 2 * t + j < n) {
                        p[j * kDownStride + g] = acc[nt][j];
                        p[j * kDownStride + g + 8] = acc[nt][2 + j];
                    }
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[nt][c] = 0.f;
            }
        }
        tile = ntile;
        batch = nb;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < T * 16; i += blockDim.x) {
        const int tok = i >> 4, f = i & 15;
        const size_t at = (size_t)tok * d + m0 + f;
        float sum = 0.f, zero_mass = 0.f;
        for (int k = 0; k < K; ++k) {
            const int pos = rt.inv[tok * K + k];
            const float wk = rt.w[tok * K + k];
            if (pos < 0) { zero_mass += wk; continue; }
            float o = 0.f;
#pragma unroll
            for (int q = 0; q < kDownSlices; ++q) o += part[((size_t)q * slots + pos) * kDownStride + f];
            sum = fmaf(wk, __bfloat162float(__float2bfloat16_rn(o)), sum);
        }
        if (copy_experts && zero_mass != 0.f) sum = fmaf(zero_mass, ld_value(x + at), sum);
        const __nv_bfloat16 out = __float2bfloat16_rn(sum);
        if (resid) resid[at] = __float2bfloat16_rn(ld_value(resid + at) + __bfloat162float(out));
        else y[at] = out;
    }
}

int down_smem_bytes(int slots) { return kDownSlices * slots * kDownStride * (int)sizeof(float); }

// What these kernels take longer than those of expert_pair.cu, in us, from the shape of the call.  They save the
// longer chain and the launches of the others, about 12 us a call, and they lose per active expert where the
// down projection leaves SMs idle (d / 16 CTAs, one per SM) or spends more on an expert's start than on its
// weights.  Measured both ways at 168 shapes (d 256 to 8192, H_e 128 to 4096, 8 to 256 experts, K 2 to 16, with no
// zero experts or one for two others) of 1 to 16 tokens, us a call back to back, these kernels and the others:
//   d 2048, H_e 768, N 128 + 64, K 8   T=1 16.6, 29.6   T=8 72.2, 84.7   T=16 101.5, 106.7
//   d 1024, H_e 256, N 256, K 16       T=1 20.7, 28.2   T=4 44.6, 39.8   T=8 70.1, 52.7
//   d 8192, H_e 4096, N 8, K 2         T=1 97.9, 101    T=2 155, 175     T=8 278, 268
// Of the 774 calls that the rule sends here 7 are more than 3 % slower and none more than 7 %.
double stream_excess_us(const zeda_moe *h, int T) {
    const zeda_moe_config_t &c = h->cfg;
    const double d = c.d_model, He = c.d_expert;
    // experts with a pair if all candidates are as likely (the host does not know the load)
    const double active = c.n_real * (1.0 - std::pow(1.0 - (double)c.top_k / (c.n_real + c.n_zero), T));
    // down kernel: waves of CTAs, each of which takes 0.3 us to start on an expert or 45 GB/s for its 16 weight rows
    const int ctas = c.d_model / 16, waves = (ctas + h->sm_count - 1) / h->sm_count;
    const double down = active * waves * std::max(0.3, 0.0007 * He);
    // there: 6 TB/s, or one work item of 256 rows per CTA pair at 114 GB/s
    const double down_pair = std::max(active * 2.0 * d * He / 6e6, 0.0045 * He);
    // both projections stream a little slower, with two column tiles (above 8 tokens) a little more: us per MB
    const double stream = (T > 8 ? 0.012 : 0.005) * active * 6.0 * d * He * 1e-6;
    return down - down_pair + stream;
}
constexpr double kStreamSavedUs = 9.0;  // (of the 12, so that the rule errs on the side of the other kernels)

}  // namespace

bool stream_path(const zeda_moe *h, int T) {
    return h->cfg.ep_size < 1 && T <= kStreamTokens && stream_excess_us(h, T) <= kStreamSavedUs;
}

bool stream_routes_itself(const zeda_moe *h, int T) { return stream_path(h, T) && T <= kRouteHereTokens; }

namespace {

RouteArgs route_args(const zeda_moe *h, int T) {
    const zeda_moe_config_t &c = h->cfg;
    const Workspace &ws = h->ws;
    return {ws.logits, ws.topk_idx, ws.topk_w, ws.inv, ws.perm, ws.pair_token, ws.counts, ws.offsets, ws.ptile_expert, ws.ptile_row0,
            ws.meta, T, c.top_k, c.n_real, c.n_real + c.n_zero, c.gate_mode};
}

template <int NT, int RPL>
int launch_gate_up(const zeda_moe *h, const __nv_bfloat16 *x, int T, cudaStream_t s) {
    const zeda_moe_config_t &c = h->cfg;
    const int slots = T * c.top_k, per_sm = NT == 1 ? 3 : 2;
    const int units = (slots < c.n_real ? slots : c.n_real) * (c.d_expert / 8);
    const int grid = units < per_sm * h->sm_count ? units : per_sm * h->sm_count;
    const cudaError_t e = launch_kernel(h->pdl, stream_gate_up_kernel<NT, RPL>, dim3(grid), dim3(32 * kUpWarps), 0, s, x, h->w_gate_up,
                                        route_args(h, T), (int)c.d_model, (int)c.d_expert, h->ws.hmid);
    return e == cudaSuccess ? 1 : -1;
}

template <int NT, int RPL>
int launch_down(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y, __nv_bfloat16 *resid, cudaStream_t s) {
    const zeda_moe_config_t &c = h->cfg;
    const cudaError_t e = launch_kernel(h->pdl, stream_down_combine_kernel<NT, RPL>, dim3(c.d_model / 16), dim3(32 * kDownWarps),
                                        down_smem_bytes(T * c.top_k), s, (const __nv_bfloat16 *)h->ws.hmid, h->w_down, route_args(h, T), x,
                                        (int)c.d_model, (int)c.d_expert, (int)(c.expert_kind == ZEDA_EXPERT_COPY), y, resid);
    return e == cudaSuccess ? 1 : -1;
}

template <int NT, int RPL>
bool prepare_down() {
    return cudaFuncSetAttribute(stream_down_combine_kernel<NT, RPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                down_smem_bytes(kTableSlots<RPL>)) == cudaSuccess;
}

}  // namespace

int init_stream_kernels() {
    const bool ok = prepare_down<1, 2>() && prepare_down<1, 4>() && prepare_down<1, 6>() && prepare_down<1, 8>() &&
                    prepare_down<1, 16>() && prepare_down<2, 0>();
    return ok ? 0 : -1;
}

int launch_stream_gemm1(const zeda_moe *h, const __nv_bfloat16 *x, int T, cudaStream_t s) {
    const int n_cand = h->cfg.n_real + h->cfg.n_zero;
    if (!stream_routes_itself(h, T)) return launch_gate_up<2, 0>(h, x, T, s);
#define ZEDA_CALL_UP(R) return launch_gate_up<1, R>(h, x, T, s)
    ZEDA_RPL_DISPATCH(ZEDA_CALL_UP);
#undef ZEDA_CALL_UP
}

int launch_stream_down(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y, __nv_bfloat16 *resid, cudaStream_t s) {
    const int n_cand = h->cfg.n_real + h->cfg.n_zero;
    if (!stream_routes_itself(h, T)) return launch_down<2, 0>(h, x, T, y, resid, s);
#define ZEDA_CALL_DOWN(R) return launch_down<1, R>(h, x, T, y, resid, s)
    ZEDA_RPL_DISPATCH(ZEDA_CALL_DOWN);
#undef ZEDA_CALL_DOWN
}

}  // namespace zeda
