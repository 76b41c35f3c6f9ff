// Internal declarations shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "zeda.h"

namespace zeda {

constexpr int kMaxCand = 512;       // N + N_Z limit (16 logits per lane in the top-K warp)
constexpr int kMaxTopK = 16;
constexpr int kSortTokens = 128;    // tokens per CTA in the counting sort (histogram / placement)
constexpr int kPairTileM = 256;     // most pair rows per tile of the expert kernels (one CTA pair, N <= 256)
constexpr int kMidTileM = 128;      // tile rows of the geometry for mid-sized batches
constexpr int kMaxEpRanks = 64;     // expert-parallel group size limit
constexpr int kStreamTokens = 16;   // calls of at most this many tokens may run the expert kernels of small_batch.cu
constexpr int kStreamSlots = kStreamTokens * kMaxTopK;  // their largest slot table

constexpr int kTileRouterTokens = 256;     // calls of at least this many tokens have their logits from the tensor cores
// From so many tokens on, up to so many candidates and where pair_router_path says so, the router with top-K.  Below,
// tiles of 256 tokens would need up to eight slices of the reduction axis to cover the SMs: measured with them, one layer
// of 777 tokens took 227.9 us with the logits' own kernel and 228.3 with it, 2048 tokens 256.3 and 257.1.  It has three.
constexpr int kPairRouterTokens = 4096;
constexpr int kPairRouterMaxCand = 256;
constexpr int kPairRouterMaxSliced = 160;  // its CTAs where it slices the reduction axis (bounds the statistics' buffer)
constexpr int kHostMaxChunks = 3;   // of the host-buffer entry point

// Device-resident counters of one call.
enum MetaSlot {
    kMetaPairs = 0,      // P
    kMetaActive = 1,     // U
    kMetaZeroSlots = 2,  // slots that landed on zero experts
    kMetaError = 5,      // sticky error word written by bounded device waits
    kMetaMaxRows = 6,    // largest per-expert pair count
    kMetaPairTiles = 7,  // entries of the expert kernels' tile list
    kMetaNextItem1 = 8,  // next unclaimed work item of the GEMM1 kernel (reset by the routing pass)
    kMetaNextItem2 = 9,  // the same for GEMM2
    kMetaRouted = 10,    // smallest batches: the routing tables of the call are in the workspace (the router clears it)
    kMetaCount = 16
};

struct Workspace {
    int32_t *topk_idx;     // [maxT*K]
    float *topk_w;         // [maxT*K]
    int32_t *inv;          // [maxT*K] slot -> sorted position, -1 for zero slots
    int32_t *perm;         // [maxT*K] sorted position -> slot
    int32_t *pair_token;   // [maxT*K] sorted position -> token
    int32_t *block_hist;   // [nblk*N]
    int32_t *counts;       // [N]
    int32_t *offsets;      // [N+1]
    int32_t *meta;         // [kMetaCount]
    int32_t *ptile_expert; // [maxTiles] tiles of at most kPairTileM pair rows of one expert
    int32_t *ptile_row0;   // [maxTiles] first row of the tile within its expert
    float *logits;         // [router_part_rows(maxT)*(N+N_Z)]: complete logits or up to eight slices of them
    float *stat_part;      // [nblk_stats * 2 * (N+N_Z)]
    __nv_bfloat16 *hmid;   // [maxT*K, He]
    __nv_bfloat16 *obuf;   // [maxT*K, d] (not on expert-parallel handles: their results go to the caller's buffer)
    __nv_bfloat16 *router_split; // [3][pad128(N+N_Z)][d] bf16 hi/mid/lo pieces of the router rows
    __nv_bfloat16 *x_stage;// [maxT, d]
    __nv_bfloat16 *y_stage;// [maxT, d]
    // expert-parallel handles only: the plan of the rows received from the group
    int32_t *ep_counts;      // [N_local] received pairs per local expert
    int32_t *ep_offsets;     // [N_local + 1]
    int32_t *ep_pair_row;    // [maxR] sorted position -> received row
    int32_t *ep_tile_expert; // [maxR / kMidTileM + N_local + 1]
    int32_t *ep_tile_row0;
};

// What one launch of the expert kernels works on: per-expert counts and offsets of the pair rows,
// the tile list, and for GEMM1 the row of the activation matrix that each pair row reads.
struct ExpertWork {
    const int32_t *counts, *offsets, *tile_expert, *tile_row0, *pair_row;
    int rows_bound;  // upper bound of the pair rows of a call (host-side; picks the kernel geometry)
    int tile_rows;   // pair rows per tile of the tile list (kPairTileM or kMidTileM)
};

// Device-side tile list written by the expert scan: experts in id order, each with its tiles of at
// most kPairTileM pair rows in row order.
struct WorkLists {
    int32_t *ptile_expert, *ptile_row0;
};

struct RouteOut {  // where one routing pass writes (user buffers or workspace)
    int32_t *topk_idx;
    float *topk_w;
    int32_t *counts;
    int32_t *offsets;
    int32_t *perm;
    int32_t *n_pairs;  // optional extra copy of P
};

struct StatsOut {  // where a statistics call wants its results (each may be NULL)
    float *f, *p_mean, *out;
};

}  // namespace zeda

struct zeda_moe {
    zeda_moe_config_t cfg;
    bool pdl;  // launch the forward kernels with programmatic stream serialization
    const float *router_w;
    const float *router_bias;
    const __nv_bfloat16 *w_gate_up;
    const __nv_bfloat16 *w_down;
    zeda::Workspace ws;
    int sm_count;
    int router_clusters8, router_clusters4;  // clusters of 8 and of 4 CTAs of the router of 33 to 255 tokens that run at a time
    int max_tiles;
    int n_local;    // experts whose weights this handle holds (n_real unless expert-parallel)
    int pair_rows;  // capacity of the pair buffers (max_tokens * top_k, or max_recv_pairs)
    int last_launches;
    void *pmaps;  // host-side tensor maps of the expert kernels (owned)
    void *router_maps;  // host-side tensor map of the split router weights (owned)
    void *pair_router;  // the same for the router with top-K, NULL where it does not take the shape (owned)
    bool profiling;
    bool profiled_last;
    int last_routed_tokens;  // T of the most recent routing pass on this handle
    cudaEvent_t ev[ZEDA_STAGE_COUNT + 1];
    // host-buffer entry point: copy streams and events of its chunk pipeline (made on first use)
    cudaStream_t copy_in, copy_out;
    cudaEvent_t ev_host[2 + 2 * zeda::kHostMaxChunks];
};

namespace zeda {

// Block histograms of the counting sort for a call of T tokens, as far as the top-K pass counts into them
// (more blocks have a histogram kernel of their own): the router kernel of the call sets them to zero.
constexpr int kFoldMaxBlocks = 256;
inline int hist_ints(const zeda_moe *h, int T) {
    const int nblk = (T + kSortTokens - 1) / kSortTokens;
    return nblk <= kFoldMaxBlocks ? nblk * h->cfg.n_real : 0;
}
#if defined(__CUDACC__)
// by all CTAs of a one- or two-dimensional grid
__device__ __forceinline__ void clear_hist(int32_t *__restrict__ hist, int n) {
    const int cta = blockIdx.y * gridDim.x + blockIdx.x;
    for (int i = cta * blockDim.x + threadIdx.x; i < n; i += gridDim.x * gridDim.y * blockDim.x) hist[i] = 0;
}
#endif

// ---- launchers (each returns the number of kernels it enqueued, or <0 on a launch error) ----
int init_route_kernels(zeda_moe *h);
// With n_parts == nullptr the logits are complete.  Otherwise the router may cut the reduction axis
// into *n_parts slices (mid-sized batches on the tensor-core path): slice p then lies at
// logits + p * T * n_cand, and launch_route_from_logits adds the slices in order.  Where the router with top-K takes the
// call, no logits are written and *n_parts is 0: the slots' ids and weights and the block histograms are there already.
// split_T: the number of tokens that the slicing is decided by, if not T (a call that is one part of a
// batch gives the batch's, so that its logits are the batch's bits).
int launch_router_logits(const zeda_moe *h, const __nv_bfloat16 *x, int T, float *logits, cudaStream_t s,
                         int *n_parts = nullptr, int split_T = 0, float *stat_part = nullptr);
int launch_route_from_logits(const zeda_moe *h, const float *logits, int T, const RouteOut &out, cudaStream_t s,
                             int n_parts = 1, const StatsOut *stats = nullptr);
int launch_topk(const zeda_moe *h, const float *logits, int n_parts, int T, float *stat_part, cudaStream_t s);
int router_split_pad(int n_cand);
int init_router_tile(zeda_moe *h);
int init_router_pair(zeda_moe *h);  // behind init_router_tile, which splits the router rows
bool pair_router_path(const zeda_moe *h, int T);
int pair_router_slices(const zeda_moe *h, int T);
int pair_router_stat_blocks(const zeda_moe *h, int T);  // CTAs that leave partial sums of the statistics
int launch_router_topk_pair(const zeda_moe *h, const __nv_bfloat16 *x, int T, int split_T, int32_t *block_hist, float *stat_part,
                            cudaStream_t s);
constexpr int kRouterMaxSplit = 8;
// rows of n_cand floats that the workspace holds for router output (complete logits or their slices)
inline long long router_part_rows(long long max_tokens, int n_cand) {
    // slices x tokens that cover 150 SMs with a tile of 128 tokens x 128 candidates each
    const long long cap = 19200 / ((n_cand + 127) / 128);
    const long long want = kRouterMaxSplit * max_tokens < cap ? kRouterMaxSplit * max_tokens : cap;
    return max_tokens > want ? max_tokens : want;
}
int router_split_factor(const zeda_moe *h, int T);
int launch_router_logits_tile(const zeda_moe *h, const __nv_bfloat16 *x, int T, float *logits, int split, cudaStream_t s);
int init_pair_kernels(zeda_moe *h);
// Pair rows per tile for a call of T tokens on this handle: the routing pass builds the tile list with
// it and the expert kernels of the same call are picked to match.
int tile_rows_for(const zeda_moe *h, int T);
int ep_tile_rows_for(const zeda_moe *h, int n_rows);
int launch_token_zero_share(const zeda_moe *h, int T, float *out, cudaStream_t s);
int launch_experts_gemm1_pair(const zeda_moe *h, const __nv_bfloat16 *x, const ExpertWork &w, cudaStream_t s);
// out: where the results go, in sorted order or (expert-parallel handles) in the order of pair_row
int launch_experts_gemm2_pair(const zeda_moe *h, const ExpertWork &w, __nv_bfloat16 *out, cudaStream_t s);
// the smallest batches (small_batch.cu): GEMM1, and GEMM2 with the combine (resid given: with the residual update)
bool stream_path(const zeda_moe *h, int T);
bool stream_routes_itself(const zeda_moe *h, int T);  // the expert kernels also do the routing: logits -> y
int init_stream_kernels();
int launch_stream_gemm1(const zeda_moe *h, const __nv_bfloat16 *x, int T, cudaStream_t s);
int launch_stream_down(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y, __nv_bfloat16 *resid, cudaStream_t s);
int launch_residual_rmsnorm(bool pdl, __nv_bfloat16 *r, const __nv_bfloat16 *y, __nv_bfloat16 *h, int T, int d, float eps, cudaStream_t s);
// expert-parallel pieces (expert_parallel.cu)
int launch_ep_pack(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *send_rows, int32_t *send_counts,
                   int32_t *expert_counts, cudaStream_t s);
int launch_ep_plan(const zeda_moe *h, const int32_t *recv_counts, int n_rows, int tile_rows, cudaStream_t s);
int launch_combine_rows(const zeda_moe *h, const __nv_bfloat16 *rows, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y,
                        cudaStream_t s);
int launch_wait_selftest(const zeda_moe *h, long long limit_cycles, cudaStream_t s);
int launch_combine(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y, cudaStream_t s);
// combine fused with the residual + RMSNorm glue of a layer stack (rows of up to 2048 elements)
bool combine_glue_supported(const zeda_moe *h);
int launch_combine_glue(const zeda_moe *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *resid, __nv_bfloat16 *h_next, float eps,
                        cudaStream_t s);

void set_error(const char *fmt, ...);
// remembers the error of a failed kernel launch for the status message of the API call (the runtime's
// own "last error" may have been read and cleared by a later launch check)
void note_launch_error(cudaError_t e);

// ---- programmatic dependent launch ------------------------------------------------------------
// The kernels of one forward pass are launched back to back on one stream.  Launched with the
// attribute below, a kernel may start (launch latency, barrier and TMEM set-up) while its
// predecessor is still draining; it touches no global memory until pdl_wait() returns, which is
// when the predecessor has completed and its writes are visible.  What a kernel in front has written is read
// by volatile loads (__ldcg and those below), which the compiler keeps behind the wait.  It need not do that
// for __ldg, nor for a plain load through a __restrict__ parameter (of const data it is the same non-coherent
// load), and it did not: a placement pass met ids that were not written yet.
// Each kernel calls pdl_launch_dependents() first thing so that its successor is released as early as possible.
// The GEMM1 kernels do so behind their own wait: the routing results are complete when GEMM2 starts, which reads
// them in front of its wait, past L1 (ld.cg), where an older line could be.
// Without the attribute both calls do nothing.
#if defined(__CUDACC__)
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// *p, or `other` where `on` is false, as one predicated load
__device__ __forceinline__ float ldcg_if(bool on, const float *p, float other) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.cg.f32 %0, [%1];\n\t}" : "+f"(other) : "l"(p), "r"((unsigned)on));
    return other;
}

// a load through L1, behind the wait only: for lines that all threads of a CTA read
__device__ __forceinline__ int32_t ld_ordered(const int32_t *p) {
    int32_t v;
    asm volatile("ld.global.ca.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ float swiglu(float g, float u) { return __fdividef(g * u, 1.f + __expf(-g)); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                 Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
    if (e != cudaSuccess) note_launch_error(e);
    return e;
}
#endif

}  // namespace zeda
