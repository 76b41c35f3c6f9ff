// Host side of the C ABI: argument checks, workspace carving, stream-ordered launches.
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include "zeda_internal.h"

namespace zeda {

static thread_local char g_err[512] = "";

void set_error(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
}

namespace {

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

bool config_ok(const zeda_moe_config_t *c, const char **why) {
    const char *w = nullptr;
    if (!c) w = "config is NULL";
    else if (c->d_model < 64 || c->d_model % 64 || c->d_model > 8192) w = "d_model must be a multiple of 64 in [64, 8192]";
    else if (c->d_expert < 64 || c->d_expert % 64 || c->d_expert > 8192) w = "d_expert must be a multiple of 64 in [64, 8192]";
    else if (c->n_real < 1) w = "n_real must be >= 1";
    else if (c->n_zero < 0) w = "n_zero must be >= 0";
    else if (c->n_real + c->n_zero > kMaxCand) w = "n_real + n_zero must be <= 512";
    else if (c->top_k < 1 || c->top_k > kMaxTopK) w = "top_k must be in [1, 16]";
    else if (c->top_k > c->n_real + c->n_zero) w = "top_k exceeds the number of candidates";
    else if (c->max_tokens < 1) w = "max_tokens must be >= 1";
    else if ((long long)c->max_tokens * c->top_k >= (1LL << 27)) w = "max_tokens * top_k must be < 2^27";
    else if (c->gate_mode < 0 || c->gate_mode > 2) w = "unknown gate_mode";
    else if (c->expert_kind < 0 || c->expert_kind > 1) w = "unknown expert_kind";
    else if (c->flags & ~ZEDA_FLAG_NO_DEPENDENT_LAUNCH) w = "unknown flag";
    else if (c->ep_size < 0 || c->ep_size > kMaxEpRanks) w = "ep_size must be in [0, 64]";
    else if (c->ep_size >= 1 && (c->n_real % c->ep_size) != 0) w = "n_real must be a multiple of ep_size";
    else if (c->ep_size >= 1 && (c->ep_rank < 0 || c->ep_rank >= c->ep_size)) w = "ep_rank outside [0, ep_size)";
    else if (c->ep_size >= 1 && (c->max_recv_pairs < 1 || c->max_recv_pairs >= (1 << 27))) w = "max_recv_pairs must be in [1, 2^27)";
    if (why) *why = w;
    return w == nullptr;
}

size_t hist_bytes(const zeda_moe_config_t &c) {
    return (size_t)((c.max_tokens + kSortTokens - 1) / kSortTokens) * c.n_real * sizeof(int32_t);
}

// Walks the workspace layout; with base == nullptr it only measures.
size_t carve(const zeda_moe_config_t &c, unsigned char *base, Workspace *ws, int *max_tiles) {
    size_t off = 0;
    auto take = [&](size_t bytes) -> void * {
        void *p = base ? base + off : nullptr;
        off = align_up(off + bytes, 256);
        return p;
    };
    const size_t slots = (size_t)c.max_tokens * c.top_k;
    const size_t n_cand = (size_t)c.n_real + c.n_zero;
    const size_t nblk = (c.max_tokens + kSortTokens - 1) / kSortTokens;
    const size_t tiles = slots / kMidTileM + c.n_real + 1;
    // an expert-parallel handle holds n_local experts and sizes its pair buffers for the rows it may receive
    const bool ep = c.ep_size >= 1;
    const size_t n_local = ep ? (size_t)c.n_real / c.ep_size : (size_t)c.n_real;
    const size_t pair_rows = ep ? (size_t)c.max_recv_pairs : slots;
    const size_t ep_tiles = pair_rows / kMidTileM + n_local + 1;
    size_t nblk_stats = (c.max_tokens + 63) / 64;
    if (nblk_stats < kPairRouterMaxSliced) nblk_stats = kPairRouterMaxSliced;
    Workspace w;
    w.topk_idx = (int32_t *)take(slots * 4);
    w.topk_w = (float *)take(slots * 4);
    w.inv = (int32_t *)take(slots * 4);
    w.perm = (int32_t *)take(slots * 4);
    w.pair_token = (int32_t *)take(slots * 4);
    w.block_hist = (int32_t *)take(hist_bytes(c));
    w.counts = (int32_t *)take((size_t)c.n_real * 4);
    w.offsets = (int32_t *)take((size_t)(c.n_real + 1) * 4);
    w.meta = (int32_t *)take(kMetaCount * 4);
    w.ptile_expert = (int32_t *)take(tiles * 4);
    w.ptile_row0 = (int32_t *)take(tiles * 4);
    w.logits = (float *)take((size_t)router_part_rows(c.max_tokens, (int)n_cand) * n_cand * 4);
    w.stat_part = (float *)take(nblk_stats * 2 * n_cand * 4);
    // pair buffers carry one tile of slack rows so that a full tile may be read past the last pair
    w.hmid = (__nv_bfloat16 *)take((pair_rows + kPairTileM) * c.d_expert * 2);
    w.obuf = ep ? nullptr : (__nv_bfloat16 *)take((pair_rows + kPairTileM) * c.d_model * 2);
    w.router_split = (__nv_bfloat16 *)take((size_t)3 * router_split_pad((int)n_cand) * c.d_model * 2);
    w.x_stage = (__nv_bfloat16 *)take((size_t)c.max_tokens * c.d_model * 2);
    w.y_stage = (__nv_bfloat16 *)take((size_t)c.max_tokens * c.d_model * 2);
    w.ep_counts = w.ep_offsets = w.ep_pair_row = w.ep_tile_expert = w.ep_tile_row0 = nullptr;
    if (ep) {
        w.ep_counts = (int32_t *)take(n_local * 4);
        w.ep_offsets = (int32_t *)take((n_local + 1) * 4);
        w.ep_pair_row = (int32_t *)take(pair_rows * 4);
        w.ep_tile_expert = (int32_t *)take(ep_tiles * 4);
        w.ep_tile_row0 = (int32_t *)take(ep_tiles * 4);
    }
    if (ws) *ws = w;
    if (max_tiles) *max_tiles = (int)tiles;
    return off;
}

// text for the sticky device-side error word
const char kDeviceFailure[] = "a bounded device wait expired or a device-side check failed (code %d; 21 = the row count "
                              "passed to zeda_ep_experts is not the sum of its count matrix)";

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

thread_local cudaError_t t_launch_error = cudaSuccess;

zeda_status_t cuda_fail(const char *what, cudaError_t e) {
    if (e == cudaSuccess) e = t_launch_error;  // a launch that failed earlier in this call
    t_launch_error = cudaSuccess;
    set_error("%s: %s", what, cudaGetErrorString(e));
    return ZEDA_ERR_CUDA;
}

zeda_status_t check_call(zeda_moe_t *h, const void *in, int32_t T, const char *in_name) {
    if (!h) { set_error("handle is NULL"); return ZEDA_ERR_INVALID_ARG; }
    if (T < 0 || T > h->cfg.max_tokens) { set_error("T=%d outside [0, max_tokens=%d]", T, h->cfg.max_tokens); return ZEDA_ERR_INVALID_ARG; }
    if (T > 0 && !in) { set_error("%s is NULL", in_name); return ZEDA_ERR_INVALID_ARG; }
    if (T > 0 && !aligned16(in)) { set_error("%s is not 16-byte aligned", in_name); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    return ZEDA_OK;
}

// Routing into the workspace (+ optional user copies); returns launches or <0.
// stats: where a statistics call wants its results; the top-K pass leaves their partial sums in the workspace.
int route_into(zeda_moe_t *h, const __nv_bfloat16 *x, const float *logits_in, int T, const RouteOut &out, cudaStream_t s,
               const StatsOut *stats = nullptr) {
    int n = 0, n_parts = 1;
    h->last_routed_tokens = 0;  // until every launch is in the stream, the handle holds no batch's routing
    const float *logits = logits_in;
    if (!logits) {
        int r = launch_router_logits(h, x, T, h->ws.logits, s, &n_parts, 0, stats ? h->ws.stat_part : nullptr);
        if (r < 0) return r;
        n += r;
        logits = h->ws.logits;
    }
    int r = launch_route_from_logits(h, logits, T, out, s, n_parts, stats);
    if (r < 0) return r;
    h->last_routed_tokens = T;
    return n + r;
}

// Whether the router adds up the reduction axis alike for calls of a and of b tokens.
bool same_router_slices(const zeda_moe *h, int a, int b) {
    if (pair_router_path(h, a) != pair_router_path(h, b)) return false;
    return pair_router_path(h, a) ? pair_router_slices(h, a) == pair_router_slices(h, b) : router_split_factor(h, a) == router_split_factor(h, b);
}

// The batches that a chunk of the host-buffer call belongs to: its first `cut` tokens (a multiple of kSortTokens) to one of
// `first` tokens, the others to one of `rest`.  Its tokens are routed as in calls of those batches.
struct ChunkOf {
    int cut, first, rest;
};

// The router's part of a call of T tokens, as launch_router_logits; of a chunk whose two batches the router treats
// differently, slots of both parts are chosen apart (*n_parts = 0) and placed together behind.
int launch_router(const zeda_moe *h, const __nv_bfloat16 *x, int T, const ChunkOf *of, cudaStream_t s, int *n_parts) {
    if (!of || of->cut == 0 || of->cut >= T || same_router_slices(h, of->first, of->rest))
        return launch_router_logits(h, x, T, h->ws.logits, s, n_parts, !of ? 0 : of->cut > 0 ? of->first : of->rest);
    int n = 0;
    for (int at = 0; at < T; at = at ? T : of->cut) {
        zeda_moe part = *h;  // the same handle, with the part's slots and histogram blocks in front
        part.ws.topk_idx += (size_t)at * h->cfg.top_k;
        part.ws.topk_w += (size_t)at * h->cfg.top_k;
        part.ws.block_hist += (size_t)(at / kSortTokens) * h->cfg.n_real;
        const int tokens = at ? T - at : of->cut;
        int r = launch_router_logits(&part, x + (size_t)at * h->cfg.d_model, tokens, h->ws.logits, s, n_parts, at ? of->rest : of->first);
        if (r < 0) return r;
        n += r;
        if (*n_parts == 0) continue;  // the router has chosen
        r = launch_topk(&part, h->ws.logits, *n_parts, tokens, nullptr, s);
        if (r < 0) return r;
        n += r;
    }
    *n_parts = 0;
    return n;
}

// With resid given, the call ends in the fused combine + glue pass: resid <- bf16(resid + y) and
// the normalised residual goes where y would have gone.
zeda_status_t forward_device(zeda_moe_t *h, const __nv_bfloat16 *x, int T, __nv_bfloat16 *y, cudaStream_t s,
                             __nv_bfloat16 *resid = nullptr, float eps = 0.f, const ChunkOf *of = nullptr) {
    const bool prof = h->profiling;
    auto mark = [&](int i) { if (prof) cudaEventRecord(h->ev[i], s); };
    mark(0);
    h->last_routed_tokens = 0;
    int n_parts = 1;
    int n = launch_router(h, x, T, of, s, &n_parts);
    if (n < 0) return cuda_fail("router launch", cudaGetLastError());
    mark(1);
    RouteOut none = {};
    int r = stream_routes_itself(h, T) ? 0 : launch_route_from_logits(h, h->ws.logits, T, none, s, n_parts);
    if (r < 0) return cuda_fail("routing launch", cudaGetLastError());
    n += r;
    mark(2);
    const Workspace &ws = h->ws;
    if (stream_path(h, T)) {  // the down projection and the combine are one kernel: its time counts as GEMM2
        r = launch_stream_gemm1(h, x, T, s);
        if (r < 0) return cuda_fail("expert GEMM1 launch", cudaGetLastError());
        h->last_routed_tokens = T;  // (this kernel may have been the one that routes)
        n += r;
        mark(3);
        r = launch_stream_down(h, x, T, y, resid, s);
        if (r < 0) return cuda_fail("expert GEMM2 launch", cudaGetLastError());
        n += r;
        mark(4);
        r = resid ? launch_residual_rmsnorm(h->pdl, resid, nullptr, y, T, h->cfg.d_model, eps, s) : 0;
        if (r < 0) return cuda_fail("norm launch", cudaGetLastError());
        mark(5);
        h->profiled_last = prof;
        h->last_launches = n + r;
        return ZEDA_OK;
    }
    h->last_routed_tokens = T;
    const ExpertWork work = {ws.counts, ws.offsets, ws.ptile_expert, ws.ptile_row0, ws.pair_token, T * h->cfg.top_k, tile_rows_for(h, T)};
    r = launch_experts_gemm1_pair(h, x, work, s);
    if (r < 0) return cuda_fail("expert GEMM1 launch", cudaGetLastError());
    n += r;
    mark(3);
    r = launch_experts_gemm2_pair(h, work, ws.obuf, s);
    if (r < 0) return cuda_fail("expert GEMM2 launch", cudaGetLastError());
    n += r;
    mark(4);
    r = resid ? launch_combine_glue(h, x, T, resid, y, eps, s) : launch_combine(h, x, T, y, s);
    if (r < 0) return cuda_fail("combine launch", cudaGetLastError());
    mark(5);
    h->profiled_last = prof;
    h->last_launches = n + r;
    return ZEDA_OK;
}

}  // namespace

void note_launch_error(cudaError_t e) {
    if (t_launch_error == cudaSuccess) t_launch_error = e;
}

}  // namespace zeda

using namespace zeda;

extern "C" {

size_t zeda_moe_workspace_bytes(const zeda_moe_config_t *cfg) {
    const char *why = nullptr;
    if (!config_ok(cfg, &why)) { set_error("%s", why); return 0; }
    return carve(*cfg, nullptr, nullptr, nullptr);
}

zeda_status_t zeda_moe_create(const zeda_moe_config_t *cfg, const float *router_w, const float *router_bias,
                              const void *w_gate_up, const void *w_down, void *workspace, size_t workspace_bytes,
                              zeda_moe_t **out) {
    if (out) *out = nullptr;
    const char *why = nullptr;
    if (!config_ok(cfg, &why)) {
        set_error("%s", why);
        const bool shape = cfg && why && (strstr(why, "multiple of 64") || strstr(why, "<= 512") || strstr(why, "[1, 16]"));
        return shape ? ZEDA_ERR_UNSUPPORTED : ZEDA_ERR_INVALID_ARG;
    }
    if (!out) { set_error("out is NULL"); return ZEDA_ERR_INVALID_ARG; }
    if (!router_w || !w_gate_up || !w_down || !workspace) { set_error("a required pointer is NULL"); return ZEDA_ERR_INVALID_ARG; }
    if (!aligned16(router_w) || !aligned16(w_gate_up) || !aligned16(w_down) || (router_bias && (reinterpret_cast<uintptr_t>(router_bias) & 3u))) {
        set_error("weights must be 16-byte aligned");
        return ZEDA_ERR_INVALID_ARG;
    }
    if (reinterpret_cast<uintptr_t>(workspace) & 255u) { set_error("workspace must be 256-byte aligned"); return ZEDA_ERR_INVALID_ARG; }
    const size_t need = carve(*cfg, nullptr, nullptr, nullptr);
    if (workspace_bytes < need) { set_error("workspace has %zu bytes, %zu needed", workspace_bytes, need); return ZEDA_ERR_WORKSPACE; }
    int ndev = 0;
    cudaError_t e = cudaGetDeviceCount(&ndev);
    if (e != cudaSuccess) return cuda_fail("cudaGetDeviceCount", e);
    if (cfg->device < 0 || cfg->device >= ndev) { set_error("device %d not present (%d devices)", cfg->device, ndev); return ZEDA_ERR_INVALID_ARG; }
    e = cudaSetDevice(cfg->device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    cudaDeviceProp prop;
    e = cudaGetDeviceProperties(&prop, cfg->device);
    if (e != cudaSuccess) return cuda_fail("cudaGetDeviceProperties", e);
    if (prop.major != 10) { set_error("this library is built for sm_100a only; device is sm_%d%d", prop.major, prop.minor); return ZEDA_ERR_UNSUPPORTED; }

    zeda_moe *h = new (std::nothrow) zeda_moe();
    if (!h) { set_error("out of host memory"); return ZEDA_ERR_INVALID_ARG; }
    h->cfg = *cfg;
    h->router_w = router_w;
    h->router_bias = router_bias;
    h->w_gate_up = static_cast<const __nv_bfloat16 *>(w_gate_up);
    h->w_down = static_cast<const __nv_bfloat16 *>(w_down);
    h->sm_count = prop.multiProcessorCount;
    h->router_clusters8 = h->router_clusters4 = 0;
    h->pdl = !(cfg->flags & ZEDA_FLAG_NO_DEPENDENT_LAUNCH);
    h->last_launches = 0;
    h->last_routed_tokens = 0;
    h->n_local = cfg->ep_size >= 1 ? cfg->n_real / cfg->ep_size : cfg->n_real;
    h->pair_rows = cfg->ep_size >= 1 ? cfg->max_recv_pairs : cfg->max_tokens * cfg->top_k;
    h->pmaps = nullptr;
    h->router_maps = nullptr;
    h->pair_router = nullptr;
    h->profiling = false;
    h->profiled_last = false;
    for (auto &ev : h->ev) ev = nullptr;
    h->copy_in = h->copy_out = nullptr;
    for (auto &ev : h->ev_host) ev = nullptr;
    carve(*cfg, static_cast<unsigned char *>(workspace), &h->ws, &h->max_tiles);
    if (init_route_kernels(h) < 0) { delete h; return cuda_fail("kernel set-up", cudaGetLastError()); }
    if (init_stream_kernels() < 0) { delete h; return cuda_fail("kernel set-up", cudaGetLastError()); }
    if (init_pair_kernels(h) < 0) { delete h; return ZEDA_ERR_CUDA; }
    if (init_router_tile(h) < 0 || init_router_pair(h) < 0) {
        if (h->pmaps) free(h->pmaps);
        if (h->router_maps) free(h->router_maps);
        delete h;
        return cuda_fail("router set-up", cudaGetLastError());
    }
    e = cudaMemset(h->ws.meta, 0, kMetaCount * 4);
    if (e != cudaSuccess) { delete h; return cuda_fail("cudaMemset(meta)", e); }
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) { delete h; return cuda_fail("cudaDeviceSynchronize", e); }
    *out = h;
    return ZEDA_OK;
}

zeda_status_t zeda_route(zeda_moe_t *h, const void *x, int32_t T, int32_t *topk_idx, float *topk_w,
                         int32_t *expert_counts, int32_t *expert_offsets, int32_t *perm, int32_t *n_pairs,
                         void *stream) {
    zeda_status_t st = check_call(h, x, T, "x");
    if (st != ZEDA_OK || T == 0) return st;
    RouteOut out = {topk_idx, topk_w, expert_counts, expert_offsets, perm, n_pairs};
    int n = route_into(h, static_cast<const __nv_bfloat16 *>(x), nullptr, T, out, static_cast<cudaStream_t>(stream));
    if (n < 0) return cuda_fail("routing launch", cudaGetLastError());
    h->last_launches = n;
    return ZEDA_OK;
}

zeda_status_t zeda_route_from_logits(zeda_moe_t *h, const float *logits, int32_t T, int32_t *topk_idx, float *topk_w,
                                     int32_t *expert_counts, int32_t *expert_offsets, int32_t *perm,
                                     int32_t *n_pairs, void *stream) {
    zeda_status_t st = check_call(h, logits, T, "logits");
    if (st != ZEDA_OK || T == 0) return st;
    RouteOut out = {topk_idx, topk_w, expert_counts, expert_offsets, perm, n_pairs};
    int n = route_into(h, nullptr, logits, T, out, static_cast<cudaStream_t>(stream));
    if (n < 0) return cuda_fail("routing launch", cudaGetLastError());
    h->last_launches = n;
    return ZEDA_OK;
}

zeda_status_t zeda_router_logits(zeda_moe_t *h, const void *x, int32_t T, float *logits, void *stream) {
    zeda_status_t st = check_call(h, x, T, "x");
    if (st != ZEDA_OK || T == 0) return st;
    if (!logits) { set_error("logits is NULL"); return ZEDA_ERR_INVALID_ARG; }
    int n = launch_router_logits(h, static_cast<const __nv_bfloat16 *>(x), T, logits, static_cast<cudaStream_t>(stream));
    if (n < 0) return cuda_fail("router launch", cudaGetLastError());
    h->last_launches = n;
    return ZEDA_OK;
}

zeda_status_t zeda_moe_forward(zeda_moe_t *h, const void *x, int32_t T, void *y, void *stream) {
    zeda_status_t st = check_call(h, x, T, "x");
    if (st != ZEDA_OK || T == 0) return st;
    if (h->cfg.ep_size >= 1) { set_error("an expert-parallel handle (ep_size >= 1) runs the layer through the zeda_ep_* calls"); return ZEDA_ERR_INVALID_ARG; }
    if (!y || !aligned16(y)) { set_error("y is NULL or not 16-byte aligned"); return ZEDA_ERR_INVALID_ARG; }
    const size_t bytes = (size_t)T * h->cfg.d_model * 2;
    const char *xb = static_cast<const char *>(x), *yb = static_cast<const char *>(y);
    if (xb < yb + bytes && yb < xb + bytes) { set_error("x and y overlap"); return ZEDA_ERR_INVALID_ARG; }
    return forward_device(h, static_cast<const __nv_bfloat16 *>(x), T, static_cast<__nv_bfloat16 *>(y),
                          static_cast<cudaStream_t>(stream));
}

zeda_status_t zeda_moe_forward_residual(zeda_moe_t *h, const void *x, int32_t T, void *r, void *h_next, float eps,
                                        void *stream) {
    zeda_status_t st = check_call(h, x, T, "x");
    if (st != ZEDA_OK || T == 0) return st;
    if (h->cfg.ep_size >= 1) { set_error("an expert-parallel handle (ep_size >= 1) runs the layer through the zeda_ep_* calls"); return ZEDA_ERR_INVALID_ARG; }
    if (!combine_glue_supported(h)) { set_error("the fused residual form needs d_model <= 2048"); return ZEDA_ERR_UNSUPPORTED; }
    if (!r || !h_next || !aligned16(r) || !aligned16(h_next)) { set_error("r or h_next is NULL or not 16-byte aligned"); return ZEDA_ERR_INVALID_ARG; }
    if (!(eps >= 0.f)) { set_error("eps must be >= 0"); return ZEDA_ERR_INVALID_ARG; }
    const size_t bytes = (size_t)T * h->cfg.d_model * 2;
    const char *b[3] = {static_cast<const char *>(x), static_cast<const char *>(r), static_cast<const char *>(h_next)};
    for (int i = 0; i < 3; ++i)
        for (int j = i + 1; j < 3; ++j)
            if (b[i] < b[j] + bytes && b[j] < b[i] + bytes) { set_error("x, r and h_next overlap"); return ZEDA_ERR_INVALID_ARG; }
    return forward_device(h, static_cast<const __nv_bfloat16 *>(x), T, static_cast<__nv_bfloat16 *>(h_next),
                          static_cast<cudaStream_t>(stream), static_cast<__nv_bfloat16 *>(r), eps);
}

// The host-buffer entry point cuts large batches into chunks, so that the copy of a chunk runs under the
// layer of the one before and the copies back under the layers behind; each chunk reads the experts'
// weights again.  Below 4096 tokens a second pass over the weights costs more than the copies it hides.
// A third chunk pays from 8192 tokens on: 1234 -> 1189 us a call of 8192 tokens where every expert is active and
// a third pass over all weights costs most, 2377 -> 2128 of 16384, 4594 -> 4075 of 32768; Zipf load 1273 -> 1176,
// 2404 -> 2100, 4676 -> 4127.  At 7168 an even load loses 5 %.
// Equal chunks: with a quarter, a half and a quarter the copies back queue up behind the half (1216 us).
static const int kHostSplitMinTokens = 4096, kHostThreeChunksMinTokens = 8192;

zeda_status_t zeda_moe_forward_host(zeda_moe_t *h, const void *x_host, int32_t T, void *y_host, void *stream) {
    if (!h) { set_error("handle is NULL"); return ZEDA_ERR_INVALID_ARG; }
    if (T < 0 || T > h->cfg.max_tokens) { set_error("T=%d outside [0, max_tokens=%d]", T, h->cfg.max_tokens); return ZEDA_ERR_INVALID_ARG; }
    if (T == 0) return ZEDA_OK;
    if (h->cfg.ep_size >= 1) { set_error("an expert-parallel handle (ep_size >= 1) runs the layer through the zeda_ep_* calls"); return ZEDA_ERR_INVALID_ARG; }
    if (!x_host || !y_host) { set_error("host buffer is NULL"); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t row = (size_t)h->cfg.d_model * 2;
    if (T < kHostSplitMinTokens) {
        e = cudaMemcpyAsync(h->ws.x_stage, x_host, T * row, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return cuda_fail("copy of x to the device", e);
        zeda_status_t st = forward_device(h, h->ws.x_stage, T, h->ws.y_stage, s);
        if (st != ZEDA_OK) return st;
        e = cudaMemcpyAsync(y_host, h->ws.y_stage, T * row, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return cuda_fail("copy of y to the host", e);
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail("cudaStreamSynchronize", e);
        return ZEDA_OK;
    }
    // The layer is per token (Eq. 1), so the chunks are independent calls; their device work stays on
    // `stream`, one after the other (they share the workspace), the copies run on two streams of the handle.
    if (!h->copy_in) {
        e = cudaStreamCreateWithFlags(&h->copy_in, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->copy_out, cudaStreamNonBlocking);
        for (auto &ev : h->ev_host)
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e != cudaSuccess) return cuda_fail("stream / event creation", e);
    }
    // The result is that of the batch's two halves as calls of their own.  Three chunks give the same bits: their
    // tokens take over the halves' routers and slices, the middle chunk's in two parts where these differ, and
    // nothing else of a token's result depends on the tokens around it.  (Two chunks where the halves differ and
    // three: 8400 tokens 1264, 1240 us a call; 9300 1389, 1288; 11,400 1659, 1474; 17,000 2439, 2138.)
    const int T0 = (T / 2 + 255) / 256 * 256;  // first token of the second half
    const bool three = T >= kHostThreeChunksMinTokens;
    const int chunks = three ? kHostMaxChunks : 2;
    int at[kHostMaxChunks + 1] = {0};  // first token of each chunk
    for (int i = 1; i < chunks; ++i) at[i] = (int)(((long long)T * i / chunks + 255) / 256 * 256);
    at[chunks] = T;
    const char *xh = static_cast<const char *>(x_host);
    char *yh = static_cast<char *>(y_host);
    __nv_bfloat16 *xs = h->ws.x_stage, *ys = h->ws.y_stage;
    cudaEvent_t start = h->ev_host[0], done = h->ev_host[1], *copied = h->ev_host + 2, *computed = copied + kHostMaxChunks;
    bool ok = cudaEventRecord(start, s) == cudaSuccess && cudaStreamWaitEvent(h->copy_in, start, 0) == cudaSuccess &&
              cudaStreamWaitEvent(h->copy_out, start, 0) == cudaSuccess;
    for (int i = 0; i < chunks; ++i)
        ok = ok &&
             cudaMemcpyAsync(xs + (size_t)at[i] * h->cfg.d_model, xh + at[i] * row, (at[i + 1] - at[i]) * row, cudaMemcpyHostToDevice,
                             h->copy_in) == cudaSuccess &&
             cudaEventRecord(copied[i], h->copy_in) == cudaSuccess;
    if (!ok) return cuda_fail("copy of x to the device", cudaGetLastError());
    int launches = 0;
    for (int i = 0; i < chunks; ++i) {
        const size_t off = (size_t)at[i] * h->cfg.d_model;
        if (cudaStreamWaitEvent(s, copied[i], 0) != cudaSuccess) return cuda_fail("cudaStreamWaitEvent", cudaGetLastError());
        const ChunkOf of = {at[i] < T0 ? T0 - at[i] : 0, T0, T - T0};
        const zeda_status_t st = forward_device(h, xs + off, at[i + 1] - at[i], ys + off, s, nullptr, 0.f, &of);
        if (st != ZEDA_OK) return st;
        launches += h->last_launches;
        if (cudaEventRecord(computed[i], s) != cudaSuccess) return cuda_fail("cudaEventRecord", cudaGetLastError());
    }
    h->last_launches = launches;
    for (int i = 0; i < chunks; ++i)  // behind all launches: a copy into pageable memory holds the host up
        ok = ok && cudaStreamWaitEvent(h->copy_out, computed[i], 0) == cudaSuccess &&
             cudaMemcpyAsync(yh + at[i] * row, ys + (size_t)at[i] * h->cfg.d_model, (at[i + 1] - at[i]) * row, cudaMemcpyDeviceToHost,
                             h->copy_out) == cudaSuccess;
    if (!ok || cudaEventRecord(done, h->copy_out) != cudaSuccess) return cuda_fail("copy of y to the host", cudaGetLastError());
    zeda_status_t routed = ZEDA_OK;
    if (three) {  // the handle keeps the second half's routing: routed again under the copies back
        RouteOut none = {};
        const int n = route_into(h, xs + (size_t)T0 * h->cfg.d_model, nullptr, T - T0, none, s);
        if (n < 0) routed = cuda_fail("routing launch", cudaGetLastError());
        else h->last_launches += n;
    }
    e = cudaEventSynchronize(done);  // (also behind a failed launch: the copies write the caller's buffer)
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (routed != ZEDA_OK) return routed;
    if (e != cudaSuccess) return cuda_fail("cudaStreamSynchronize", e);
    return ZEDA_OK;
}

zeda_status_t zeda_ep_dispatch(zeda_moe_t *h, const void *x, int32_t T, void *send_rows, int32_t *send_counts,
                               int32_t *expert_counts, void *stream) {
    zeda_status_t st = check_call(h, x, T, "x");
    if (st != ZEDA_OK) return st;
    if (h->cfg.ep_size < 1) { set_error("the handle was not created for expert parallelism (ep_size = 0)"); return ZEDA_ERR_INVALID_ARG; }
    if (!send_counts) { set_error("send_counts is NULL"); return ZEDA_ERR_INVALID_ARG; }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (T == 0) {  // nothing to route: this rank sends no rows
        cudaError_t e = cudaMemsetAsync(send_counts, 0, sizeof(int32_t) * h->cfg.ep_size, s);
        if (e == cudaSuccess && expert_counts) e = cudaMemsetAsync(expert_counts, 0, sizeof(int32_t) * h->cfg.n_real, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(h->ws.meta + kMetaPairs, 0, sizeof(int32_t), s);
        return e == cudaSuccess ? ZEDA_OK : cuda_fail("cudaMemsetAsync", e);
    }
    if (!send_rows || !aligned16(send_rows)) { set_error("send_rows is NULL or not 16-byte aligned"); return ZEDA_ERR_INVALID_ARG; }
    RouteOut none = {};
    int n = route_into(h, static_cast<const __nv_bfloat16 *>(x), nullptr, T, none, s);
    if (n < 0) return cuda_fail("routing launch", cudaGetLastError());
    int r = launch_ep_pack(h, static_cast<const __nv_bfloat16 *>(x), T, static_cast<__nv_bfloat16 *>(send_rows), send_counts,
                           expert_counts, s);
    if (r < 0) return cuda_fail("pack launch", cudaGetLastError());
    h->last_launches = n + r;
    return ZEDA_OK;
}

zeda_status_t zeda_ep_experts(zeda_moe_t *h, const void *recv_rows, const int32_t *recv_counts, int32_t n_rows,
                              void *out_rows, void *stream) {
    if (!h) { set_error("handle is NULL"); return ZEDA_ERR_INVALID_ARG; }
    if (h->cfg.ep_size < 1) { set_error("the handle was not created for expert parallelism (ep_size = 0)"); return ZEDA_ERR_INVALID_ARG; }
    if (n_rows < 0 || n_rows > h->cfg.max_recv_pairs) {
        set_error("n_rows=%d outside [0, max_recv_pairs=%d]", n_rows, h->cfg.max_recv_pairs);
        return ZEDA_ERR_INVALID_ARG;
    }
    if (n_rows == 0) return ZEDA_OK;
    if (!recv_rows || !recv_counts || !out_rows || !aligned16(recv_rows) || !aligned16(out_rows)) {
        set_error("recv_rows, recv_counts and out_rows are required; rows 16-byte aligned");
        return ZEDA_ERR_INVALID_ARG;
    }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int tile_rows = ep_tile_rows_for(h, n_rows);
    int n = launch_ep_plan(h, recv_counts, n_rows, tile_rows, s);
    if (n < 0) return cuda_fail("plan launch", cudaGetLastError());
    const Workspace &ws = h->ws;
    const ExpertWork work = {ws.ep_counts, ws.ep_offsets, ws.ep_tile_expert, ws.ep_tile_row0, ws.ep_pair_row, n_rows, tile_rows};
    int r = launch_experts_gemm1_pair(h, static_cast<const __nv_bfloat16 *>(recv_rows), work, s);
    if (r < 0) return cuda_fail("expert GEMM1 launch", cudaGetLastError());
    n += r;
    r = launch_experts_gemm2_pair(h, work, static_cast<__nv_bfloat16 *>(out_rows), s);
    if (r < 0) return cuda_fail("expert GEMM2 launch", cudaGetLastError());
    h->last_launches = n + r;
    return ZEDA_OK;
}

zeda_status_t zeda_ep_combine(zeda_moe_t *h, const void *x, const void *back_rows, int32_t T, void *y, void *stream) {
    zeda_status_t st = check_call(h, x, T, "x");
    if (st != ZEDA_OK || T == 0) return st;
    if (h->cfg.ep_size < 1) { set_error("the handle was not created for expert parallelism (ep_size = 0)"); return ZEDA_ERR_INVALID_ARG; }
    if (!y || !aligned16(y) || !back_rows || !aligned16(back_rows)) { set_error("back_rows and y are required, 16-byte aligned"); return ZEDA_ERR_INVALID_ARG; }
    int r = launch_combine_rows(h, static_cast<const __nv_bfloat16 *>(back_rows), static_cast<const __nv_bfloat16 *>(x), T,
                                static_cast<__nv_bfloat16 *>(y), static_cast<cudaStream_t>(stream));
    if (r < 0) return cuda_fail("combine launch", cudaGetLastError());
    h->last_launches = r;
    return ZEDA_OK;
}

zeda_status_t zeda_moe_stats(zeda_moe_t *h, const void *x, int32_t T, float *f, float *p_mean, float *out, void *stream) {
    zeda_status_t st = check_call(h, x, T, "x");
    if (st != ZEDA_OK || T == 0) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    RouteOut none = {};
    const StatsOut stats = {f, p_mean, out};
    int n = route_into(h, static_cast<const __nv_bfloat16 *>(x), nullptr, T, none, s, &stats);
    if (n < 0) return cuda_fail("routing launch", cudaGetLastError());
    h->last_launches = n;
    return ZEDA_OK;
}

zeda_status_t zeda_moe_token_zero_share(zeda_moe_t *h, int32_t T, float *r_ze, void *stream) {
    if (!h) { set_error("handle is NULL"); return ZEDA_ERR_INVALID_ARG; }
    if (T == 0) return ZEDA_OK;
    if (T < 0 || T != h->last_routed_tokens) {
        set_error("T=%d is not the token count of the last routing pass on this handle (%d)", T, h->last_routed_tokens);
        return ZEDA_ERR_INVALID_ARG;
    }
    if (!r_ze) { set_error("r_ze is NULL"); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    if (launch_token_zero_share(h, T, r_ze, static_cast<cudaStream_t>(stream)) < 0)
        return cuda_fail("token_zero_share launch", cudaGetLastError());
    return ZEDA_OK;
}

zeda_status_t zeda_moe_last_counters(zeda_moe_t *h, int64_t out[4], void *stream) {
    if (!h || !out) { set_error("NULL argument"); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    int32_t meta[kMetaCount];
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    e = cudaMemcpyAsync(meta, h->ws.meta, sizeof meta, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return cuda_fail("cudaMemcpyAsync(meta)", e);
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail("cudaStreamSynchronize", e);
    out[0] = meta[kMetaPairs];
    out[1] = meta[kMetaActive];
    out[2] = meta[kMetaZeroSlots];
    out[3] = h->last_launches;
    if (meta[kMetaError] != 0) { set_error(kDeviceFailure, meta[kMetaError]); return ZEDA_ERR_TIMEOUT; }
    return ZEDA_OK;
}

zeda_status_t zeda_moe_selftest_wait(zeda_moe_t *h, int32_t limit_us, void *stream) {
    if (!h) { set_error("handle is NULL"); return ZEDA_ERR_INVALID_ARG; }
    if (limit_us < 1 || limit_us > 100000) { set_error("limit_us must be in [1, 100000]"); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    int khz = 0;
    e = cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaDeviceGetAttribute", e);
    const long long cycles = (long long)limit_us * (khz > 0 ? khz : 1000000) / 1000;
    if (launch_wait_selftest(h, cycles, static_cast<cudaStream_t>(stream)) < 0)
        return cuda_fail("self-test launch", cudaGetLastError());
    return ZEDA_OK;
}

zeda_status_t zeda_moe_clear_error(zeda_moe_t *h, void *stream) {
    if (!h) { set_error("handle is NULL"); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    e = cudaMemsetAsync(h->ws.meta + kMetaError, 0, sizeof(int32_t), static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail("cudaMemsetAsync", e);
    return ZEDA_OK;
}

zeda_status_t zeda_moe_set_profiling(zeda_moe_t *h, int32_t enable) {
    if (!h) { set_error("handle is NULL"); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaSetDevice(h->cfg.device);
    if (e != cudaSuccess) return cuda_fail("cudaSetDevice", e);
    if (enable && !h->ev[0]) {
        for (auto &ev : h->ev) {
            e = cudaEventCreate(&ev);
            if (e != cudaSuccess) return cuda_fail("cudaEventCreate", e);
        }
    }
    h->profiling = enable != 0;
    if (!enable) h->profiled_last = false;
    return ZEDA_OK;
}

zeda_status_t zeda_moe_stage_ms(zeda_moe_t *h, float ms[ZEDA_STAGE_COUNT]) {
    if (!h || !ms) { set_error("NULL argument"); return ZEDA_ERR_INVALID_ARG; }
    if (!h->profiled_last) { set_error("the last forward call was not profiled"); return ZEDA_ERR_INVALID_ARG; }
    cudaError_t e = cudaEventSynchronize(h->ev[ZEDA_STAGE_COUNT]);
    if (e != cudaSuccess) return cuda_fail("cudaEventSynchronize", e);
    for (int i = 0; i < ZEDA_STAGE_COUNT; ++i) {
        e = cudaEventElapsedTime(&ms[i], h->ev[i], h->ev[i + 1]);
        if (e != cudaSuccess) return cuda_fail("cudaEventElapsedTime", e);
    }
    return ZEDA_OK;
}

zeda_status_t zeda_moe_destroy(zeda_moe_t *h) {
    if (!h) return ZEDA_OK;
    zeda_status_t st = ZEDA_OK;
    if (cudaSetDevice(h->cfg.device) == cudaSuccess) {
        int32_t err = 0;
        cudaError_t e = cudaDeviceSynchronize();
        if (e == cudaSuccess) e = cudaMemcpy(&err, h->ws.meta + kMetaError, 4, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) st = cuda_fail("zeda_moe_destroy", e);
        else if (err != 0) { set_error(kDeviceFailure, err); st = ZEDA_ERR_TIMEOUT; }
    }
    for (auto &ev : h->ev) if (ev) cudaEventDestroy(ev);
    for (auto &ev : h->ev_host) if (ev) cudaEventDestroy(ev);
    if (h->copy_in) cudaStreamDestroy(h->copy_in);
    if (h->copy_out) cudaStreamDestroy(h->copy_out);
    if (h->pmaps) free(h->pmaps);
    if (h->router_maps) free(h->router_maps);
    if (h->pair_router) free(h->pair_router);
    delete h;
    return st;
}

const char *zeda_last_error(void) { return g_err; }

const char *zeda_version(void) { return "zeda-moe 0.1 (sm_100a)"; }

}  // extern "C"
