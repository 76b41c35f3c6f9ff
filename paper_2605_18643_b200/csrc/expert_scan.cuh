// The expert scan shared by the routing pass and the expert-parallel plan: from per-expert pair
// counts to exclusive offsets, the counters of the call and the tile list of the expert kernels.
#pragma once

#include "zeda_internal.h"

namespace zeda {

constexpr unsigned kFull = 0xffffffffu;

struct ScanShared {
    int32_t cnt[kMaxCand];
    int32_t off[kMaxCand + 1];
    int32_t ptile[kMaxCand + 1];  // exclusive scan of the experts' tile counts
    int4 chunk[kMaxCand / 32];    // per 32 experts: pairs, tiles, active experts, most pairs of one expert
};

// From per-expert pair counts in sh.cnt: exclusive offsets, P, U, and the tile list of the expert
// kernels (experts in id order, each with its tiles of tile_rows rows in row order; the last tile of
// an expert may be ragged).  Called by every thread of the CTA (blockDim.x >= 32); contains CTA
// barriers.
__device__ __forceinline__ void finish_expert_scan(ScanShared &sh, int n_real, int total_slots,
                                                   int32_t *__restrict__ counts, int32_t *__restrict__ offsets,
                                                   int32_t *__restrict__ n_pairs_out, int32_t *__restrict__ meta,
                                                   const WorkLists &wl, bool write_global = true,
                                                   int list_part = 0, int list_parts = 1, int tile_rows = kPairTileM) {
    // every warp scans chunks of 32 experts with shuffle prefix sums (a single warp walking all chunks is a
    // chain of 4 x 17 dependent shuffles for 128 experts); the chunk totals are then added up by every thread
    const int lane = threadIdx.x & 31, n_chunks = (n_real + 31) / 32;
    for (int ch = threadIdx.x >> 5; ch < n_chunks; ch += blockDim.x >> 5) {
        const int i = 32 * ch + lane;
        const int c = (i < n_real) ? sh.cnt[i] : 0;
        const int pt = (c + tile_rows - 1) / tile_rows;
        int so = c, sp = pt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(kFull, so, o);
            const int q = __shfl_up_sync(kFull, sp, o);
            if (lane >= o) { so += a; sp += q; }
        }
        const int active = __popc(__ballot_sync(kFull, c > 0)), mx = __reduce_max_sync(kFull, c);
        if (i < n_real) {
            sh.off[i] = so - c;
            sh.ptile[i] = sp - pt;
        }
        if (lane == 31) sh.chunk[ch] = make_int4(so, sp, active, mx);
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= n_real; i += blockDim.x) {  // entry n_real: the totals
        int off = 0, tiles = 0, active = 0, max_rows = 0;
        const int before = i < n_real ? i >> 5 : n_chunks;
        for (int ch = 0; ch < before; ++ch) {
            const int4 v = sh.chunk[ch];
            off += v.x;
            tiles += v.y;
            active += v.z;
            max_rows = max(max_rows, v.w);
        }
        if (i < n_real) {
            sh.off[i] += off;
            sh.ptile[i] += tiles;
        } else {
            sh.off[n_real] = off;
            sh.ptile[n_real] = tiles;
            if (write_global) {
                meta[kMetaPairs] = off;
                meta[kMetaActive] = active;
                meta[kMetaZeroSlots] = total_slots - off;
                meta[kMetaPairTiles] = tiles;
                meta[kMetaMaxRows] = max_rows;
                meta[kMetaNextItem1] = 0;
                meta[kMetaNextItem2] = 0;
                if (n_pairs_out) *n_pairs_out = off;
            }
        }
    }
    __syncthreads();
    if (write_global) {  // (uniform over the CTA)
        for (int e = threadIdx.x; e < n_real; e += blockDim.x) {
            if (counts) counts[e] = sh.cnt[e];
            offsets[e] = sh.off[e];
        }
        if (threadIdx.x == 0) offsets[n_real] = sh.off[n_real];
    }
    // Tile list: every CTA that runs this scan holds the same prefix sums, so the CTAs share the
    // filling (part list_part of list_parts); a CTA outside that sharing passes list_parts = 0.
    if (list_parts <= 0) return;
    // entry i belongs to the expert whose first-entry index is the last one <= i
    const int total = sh.ptile[n_real];
    for (int i = list_part * blockDim.x + threadIdx.x; i < total; i += list_parts * blockDim.x) {
        int lo = 0, hi = n_real;  // invariant: ptile[lo] <= i < ptile[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (sh.ptile[mid] <= i) lo = mid; else hi = mid;
        }
        wl.ptile_expert[i] = lo;
        wl.ptile_row0[i] = (i - sh.ptile[lo]) * tile_rows;
    }
}

}  // namespace zeda
