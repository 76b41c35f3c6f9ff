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
    static_assert((kPairTileM & (kPairTileM - 1)) == 0 && (kMidTileM & (kMidTileM - 1)) == 0, "tile heights are powers of two");
    const int tile_shift = 31 - __clz(tile_rows);
    // One warp, each lane a run of consecutive experts: one shuffle prefix sum whatever n_real is.  (All warps over
    // chunks of 32 experts and their totals behind one more barrier: 0.3 us longer up to 64 experts.)
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, run = (n_real + 31) / 32, e0 = min(n_real, lane * run), e1 = min(n_real, e0 + run);
        int pairs = 0, tiles = 0, active = 0, max_rows = 0;
#pragma unroll 4
        for (int e = e0; e < e1; ++e) {
            const int c = sh.cnt[e];
            pairs += c;
            tiles += (c + tile_rows - 1) >> tile_shift;
            active += c > 0 ? 1 : 0;
            max_rows = max(max_rows, c);
        }
        int so = pairs, sp = tiles;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(kFull, so, o);
            const int q = __shfl_up_sync(kFull, sp, o);
            if (lane >= o) { so += a; sp += q; }
        }
        int off = so - pairs, first = sp - tiles;
#pragma unroll 4
        for (int e = e0; e < e1; ++e) {
            const int c = sh.cnt[e];
            sh.off[e] = off;
            sh.ptile[e] = first;
            off += c;
            first += (c + tile_rows - 1) >> tile_shift;
        }
        active = __reduce_add_sync(kFull, active);
        max_rows = __reduce_max_sync(kFull, max_rows);
        if (lane == 31) {
            sh.off[n_real] = so;
            sh.ptile[n_real] = sp;
            if (write_global) {
                meta[kMetaPairs] = so;
                meta[kMetaActive] = active;
                meta[kMetaZeroSlots] = total_slots - so;
                meta[kMetaPairTiles] = sp;
                meta[kMetaMaxRows] = max_rows;
                meta[kMetaNextItem1] = 0;
                meta[kMetaNextItem2] = 0;
                if (n_pairs_out) *n_pairs_out = so;
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
