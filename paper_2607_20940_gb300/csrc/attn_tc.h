// Tensor-core MSSA attention (tcgen05 + TMA) launcher interface.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "kernels.h"

namespace msf {

// Tensor-map slots of the context segments.
enum : int { kMapSink = 0, kMapHist = 1, kMapWin = 2, kMapPyr0 = 3 };
// Segments of groups with a pyramid part use map kMapPyr0 + group index;
// build_attn_args marks them kMapPyr and the launcher resolves the slot.
constexpr int kMapPyr = -1;
constexpr int kNumMaps = kMapPyr0 + MSF_MAX_GROUPS;

// What the attention kernels know of a query group: its context as 128-row
// tiles of up to three segments.
struct TcSeg {
    int map;
    int row0;
    int len;
    int tile0;  // first tile of this segment in the item's tile sequence
};
struct TcGroup {
    int q_begin, q_end;
    int n_qb;        // 256-row query blocks
    int n_items;     // B * H * n_qb
    int n_seg;
    int n_tiles;     // tiles per item
    int n_virt;      // item stride in the tile sequence: n_tiles + lead tiles
    long long tile_base;  // first tile of this group in the global sequence
    int item_base;        // first item index of this group (merge counters)
    TcSeg seg[kMaxSeg];
};
struct TcMaps {
    CUtensorMap q;
    CUtensorMap k[kNumMaps];
    CUtensorMap v[kNumMaps];
};

// What a bf16 attention call does on a device with `sms` SMs (host only).
struct AttnRoute {
    int cluster;    // > 0: the small-call kernel with clusters of so many CTAs
    int whole;      // 1: the persistent kernel on whole blocks, 0: on an even split
    int ctas;       // CTAs of the persistent kernel
    int dp_rounds;  // even split: rounds of whole blocks before it
    int pieces;     // most pieces of a block of the split (attn_route only)
};
AttnRoute attn_route(const Plan& P, const AttnArgs& a, int sms);

// With `pool` (bf16 jobs), the launch also builds that K/V pyramid: every CTA
// pools a share of it first, and tiles of pyramid segments wait until all
// shares are written.
msf_status launch_attn_tc(msf_plan_t plan, const AttnArgs& a, cudaStream_t st,
                          const PoolBatch* pool = nullptr);
// Tensor map of a [B, rows, H, D] bf16 tensor as 4-D {D, H, rows, B}, boxes of
// 64 x 1 x 128 x 1 with 128-byte swizzle (one K-major MMA chunk); rows past
// `rows` load as zeros.
bool encode_rows(CUtensorMap* m, const void* base, int D, int H, int rows, int B,
                 long long bstride_bytes);
void tc_cache_free(msf_plan_t plan);
void tc_cache_invalidate(msf_plan_t plan);

}  // namespace msf
