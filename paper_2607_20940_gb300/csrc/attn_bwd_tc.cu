// MSSA backward on the sm_103a tensor cores (bf16 operands, fp32 accumulation).
//
// Same mathematics as the CUDA-core backward (attn_bwd.cu): with the
// forward's row log-sum-exp, P = exp(c S - lse) is rebuilt tile by tile and
//   dS = P * (dP - delta),  dP = dO V^T,  delta = rowsum(dO * O)
//   dQ = c dS K,  dK = c dS^T Q,  dV = P^T dO.
// One persistent launch (a CTA per SM) runs two kinds of items, no atomics:
//
// dq item: a 128-row query tile of one (stream, head, group). It walks the
//   group's whole context (sink, history or pyramid part, window suffix) in
//   128-row K/V tiles:
//     S = Q K^T (SS, two buffers), dP = dO V^T (SS)  -> TMEM
//     softmax warps: dS (bf16, over S's columns)      -> TMEM
//     dQ += dS K (TS, K read MN-major)               -> TMEM
//   then scales dQ by c and stores it.
// dk/dv item: a 128-row tile of context rows that come from the window. It
//   walks its group's queries in 128-row tiles:
//     S^T = K Q^T (SS), dP^T = V dO^T (SS)            -> TMEM (lanes = keys)
//     softmax warps: P^T over S^T, then dS^T over dP^T -> TMEM
//     dV += P^T dO (TS), dK += dS^T Q (TS)           -> TMEM
//   then writes c dK and dV (fp32) to its rows of the context-gradient
//   buffers. A gather kernel applies the adjoint of Subsample afterwards.
//
// CTA c takes items c, 2G-1-c, 2G+c, ... of the list sorted by cost (G CTAs,
// back and forth so that no CTA always gets a round's longest), or a list of its
// own where that ends earlier (place_items), and its roles run on from item to
// item: the next item's loads and first MMAs overlap the
// output of the one before, and tensor memory and barriers are set up once.
// On the 480p layer an item used to cost 5-9 us besides its tiles.
//
// Roles (384 threads): warp 0 TMA producer, warp 1 MMA issuer (warp-wide
// loop, one elected lane issues), warp 2 TMEM allocation, warps 4-11 the
// softmax: a thread per TMEM lane (query row or key row) and column half,
// warps 4-7 columns 0-63, warps 8-11 columns 64-127. Each half writes its
// bf16 P / dS into its own columns (the MMA that reads them takes its A
// operand per 16-column step), so the halves never wait for each other.
// The tensor pipe executes MMAs in issue order, so an MMA that overwrites S
// or dP never overtakes the MMA that reads the bf16 P or dS stored there.
// Every wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "attn_bwd_tc.h"
#include "attn_tc.h"
#include "bwd_items.h"
#include "ptx.cuh"

namespace msf {
namespace {

constexpr int kBM = 128;       // rows of every Q / dO / K / V tile
constexpr int kThreads = 384;  // 12 warps
constexpr long long kWaitLimit = 2000000000LL;  // ~1 s of SM clock
constexpr float kLog2e = 1.4426950408889634f;

struct BSeg {
    int map, row0, len, tile0;
};
struct BGroupQ {
    int q_begin, q_end;
    int n_qt;  // 128-row query tiles
    int n_seg, n_tiles;
    BSeg seg[kMaxSeg];
};
struct BGrad {
    int map, row0, len, kt0;  // row0 relative to the map; kt0 = first key tile of the run
    int crow0;                // first row of the run in the context-gradient buffers
};
struct BGroupK {
    int q_begin, q_end, n_qt;
    int n_kt;  // key tiles of this group (all runs)
    int n_grad;
    BGrad gr[kMaxGradSeg];
};
struct BwdTcParams {
    int H, B, N;
    float scale, scale_log2;
    const float* lse;
    const float* delta;
    __nv_bfloat16* dq;
    float* dk_ctx;
    float* dv_ctx;
    int R;  // rows per stream of the context-gradient buffers
    unsigned int* status;
    long long wait_limit;
    int dq_v8, ctx_v8;  // 32-byte aligned outputs: 32-byte stores
    int n_items;
    // dq work
    BGroupQ g[MSF_MAX_GROUPS];
    // dK/dV work
    BGroupK kg[MSF_MAX_GROUPS];
    // Item ranges, most expensive items first: kind 0 =
    // dq items of group g[group], kind 1 = dK/dV items of kg[group].
    int n_ranges;
    struct Range {
        int kind, group, base;
    } range[2 * MSF_MAX_GROUPS];
};
struct BwdMaps {
    CUtensorMap q, dout;
    CUtensorMap k[kNumMaps];
    CUtensorMap v[kNumMaps];
};

// Barriers of the roles; an index counts phases from the launch's start.
struct BwdBars {
    // dq items: Q and dO, the K and V rings, S + dP ready, dP read, dS written, dQ complete
    uint64_t qg_full, qg_empty, k_full[3], k_empty[3], v_full[2], v_empty[2];
    // (ds_full by tile parity: dP_{j+1} may be read by one warp before another
    // has written dS_j)
    uint64_t sdp_full, dp_free, ds_full[2], dq_full;
    // dk/dv items: K, V, the Q and dO rings, S^T ready, P^T written, dP^T
    // ready, dS^T written, dV and dK complete; the warps of a half meet
    uint64_t kst_full, kst_empty, vst_full, vst_empty, q_full[3], q_empty[3], g_full[2], g_empty[2];
    uint64_t st_full, p_full, dpt_full, dst_full, kv_full, meet[2];
    uint64_t item_done[kDoneBars], drain;
    uint32_t tmem_base;
    int abort_flag;
};

// Dynamic shared memory of the launch (no static part, so that its base is
// 1024-byte aligned): seven 128 x D bf16 tiles (dq items: Q, dO, a 3-deep K
// ring and a 2-deep V ring; dk/dv items: K, V, a 3-deep Q ring and a 2-deep
// dO ring), the per-query statistics of two query tiles, the barriers. At
// least 120 KB, so that one CTA (and one 512-column TMEM allocation) sits on
// an SM.
template <int D>
struct BCfg {
    static constexpr int kTile = kBM * D * 2;
    static constexpr int kStats = 7 * kTile;
    static constexpr int kBars = kStats + 4 * kBM * 4;
    static constexpr int kUsed = kBars + (int)sizeof(BwdBars);
    static constexpr int kSmem = kUsed > 120 * 1024 ? kUsed : 120 * 1024;
};
static_assert(BCfg<128>::kSmem <= 227 * 1024, "shared memory of the launch");

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// K-step offset (16-byte units) inside a K-major SW128 tile of 128 rows.
__device__ __forceinline__ uint64_t kmajor_step(int kk) {
    constexpr int kChunk = kBM * 128;
    return (uint64_t)(((kk / 4) * kChunk + (kk % 4) * 32) >> 4);
}

// 128 rows x D of a [B, rows, H, D] tensor: D/64 swizzled boxes.
template <int D>
__device__ __forceinline__ void load_tile(unsigned char* dst, const CUtensorMap* m, uint64_t* bar,
                                          int h, int row, int b) {
#pragma unroll
    for (int c = 0; c < D / 64; ++c) ptx::tma_load_4d(dst + c * (kBM * 128), m, bar, c * 64, h, row, b);
}

// The parts of an item that every role needs.
struct BItem {
    int kind, gi;
    int h, b;
    int n;     // tiles it walks: K/V tiles (dq), query tiles (dk/dv)
    int row0;  // dq: first query; dk/dv: first context row in its tensor map
    int map;   // dk/dv: tensor map of K and V
    int crow;  // dk/dv: first row in the context-gradient buffers
    int rows;  // valid rows of the own tile
};

__device__ __forceinline__ BItem item_of(const BwdTcParams& p, int idx) {
    int r = 0;
    while (r + 1 < p.n_ranges && idx >= p.range[r + 1].base) ++r;
    const int local = idx - p.range[r].base;
    BItem it;
    it.kind = p.range[r].kind;
    it.gi = p.range[r].group;
    if (it.kind == 0) {
        const BGroupQ& G = p.g[it.gi];
        const int qt = local % G.n_qt;
        it.h = (local / G.n_qt) % p.H;
        it.b = local / (G.n_qt * p.H);
        it.n = G.n_tiles;
        it.row0 = G.q_begin + qt * kBM;
        it.map = 0;
        it.crow = 0;
        it.rows = min(kBM, G.q_end - it.row0);
    } else {
        const BGroupK& K = p.kg[it.gi];
        const int kt_all = local % K.n_kt;
        it.h = (local / K.n_kt) % p.H;
        it.b = local / (K.n_kt * p.H);
        int s = 0;
        while (s + 1 < K.n_grad && kt_all >= K.gr[s + 1].kt0) ++s;
        const int off = (kt_all - K.gr[s].kt0) * kBM;
        it.n = K.n_qt;
        it.row0 = K.gr[s].row0 + off;
        it.map = K.gr[s].map;
        it.crow = K.gr[s].crow0 + off;
        it.rows = min(kBM, K.gr[s].len - off);
    }
    return it;
}

// K/V tile u of a dq item of group G.
__device__ __forceinline__ void kv_tile(const BGroupQ& G, int u, int& map, int& row, int& valid) {
    int s = 0;
    while (s < G.n_seg - 1 && u >= G.seg[s + 1].tile0) ++s;
    const int kt = u - G.seg[s].tile0;
    map = G.seg[s].map;
    row = G.seg[s].row0 + kt * kBM;
    valid = min(kBM, G.seg[s].len - kt * kBM);
}

// k-th item of this CTA (n_items or more: none left).
__device__ __forceinline__ int next_item(const BwdTcParams& p, const BwdOrder& o, int k) {
    const int g = (int)gridDim.x, c = (int)blockIdx.x;
    if (!o.on) return k * g + ((k & 1) ? g - 1 - c : c);
    const int at = o.first[c] + k;
    return at < o.first[c + 1] ? o.item[at] : p.n_items;
}

// 64 fp32 columns of a row scaled by mul: 32-byte stores when aligned.
__device__ __forceinline__ void store_f32(float* dst, const uint32_t (&o)[32], float mul, bool v8) {
    uint32_t x[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) x[e] = __float_as_uint(__uint_as_float(o[e]) * mul);
    if (v8) {
#pragma unroll
        for (int e = 0; e < 4; ++e) ptx::st_global_v8(dst + 8 * e, x + 8 * e);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
            reinterpret_cast<uint4*>(dst)[e] = make_uint4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]);
    }
}

// TMEM columns, dq items: S of even tiles [0,128), of odd tiles [128,256), dP
// [256,384), dQ from 384. The softmax warps first copy dP_j into registers and
// release it, so dP_{j+1} (and S_{j+1}, issued a tile ahead into the other S
// buffer) run on the tensor pipe while they compute dS_j; dQ_j and S_{j+2}
// then run while the softmax works on tile j+1.
// dk/dv items: S^T [0,128), dP^T [128,256), dV from 256, dK from 256 + D. Two
// phases per query tile keep the pipe busy: once P^T_i is written, dV_i and
// S^T_{i+1} run while the softmax turns dP^T_i into dS^T_i; then dK_i and
// dP^T_{i+1} run while it turns S^T_{i+1} into P^T_{i+1}. All MMAs are 128
// columns wide: the two 64-query halves of the version before had 64-wide ones
// with both operands in shared memory, whose reads bound them (a probe that only
// issues MMAs: 48 cycles against 64 of a 128-wide one).
template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    bwd_tc_kernel(const __grid_constant__ BwdMaps maps, const __grid_constant__ BwdTcParams p,
                  const __grid_constant__ BwdOrder order) {
    using C = BCfg<D>;
    extern __shared__ __align__(1024) unsigned char smem[];
    BwdBars& bar = *reinterpret_cast<BwdBars*>(smem + C::kBars);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (ptx::smem_u32(smem) & 1023u) {  // the swizzled tiles need it
        if (threadIdx.x == 0) atomicOr(p.status, kDevTimeout);
        return;
    }
    if (threadIdx.x == 0) {
        bar.abort_flag = 0;
        uint64_t* one[] = {&bar.qg_full, &bar.qg_empty, &bar.sdp_full, &bar.dq_full, &bar.kst_full, &bar.kst_empty,
                           &bar.vst_full, &bar.vst_empty, &bar.st_full, &bar.dpt_full, &bar.kv_full, &bar.drain};
        for (uint64_t* x : one) ptx::mbar_init(x, 1);
        for (int s = 0; s < 3; ++s) {
            ptx::mbar_init(&bar.k_full[s], 1);
            ptx::mbar_init(&bar.k_empty[s], 1);
            ptx::mbar_init(&bar.q_full[s], 1);
            ptx::mbar_init(&bar.q_empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(&bar.v_full[s], 1);
            ptx::mbar_init(&bar.v_empty[s], 1);
            ptx::mbar_init(&bar.g_full[s], 1);
            ptx::mbar_init(&bar.g_empty[s], 1);
            ptx::mbar_init(&bar.meet[s], 4);
        }
        ptx::mbar_init(&bar.dp_free, 8);
        ptx::mbar_init(&bar.ds_full[0], 8);
        ptx::mbar_init(&bar.ds_full[1], 8);
        ptx::mbar_init(&bar.p_full, 8);
        ptx::mbar_init(&bar.dst_full, 8);
        for (int s = 0; s < kDoneBars; ++s) ptx::mbar_init(&bar.item_done[s], 8);
        ptx::fence_mbar_init();
    }
    if (warp == 2) {
        ptx::tmem_alloc(&bar.tmem_base, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tbase = bar.tmem_base;
    volatile int* abort_p = &bar.abort_flag;
    volatile int never = 0;
    // Only delta comes from the launch right before this one (bwd_delta_kernel,
    // on every path), and that launch let this one start after its own wait,
    // when q, k, v, dO and lse were complete: the softmax warps wait, the first
    // loads and MMAs need not.
    ptx::grid_dep_launch();

    if (warp == 0) {
        // ============================ TMA producer ============================
        if (lane == 0) {
            bool ok = true;
            // tiles issued so far to each ring, items of each kind
            int nk = 0, nv = 0, nq = 0, ng = 0, n_dq = 0, n_kst = 0, n_vst = 0;
            auto take = [&](uint64_t* empty, uint32_t parity) {
                ok = ok && ptx::mbar_wait_bounded(empty, parity, abort_p, p.wait_limit);
                return ok;
            };
            int prev_kind = -1;
            for (int k = 0; ok; ++k) {
                const int idx = next_item(p, order, k);
                if (idx >= p.n_items) break;
                const BItem it = item_of(p, idx);
                // The item before the last is done (so that every phase of
                // item_done is seen); on a change of kind the last one too,
                // whose tiles this one's overwrite.
                auto done = [&](int i) { return take(&bar.item_done[done_bar(i)], done_parity(i)); };
                if (k >= 2 && !done(k - 2)) break;
                if (k >= 1 && it.kind != prev_kind && !done(k - 1)) break;
                prev_kind = it.kind;
                if (it.kind == 0) {
                    const BGroupQ& G = p.g[it.gi];
                    if (!take(&bar.qg_empty, (uint32_t)((n_dq & 1) ^ 1))) break;
                    ptx::mbar_arrive_expect_tx(&bar.qg_full, 2 * C::kTile);
                    load_tile<D>(smem, &maps.q, &bar.qg_full, it.h, it.row0, it.b);
                    load_tile<D>(smem + C::kTile, &maps.dout, &bar.qg_full, it.h, it.row0, it.b);
                    ++n_dq;
                    for (int j = 0; j < it.n; ++j) {
                        int map, row, valid;
                        kv_tile(G, j, map, row, valid);
                        const int ks = nk % 3, vs = nv & 1;
                        if (!take(&bar.k_empty[ks], (uint32_t)(((nk / 3) & 1) ^ 1))) break;
                        ptx::mbar_arrive_expect_tx(&bar.k_full[ks], C::kTile);
                        load_tile<D>(smem + (2 + ks) * C::kTile, &maps.k[map], &bar.k_full[ks], it.h, row, it.b);
                        ++nk;
                        if (!take(&bar.v_empty[vs], (uint32_t)(((nv >> 1) & 1) ^ 1))) break;
                        ptx::mbar_arrive_expect_tx(&bar.v_full[vs], C::kTile);
                        load_tile<D>(smem + (5 + vs) * C::kTile, &maps.v[map], &bar.v_full[vs], it.h, row, it.b);
                        ++nv;
                    }
                } else {
                    const BGroupK& K = p.kg[it.gi];
                    if (!take(&bar.kst_empty, (uint32_t)((n_kst & 1) ^ 1))) break;
                    ptx::mbar_arrive_expect_tx(&bar.kst_full, C::kTile);
                    load_tile<D>(smem, &maps.k[it.map], &bar.kst_full, it.h, it.row0, it.b);
                    ++n_kst;
                    for (int i = 0; i < it.n; ++i) {
                        const int qs = nq % 3, gs = ng & 1, row = K.q_begin + i * kBM;
                        if (!take(&bar.q_empty[qs], (uint32_t)(((nq / 3) & 1) ^ 1))) break;
                        ptx::mbar_arrive_expect_tx(&bar.q_full[qs], C::kTile);
                        load_tile<D>(smem + (2 + qs) * C::kTile, &maps.q, &bar.q_full[qs], it.h, row, it.b);
                        ++nq;
                        if (i == 0) {
                            if (!take(&bar.vst_empty, (uint32_t)((n_vst & 1) ^ 1))) break;
                            ptx::mbar_arrive_expect_tx(&bar.vst_full, C::kTile);
                            load_tile<D>(smem + C::kTile, &maps.v[it.map], &bar.vst_full, it.h, it.row0, it.b);
                            ++n_vst;
                        }
                        if (!take(&bar.g_empty[gs], (uint32_t)(((ng >> 1) & 1) ^ 1))) break;
                        ptx::mbar_arrive_expect_tx(&bar.g_full[gs], C::kTile);
                        load_tile<D>(smem + (5 + gs) * C::kTile, &maps.dout, &bar.g_full[gs], it.h, row, it.b);
                        ++ng;
                    }
                }
            }
            if (!ok) {
                // every copy issued lands before the CTA exits
                auto landed = [&](uint64_t* full, int n) {
                    if (n > 0) ptx::mbar_wait_bounded(full, (uint32_t)((n - 1) & 1), &never, kWaitLimit);
                };
                landed(&bar.qg_full, n_dq);
                landed(&bar.kst_full, n_kst);
                landed(&bar.vst_full, n_vst);
                for (int s = 0; s < 3; ++s) {
                    landed(&bar.k_full[s], (nk + 2 - s) / 3);
                    landed(&bar.q_full[s], (nq + 2 - s) / 3);
                }
                for (int s = 0; s < 2; ++s) {
                    landed(&bar.v_full[s], (nv + 1 - s) / 2);
                    landed(&bar.g_full[s], (ng + 1 - s) / 2);
                }
                atomicOr(p.status, kDevTimeout);
            }
        }
    } else if (warp == 1) {
        // ============================= MMA issuer =============================
        // Two probe points per tile. A tcgen05.mma holds its issuing thread
        // about as long as the tensor pipe takes to run it, and only ~250
        // cycles of work stay in flight after the last issue, so every
        // barrier check here is pipe time: the probes of each point go out
        // together, and the bounded waits run only if one is not ready.
        constexpr uint32_t idS = ptx::idesc_bf16(kBM, kBM, false, false);
        constexpr uint32_t idO = ptx::idesc_bf16(kBM, D, false, true);
        constexpr uint64_t kTileDesc = (uint64_t)(C::kTile >> 4);
        const uint64_t desc = ptx::sdesc_sw128(ptx::smem_u32(smem), 16, 1024);          // tile 0, K-major
        const uint64_t desc_mn = ptx::sdesc_sw128(ptx::smem_u32(smem), kBM * 128, 1024);  // tile 0, MN-major
        auto wait_all = [&](uint64_t* b, uint32_t parity) {
            const bool r = ptx::mbar_wait_bounded(b, parity, abort_p, p.wait_limit);
            return __all_sync(0xffffffffu, r);
        };
        // D[128 x 128] = tile a x tile b^T
        auto mma_tiles = [&](uint32_t d, int a, int b) {
            const uint64_t ad = desc + (uint64_t)a * kTileDesc, bd = desc + (uint64_t)b * kTileDesc;
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
                ptx::mma_ss(d, ad + kmajor_step(kk), bd + kmajor_step(kk), idS, kk > 0 ? 1u : 0u);
        };
        // D[128 x D] (+)= bf16 tile at TMEM column a (64 columns per half) x tile b
        auto mma_out = [&](uint32_t d, uint32_t a, int b, bool acc) {
            const uint64_t bd = desc_mn + (uint64_t)b * kTileDesc;
#pragma unroll
            for (int kk = 0; kk < kBM / 16; ++kk)
                ptx::mma_ts(d, a + 64 * (kk / 4) + (kk % 4) * 8, bd + (uint64_t)(kk * (2048 >> 4)), idO,
                            (acc || kk > 0) ? 1u : 0u);
        };
        bool ok = true;
        int nk = 0, nv = 0, nq = 0, ng = 0;  // ring tiles consumed
        int tq = 0, tk = 0;                  // tiles done of each kind
        int iq = 0, ik = 0;                  // items done of each kind
        for (int k = 0; ok; ++k) {
            const int idx = next_item(p, order, k);
            if (idx >= p.n_items) break;
            const BItem it = item_of(p, idx);
            const int n = it.n;
            if (it.kind == 0) {
                auto issue_s = [&](int j) { mma_tiles(tbase + (j & 1) * 128, 0, 2 + (nk + j) % 3); };
                auto issue_dp = [&](int j) {
                    const int vs = (nv + j) & 1;
                    mma_tiles(tbase + 256, 1, 5 + vs);
                    ptx::mma_commit(&bar.v_empty[vs]);
                    ptx::mma_commit(&bar.sdp_full);
                    if (j + 1 == n) ptx::mma_commit(&bar.qg_empty);  // the last S went out before
                };
                auto k_full = [&](int j) { return &bar.k_full[(nk + j) % 3]; };
                auto k_par = [&](int j) { return (uint32_t)(((nk + j) / 3) & 1); };
                auto v_full = [&](int j) { return &bar.v_full[(nv + j) & 1]; };
                auto v_par = [&](int j) { return (uint32_t)(((nv + j) >> 1) & 1); };
                ok = wait_all(&bar.qg_full, (uint32_t)(iq & 1)) && wait_all(k_full(0), k_par(0)) &&
                     wait_all(v_full(0), v_par(0));
                if (ok) {
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) {
                        issue_s(0);
                        issue_dp(0);
                    }
                    __syncwarp();
                    if (n > 1) {
                        ok = wait_all(k_full(1), k_par(1));
                        if (ok) {
                            ptx::tc_fence_after();
                            if (ptx::elect_one_sync()) issue_s(1);
                            __syncwarp();
                        }
                    }
                }
                for (int j = 0; j < n && ok; ++j, ++tq) {
                    const bool next = j + 1 < n, next2 = j + 2 < n;
                    const uint32_t par = (uint32_t)(tq & 1);
                    {
                        const bool rd = ptx::mbar_try_wait(&bar.dp_free, par);
                        const bool rv = !next || ptx::mbar_try_wait(v_full(j + 1), v_par(j + 1));
                        if (!__all_sync(0xffffffffu, rd && rv))
                            ok = wait_all(&bar.dp_free, par) && (!next || wait_all(v_full(j + 1), v_par(j + 1)));
                    }
                    if (!ok) break;
                    if (next) {
                        ptx::tc_fence_after();
                        if (ptx::elect_one_sync()) issue_dp(j + 1);
                        __syncwarp();
                    }
                    // dS_j, and K_{j+2} for the S two tiles ahead; if K has not
                    // landed yet, dQ_j goes first and S_{j+2} after its own wait.
                    bool k_ready;
                    {
                        const uint32_t dpar = (uint32_t)((tq >> 1) & 1);
                        const bool rs = ptx::mbar_try_wait(&bar.ds_full[par], dpar);
                        k_ready = !next2 || ptx::mbar_try_wait(k_full(j + 2), k_par(j + 2));
                        k_ready = __all_sync(0xffffffffu, k_ready);
                        if (!__all_sync(0xffffffffu, rs)) ok = wait_all(&bar.ds_full[par], dpar);
                    }
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) {
                        const int ks = (nk + j) % 3;
                        mma_out(tbase + 384, tbase + (j & 1) * 128, 2 + ks, j > 0);
                        ptx::mma_commit(&bar.k_empty[ks]);
                        if (!next) ptx::mma_commit(&bar.dq_full);
                        if (next2 && k_ready) issue_s(j + 2);
                    }
                    __syncwarp();
                    if (next2 && !k_ready) {
                        ok = wait_all(k_full(j + 2), k_par(j + 2));
                        if (!ok) break;
                        ptx::tc_fence_after();
                        if (ptx::elect_one_sync()) issue_s(j + 2);
                        __syncwarp();
                    }
                }
                nk += n;
                nv += n;
                ++iq;
            } else {
                auto q_full = [&](int i) { return &bar.q_full[(nq + i) % 3]; };
                auto q_par = [&](int i) { return (uint32_t)(((nq + i) / 3) & 1); };
                auto g_full = [&](int i) { return &bar.g_full[(ng + i) & 1]; };
                auto g_par = [&](int i) { return (uint32_t)(((ng + i) >> 1) & 1); };
                auto issue_st = [&](int i) {  // S^T = K Q_i^T
                    mma_tiles(tbase, 0, 2 + (nq + i) % 3);
                    ptx::mma_commit(&bar.st_full);
                    if (i + 1 == n) ptx::mma_commit(&bar.kst_empty);
                };
                auto issue_dpt = [&](int i) {  // dP^T = V dO_i^T
                    mma_tiles(tbase + 128, 1, 5 + ((ng + i) & 1));
                    ptx::mma_commit(&bar.dpt_full);
                    if (i + 1 == n) ptx::mma_commit(&bar.vst_empty);
                };
                ok = wait_all(&bar.kst_full, (uint32_t)(ik & 1)) && wait_all(q_full(0), q_par(0));
                if (ok) {
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) issue_st(0);
                    __syncwarp();
                    ok = wait_all(&bar.vst_full, (uint32_t)(ik & 1)) && wait_all(g_full(0), g_par(0));
                }
                if (ok) {
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) issue_dpt(0);
                    __syncwarp();
                }
                for (int i = 0; i < n && ok; ++i, ++tk) {
                    const bool next = i + 1 < n;
                    const uint32_t par = (uint32_t)(tk & 1);
                    // P^T_i and the next Q: dV_i, S^T_{i+1}
                    bool ready;
                    {
                        const bool rp = ptx::mbar_try_wait(&bar.p_full, par);
                        ready = !next || ptx::mbar_try_wait(q_full(i + 1), q_par(i + 1));
                        ready = __all_sync(0xffffffffu, ready);
                        if (!__all_sync(0xffffffffu, rp)) ok = wait_all(&bar.p_full, par);
                    }
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) {
                        const int gs = (ng + i) & 1;
                        mma_out(tbase + 256, tbase, 5 + gs, i > 0);
                        ptx::mma_commit(&bar.g_empty[gs]);  // dP^T_i went out before
                        if (next && ready) issue_st(i + 1);
                    }
                    __syncwarp();
                    if (next && !ready) {
                        ok = wait_all(q_full(i + 1), q_par(i + 1));
                        if (!ok) break;
                        ptx::tc_fence_after();
                        if (ptx::elect_one_sync()) issue_st(i + 1);
                        __syncwarp();
                    }
                    // dS^T_i and the next dO: dK_i, dP^T_{i+1}
                    {
                        const bool rs = ptx::mbar_try_wait(&bar.dst_full, par);
                        ready = !next || ptx::mbar_try_wait(g_full(i + 1), g_par(i + 1));
                        ready = __all_sync(0xffffffffu, ready);
                        if (!__all_sync(0xffffffffu, rs)) ok = wait_all(&bar.dst_full, par);
                    }
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) {
                        const int qs = (nq + i) % 3;
                        mma_out(tbase + 256 + D, tbase + 128, 2 + qs, i > 0);
                        ptx::mma_commit(&bar.q_empty[qs]);
                        if (!next)
                            ptx::mma_commit(&bar.kv_full);
                        else if (ready)
                            issue_dpt(i + 1);
                    }
                    __syncwarp();
                    if (next && !ready) {
                        ok = wait_all(g_full(i + 1), g_par(i + 1));
                        if (!ok) break;
                        ptx::tc_fence_after();
                        if (ptx::elect_one_sync()) issue_dpt(i + 1);
                        __syncwarp();
                    }
                }
                nq += n;
                ng += n;
                ++ik;
            }
        }
        if (!ok) {
            if (ptx::elect_one_sync()) ptx::mma_commit(&bar.drain);
            __syncwarp();
            ptx::mbar_wait_bounded(&bar.drain, 0, &never, kWaitLimit);
            if (lane == 0) atomicOr(p.status, kDevTimeout);
        }
    } else if (warp >= 4) {
        // ============== softmax: one thread per own row and column half ==============
        const int half = (warp - 4) / 4;
        const int wq = warp % 4;
        const int r = wq * 32 + lane;
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        constexpr int DH = D / 2;  // output columns of this thread
        const uint64_t sl2x2 = ptx::f2_pack(p.scale_log2, p.scale_log2);
        bool ok = true;
        auto wait_all = [&](uint64_t* b, uint32_t parity) {
            return (bool)__all_sync(0xffffffffu, ptx::mbar_wait_bounded(b, parity, abort_p, p.wait_limit));
        };
        auto arrive = [&](uint64_t* b) {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(b);
        };
        int tq = 0, tk = 0, iq = 0, ik = 0;
        ptx::grid_dep_wait();
        for (int k = 0; ok; ++k) {
            const int idx = next_item(p, order, k);
            if (idx >= p.n_items) break;
            const BItem it = item_of(p, idx);
            const int n = it.n;
            const size_t head = ((size_t)it.b * p.H + it.h) * p.N;  // row of lse and delta
            if (it.kind == 0) {
                const BGroupQ& G = p.g[it.gi];
                const uint32_t tP = tbase + 256 + 64 * half + lane_off;
                const int q = it.row0 + r;
                const bool qv = r < it.rows;
                const float nl = qv ? -p.lse[head + q] * kLog2e : -INFINITY;  // -lse in log2 units
                const float dl = qv ? p.delta[head + q] : 0.f;
                const uint64_t nlx2 = ptx::f2_pack(nl, nl), ndlx2 = ptx::f2_pack(-dl, -dl);
                for (int j = 0; j < n; ++j, ++tq) {
                    int map, row, valid;
                    kv_tile(G, j, map, row, valid);
                    ok = wait_all(&bar.sdp_full, (uint32_t)(tq & 1));
                    if (!ok) break;
                    ptx::tc_fence_after();
                    // this half's dP_j into registers, then release its columns
                    uint32_t dp[2][32];
                    ptx::tmem_ld32(tP, dp[0]);
                    ptx::tmem_ld32(tP + 32, dp[1]);
                    ptx::tmem_wait_ld();
                    ptx::tc_fence_before();
                    arrive(&bar.dp_free);
                    const uint32_t tS = tbase + (j & 1) * 128 + 64 * half + lane_off;
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) {
                        uint32_t s[32];
                        ptx::tmem_ld32(tS + 32 * c2, s);
                        ptx::tmem_wait_ld();
                        const int lim = valid - (64 * half + 32 * c2);
                        if (lim < 32) {
                            // keys past the segment's end: score -inf, probability 0
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if (e >= lim) s[e] = 0xff800000u;
                        }
                        uint32_t pk[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const uint64_t arg = ptx::f2_fma(
                                ptx::f2_pack(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1])), sl2x2, nlx2);
                            float a0, a1;
                            ptx::f2_unpack(arg, a0, a1);
                            const uint64_t pp = ptx::f2_pack(ex2(a0), ex2(a1));
                            const uint64_t dd = ptx::f2_add(
                                ptx::f2_pack(__uint_as_float(dp[c2][2 * e]), __uint_as_float(dp[c2][2 * e + 1])),
                                ndlx2);
                            const uint64_t ds = ptx::f2_mul(pp, dd);
                            float d0, d1;
                            ptx::f2_unpack(ds, d0, d1);
                            pk[e] = ptx::pack_bf16(d0, d1);
                        }
                        ptx::tmem_st16(tS + 16 * c2, pk);
                    }
                    ptx::tmem_wait_st();
                    ptx::tc_fence_before();
                    arrive(&bar.ds_full[tq & 1]);
                }
                ok = ok && wait_all(&bar.dq_full, (uint32_t)(iq & 1));
                if (!ok) break;
                ++iq;
                // each half stores D/2 columns of its row
                ptx::tc_fence_after();
                const uint32_t tQ = tbase + 384 + DH * half + lane_off;
                __nv_bfloat16* dst = p.dq + (((size_t)it.b * p.N + (qv ? q : 0)) * p.H + it.h) * D + DH * half;
                uint32_t o[DH / 32][32];
#pragma unroll
                for (int c = 0; c < DH / 32; ++c) ptx::tmem_ld32(tQ + 32 * c, o[c]);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < DH / 32; ++c) {
                    uint32_t pk[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        pk[e] = ptx::pack_bf16(__uint_as_float(o[c][2 * e]) * p.scale,
                                               __uint_as_float(o[c][2 * e + 1]) * p.scale);
                    if (qv && p.dq_v8) {
                        ptx::st_global_v8(dst + 32 * c, pk);
                        ptx::st_global_v8(dst + 32 * c + 16, pk + 8);
                    } else if (qv) {
                        uint4* d4 = reinterpret_cast<uint4*>(dst + 32 * c);
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            d4[e] = make_uint4(pk[4 * e], pk[4 * e + 1], pk[4 * e + 2], pk[4 * e + 3]);
                    }
                }
            } else {
                const BGroupK& K = p.kg[it.gi];
                const uint32_t tS = tbase + 64 * half + lane_off, tP = tbase + 128 + 64 * half + lane_off;
                float* stats = reinterpret_cast<float*>(smem + C::kStats) + 128 * half;
                for (int i = 0; i < n; ++i, ++tk) {
                    const uint32_t par = (uint32_t)(tk & 1);
                    // This half's 64 per-query statistics, shared by its 128 key
                    // rows: threads 0-63 of the half load -lse (log2 units),
                    // 64-127 -delta, into the buffer of the tile's parity.
                    float* L = stats + 256 * par;
                    {
                        const int q = K.q_begin + i * kBM + 64 * half + (r & 63);
                        const bool qv = q < K.q_end;
                        if (r < 64)
                            L[r] = qv ? -p.lse[head + q] * kLog2e : -INFINITY;
                        else
                            L[r] = qv ? -p.delta[head + q] : 0.f;
                    }
                    arrive(&bar.meet[half]);
                    ok = wait_all(&bar.meet[half], par) && wait_all(&bar.st_full, par);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    uint64_t pf[32];  // P^T, fp32 pairs
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) {
                        uint32_t s[32], pk[16];
                        ptx::tmem_ld32(tS + 32 * c2, s);
                        ptx::tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const float2 l2 = *reinterpret_cast<const float2*>(L + 32 * c2 + 2 * e);
                            const uint64_t arg = ptx::f2_fma(
                                ptx::f2_pack(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1])), sl2x2,
                                ptx::f2_pack(l2.x, l2.y));
                            float a0, a1;
                            ptx::f2_unpack(arg, a0, a1);
                            const float p0 = ex2(a0), p1 = ex2(a1);
                            pf[16 * c2 + e] = ptx::f2_pack(p0, p1);
                            pk[e] = ptx::pack_bf16(p0, p1);
                        }
                        ptx::tmem_st16(tS + 16 * c2, pk);
                    }
                    ptx::tmem_wait_st();
                    ptx::tc_fence_before();
                    arrive(&bar.p_full);
                    ok = wait_all(&bar.dpt_full, par);
                    if (!ok) break;
                    ptx::tc_fence_after();
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) {
                        uint32_t dp[32], pk[16];
                        ptx::tmem_ld32(tP + 32 * c2, dp);
                        ptx::tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const float2 d2 = *reinterpret_cast<const float2*>(L + 64 + 32 * c2 + 2 * e);
                            const uint64_t dd = ptx::f2_add(
                                ptx::f2_pack(__uint_as_float(dp[2 * e]), __uint_as_float(dp[2 * e + 1])),
                                ptx::f2_pack(d2.x, d2.y));
                            float d0, d1;
                            ptx::f2_unpack(ptx::f2_mul(pf[16 * c2 + e], dd), d0, d1);
                            pk[e] = ptx::pack_bf16(d0, d1);
                        }
                        ptx::tmem_st16(tP + 16 * c2, pk);
                    }
                    ptx::tmem_wait_st();
                    ptx::tc_fence_before();
                    arrive(&bar.dst_full);
                }
                ok = ok && wait_all(&bar.kv_full, (uint32_t)(ik & 1));
                if (!ok) break;
                ++ik;
                // each half stores D/2 columns of its dK and dV rows
                ptx::tc_fence_after();
                const size_t off = (((size_t)it.b * p.R + it.crow + r) * p.H + it.h) * D + DH * half;
                const bool rv = r < it.rows;
#pragma unroll
                for (int which = 0; which < 2; ++which) {
                    float* dst = (which == 0 ? p.dv_ctx : p.dk_ctx) + off;
                    const float mul = which == 0 ? 1.f : p.scale;
                    uint32_t o[DH / 32][32];
#pragma unroll
                    for (int c = 0; c < DH / 32; ++c)
                        ptx::tmem_ld32(tbase + 256 + which * D + DH * half + 32 * c + lane_off, o[c]);
                    ptx::tmem_wait_ld();
                    if (rv) {
#pragma unroll
                        for (int c = 0; c < DH / 32; ++c) store_f32(dst + 32 * c, o[c], mul, p.ctx_v8 != 0);
                    }
                }
            }
            // the item's accumulators are read: the next item's MMAs may
            // overwrite them (its first P or dS is written after this)
            ptx::tc_fence_before();
            arrive(&bar.item_done[done_bar(k)]);
        }
        if (!ok && lane == 0) atomicOr(p.status, kDevTimeout);
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tbase, 512);
    }
}

bool encode_all(BwdMaps& m, const Plan& P, const BwdTcInput& in) {
    const long long row = (long long)P.H * P.D * 2;
    if (!encode_rows(&m.q, in.q, P.D, P.H, P.N, P.B, (long long)P.N * row)) return false;
    if (!encode_rows(&m.dout, in.dout, P.D, P.H, P.N, P.B, (long long)P.N * row)) return false;
    bool done[kNumMaps] = {false};
    for (int gi = 0; gi < in.a->n_groups; ++gi) {
        const AttnGroup& ag = in.a->g[gi];
        for (int s = 0; s < ag.n_seg; ++s) {
            const Segment& sg = ag.seg[s];
            int slot = sg.map_id, rows = sg.rows_total;
            const char* kb = sg.k;
            const char* vb = sg.v;
            if (slot == kMapPyr) {
                slot = kMapPyr0 + gi;
                kb += (size_t)sg.row0 * row;
                vb += (size_t)sg.row0 * row;
                rows = sg.len;
            } else if (slot == kMapHist) {
                rows = sg.len;
            }
            if (done[slot]) continue;
            if (!encode_rows(&m.k[slot], kb, P.D, P.H, rows, P.B, sg.bstride) ||
                !encode_rows(&m.v[slot], vb, P.D, P.H, rows, P.B, sg.bstride))
                return false;
            done[slot] = true;
        }
    }
    return true;
}

// Every item of a gradient, host only: the groups, the ranges and the classes of
// equal items; returns the number of classes.
int fill_items(const Plan& P, const AttnArgs& a, const BwdGroup* bg, BwdTcParams& tp, ItemClass* rs) {
    // dQ: every query tile of every group, longest contexts first.
    int order[MSF_MAX_GROUPS];
    int len[MSF_MAX_GROUPS];
    for (int i = 0; i < a.n_groups; ++i) {
        order[i] = i;
        len[i] = 0;
        for (int s = 0; s < a.g[i].n_seg; ++s) len[i] += a.g[i].seg[s].len;
    }
    for (int i = 0; i < a.n_groups; ++i)
        for (int k = i + 1; k < a.n_groups; ++k)
            if (len[order[k]] > len[order[i]]) {
                const int t = order[i];
                order[i] = order[k];
                order[k] = t;
            }
    for (int oi = 0; oi < a.n_groups; ++oi) {
        const int gi = order[oi];
        const AttnGroup& ag = a.g[gi];
        BGroupQ& g = tp.g[oi];
        g.q_begin = ag.q_begin;
        g.q_end = ag.q_end;
        g.n_qt = (ag.q_end - ag.q_begin + kBM - 1) / kBM;
        g.n_seg = ag.n_seg;
        g.n_tiles = 0;
        for (int s = 0; s < ag.n_seg; ++s) {
            const Segment& sg = ag.seg[s];
            BSeg& bs = g.seg[s];
            bs.map = sg.map_id == kMapPyr ? kMapPyr0 + gi : sg.map_id;
            bs.row0 = sg.map_id == kMapPyr ? 0 : sg.row0;
            bs.len = sg.len;
            bs.tile0 = g.n_tiles;
            g.n_tiles += (sg.len + kBM - 1) / kBM;
        }
    }
    // dK/dV: every group's window-derived rows in one launch, groups with
    // the most query tiles first.
    int korder[MSF_MAX_GROUPS];
    int nk = 0;
    for (int gi = 0; gi < a.n_groups; ++gi)
        if (bg[gi].n_gseg > 0 && bg[gi].q_end > bg[gi].q_begin) korder[nk++] = gi;
    for (int i = 0; i < nk; ++i)
        for (int k = i + 1; k < nk; ++k)
            if (bg[korder[k]].q_end - bg[korder[k]].q_begin >
                bg[korder[i]].q_end - bg[korder[i]].q_begin) {
                const int t = korder[i];
                korder[i] = korder[k];
                korder[k] = t;
            }
    for (int oi = 0; oi < nk; ++oi) {
        const int gi = korder[oi];
        const BwdGroup& b = bg[gi];
        BGroupK& kg = tp.kg[oi];
        kg.q_begin = b.q_begin;
        kg.q_end = b.q_end;
        kg.n_qt = (b.q_end - b.q_begin + kBM - 1) / kBM;
        kg.n_grad = b.n_gseg;
        int kt0 = 0;
        for (int s = 0; s < b.n_gseg; ++s) {
            const GradSeg& gs = b.gseg[s];
            BGrad& g = kg.gr[s];
            g.map = gs.map_id == kMapPyr ? kMapPyr0 + gi : gs.map_id;
            // pyramid rows are addressed from the group's pyramid part, the
            // ring from its first slot, the window from token 0
            g.row0 = gs.map_id == kMapPyr ? gs.row0 - P.groups[gi].pyr_offset : gs.row0;
            g.len = gs.len;
            g.kt0 = kt0;
            g.crow0 = gs.crow0;
            kt0 += (gs.len + kBM - 1) / kBM;
        }
        kg.n_kt = kt0;
    }
    // Ranges with the most MMA blocks per item first; the times are from
    // globaltimer stamps over eight windows of 1 to 175 tiles an item (within
    // 8 % from two tiles on).
    const bool d128 = P.D == 128;
    int nr = 0;
    for (int oi = 0; oi < a.n_groups; ++oi) {
        const int n = tp.g[oi].n_tiles;
        if (tp.g[oi].n_qt > 0)
            rs[nr++] = {0, oi, tp.g[oi].n_qt * P.H * P.B, 3 * n, d128 ? 1200 + 1085 * n : 1500 + 710 * n, 0};
    }
    for (int oi = 0; oi < nk; ++oi) {
        const int n = tp.kg[oi].n_qt;
        if (tp.kg[oi].n_kt > 0)
            rs[nr++] = {1, oi, tp.kg[oi].n_kt * P.H * P.B, 4 * n, d128 ? 4500 + 1355 * n : 2600 + 1110 * n, 0};
    }
    for (int i = 0; i < nr; ++i)
        for (int k = i + 1; k < nr; ++k)
            if (rs[k].blocks > rs[i].blocks) {
                const ItemClass t = rs[i];
                rs[i] = rs[k];
                rs[k] = t;
            }
    int total = 0;
    for (int i = 0; i < nr; ++i) {
        tp.range[i].kind = rs[i].kind;
        tp.range[i].group = rs[i].group;
        tp.range[i].base = rs[i].base = total;
        total += rs[i].count;
    }
    tp.n_ranges = nr;
    tp.n_items = total;
    return nr;
}

}  // namespace

void bwd_route(const Plan& P, const AttnArgs& a, const BwdGroup* bg, int sms, BwdRoute* out) {
    BwdTcParams tp;
    memset(&tp, 0, sizeof(tp));
    ItemClass rs[2 * MSF_MAX_GROUPS];
    const int nr = fill_items(P, a, bg, tp, rs);
    BwdOrder order;
    place_items(order, rs, nr, tp.n_items, tp.n_items < sms ? tp.n_items : sms);
    *out = {tp.n_items, order.on};
}

msf_status launch_bwd_tc(msf_plan_t plan, const BwdTcInput& in, cudaStream_t st) {
    const Plan& P = *plan;
    const AttnArgs& a = *in.a;
    BwdMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (!encode_all(maps, P, in)) {
        set_cuda_error((int)cudaErrorInvalidValue);
        return MSF_ERR_CUDA;
    }
    BwdTcParams tp;
    memset(&tp, 0, sizeof(tp));
    tp.H = P.H;
    tp.B = P.B;
    tp.N = P.N;
    tp.scale = P.scale;
    tp.scale_log2 = P.scale * kLog2e;
    tp.lse = in.lse;
    tp.delta = in.delta;
    tp.dq = (__nv_bfloat16*)in.dq;
    tp.dk_ctx = in.dk_ctx;
    tp.dv_ctx = in.dv_ctx;
    tp.R = in.R;
    tp.status = a.status;
    tp.wait_limit = kWaitLimit;
    ItemClass rs[2 * MSF_MAX_GROUPS];
    const int nr = fill_items(P, a, in.g, tp, rs), total = tp.n_items;
    if (total == 0) return MSF_OK;
    // Rows of one head are a multiple of 32 bytes, so the bases decide.
    tp.dq_v8 = (uintptr_t)in.dq % 32 == 0;
    tp.ctx_v8 = (uintptr_t)in.dk_ctx % 32 == 0 && (uintptr_t)in.dv_ctx % 32 == 0;
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) {
        set_cuda_error((int)e);
        return MSF_ERR_CUDA;
    }
    const int grid = total < sms ? total : sms;
    BwdOrder placed;
    place_items(placed, rs, nr, total, grid);
    const bool d128 = P.D == 128;
    const int smem = d128 ? BCfg<128>::kSmem : BCfg<64>::kSmem;
    e = d128 ? set_smem_attr((const void*)bwd_tc_kernel<128>, BCfg<128>::kSmem)
             : set_smem_attr((const void*)bwd_tc_kernel<64>, BCfg<64>::kSmem);
    if (e != cudaSuccess) {
        set_cuda_error((int)e);
        return MSF_ERR_CUDA;
    }
    e = d128 ? launch_pdl(bwd_tc_kernel<128>, dim3((unsigned)grid), dim3(kThreads), smem, st, maps, tp, placed)
             : launch_pdl(bwd_tc_kernel<64>, dim3((unsigned)grid), dim3(kThreads), smem, st, maps, tp, placed);
    if (e != cudaSuccess) {
        set_cuda_error((int)e);
        return MSF_ERR_CUDA;
    }
    return MSF_OK;
}

}  // namespace msf
