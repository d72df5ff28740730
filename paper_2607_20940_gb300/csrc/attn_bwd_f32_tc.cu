// fp32 MSSA backward on the sm_103a tensor cores: operands as three bf16
// planes, six plane products per product, smallest first (see attn_f32_tc.cu).
//
// With the forward's row log-sum-exp, P = exp(c S - lse) and
//   dS = P * (dP - delta),  dP = dO V^T,  delta = rowsum(dO * O)
//   dQ = c dS K,  dK = c dS^T Q,  dV = P^T dO.
// A unit owns one 128-row tile of "own" rows and walks a range of 128-row
// tiles of "other" rows, and every kind has one shape:
//   kind   own rows          S operands   dP operands   output += A x B
//   dQ     queries           Q,  K        dO, V         dS   x K
//   dK     window context    K,  Q        V,  dO        dS^T x Q
//   dV     window context    K,  Q        -             P^T  x dO
// (dK and dV are separate units: their P^T and dS^T planes together with both
// outputs would not fit tensor memory; S^T twice costs a sixth more MMAs.)
// The own S operand's planes stay in shared memory, the own dP operand's in
// tensor memory (the A operand of dP), and the other rows' planes stream
// through a 4-deep ring of 128-row plane tiles. Each tile's output is read out
// and added in fp32 registers, so no accumulator carries over tiles.
//
// TMEM columns: S [0,128), dP [128,256), output [192, 192 + D), own dP
// operand's planes from 320 (64 each). The planes of dS (P) are written over
// S (h, m) and [128,192) (l); the output takes dP's place once it is read.
// Bound: the tensor pipe, 144 MMAs of 64 cycles per tile pair for dQ and dK, 96
// for dV, plus the softmax between dP and the output (the exponentials
// run beside the dP MMAs). A small window (two 16 x 24 frames per state, 1008
// tokens, 4 heads x 128) takes 86 us where the CUDA-core kernels take 1422 us,
// with relative errors against 64 bits of 5.1-6.1e-7 (CUDA cores 6.5-8.5e-7).
// At D = 128 ptxas spills 44 bytes of the 168 registers.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "attn_bwd_tc.h"
#include "attn_f32_tc.h"
#include "f32_range.cuh"
#include "ptx.cuh"

namespace msf {
namespace {

constexpr int kBM = 128;       // rows of every tile
constexpr int kThreads = 384;  // 12 warps
constexpr int kRing = 4;       // plane tiles in flight
constexpr int kPCol = 128, kLCol = 128, kOutCol = 192, kACol = 320;
constexpr long long kWaitLimit = 2000000000LL;  // ~1 s of SM clock
constexpr float kLog2e = 1.4426950408889634f;
// Register split as in attn_f32_tc.cu.
constexpr int kLaunchRegs = 168, kCtrlRegs = 104, kSoftmaxRegs = 192;
static_assert(4 * kCtrlRegs + 8 * kSoftmaxRegs <= 12 * kLaunchRegs, "register split");

enum : int { kDq = 0, kDk = 1, kDv = 2 };

struct FBSeg {
    int map, row0, len, tile0;
};
struct FBGrad {
    const float* v;      // stream 0, the run's first row
    long long vbstride;  // elements
    int map, row0, len, tile0;
    int crow0;           // first row of the run in the context-gradient buffers
};
struct FBGroup {
    int q_begin, q_end;
    int n_seg;
    FBSeg seg[kMaxSeg];
    int n_grad;
    FBGrad gr[kMaxGradSeg];
};
struct FBClass {
    int kind, group;
    int n_own;      // own tiles per (stream, head)
    int n_tiles;    // other tiles
    int n_split;    // units per own tile
    int unit_base;  // first unit (block)
    int slot_base;  // first partial slot (n_split > 1)
    int item_base;  // first own tile of the merge launch (n_split > 1)
};
struct FBParams {
    int H, B, N, R;
    float scale, scale_log2;
    const float* lse;
    const float* delta;
    const float* dout;
    float* dq;
    float* dk_ctx;
    float* dv_ctx;
    float* partials;  // [slot][128][D]
    F32Range range;
    unsigned int* status;
    long long wait_limit;
    int n_classes;
    FBClass c[kMaxF32Classes];  // longest units first
    FBGroup g[MSF_MAX_GROUPS];
};

template <int D>
struct FBCfg {
    static constexpr int kTile = kBM * D * 2;
    static constexpr int kSmem = (3 + kRing) * kTile + 1024 > 120 * 1024 ? (3 + kRing) * kTile + 1024 : 120 * 1024;
    static constexpr int kSlot = kBM * D;
};
static_assert(FBCfg<128>::kSmem + 2048 <= 227 * 1024, "shared memory of the launch");

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Own tile `own` of class c: the run it belongs to (dK, dV) and its tile there.
__device__ __forceinline__ int grad_run(const FBGroup& G, int own) {
    int s = 0;
    while (s + 1 < G.n_grad && own >= G.gr[s + 1].tile0) ++s;
    return s;
}

// Where row r of own tile `own` goes: its output row, or NULL past the end.
template <int D>
__device__ __forceinline__ float* out_row(const FBParams& p, const FBClass& c, int own, int h, int b, int r) {
    const FBGroup& G = p.g[c.group];
    if (c.kind == kDq) {
        const int q = G.q_begin + own * kBM + r;
        return q < G.q_end ? p.dq + (((size_t)b * p.N + q) * p.H + h) * D : nullptr;
    }
    const FBGrad& gr = G.gr[grad_run(G, own)];
    const int k = (own - gr.tile0) * kBM + r;
    float* base = c.kind == kDk ? p.dk_ctx : p.dv_ctx;
    return k < gr.len ? base + (((size_t)b * p.R + gr.crow0 + k) * p.H + h) * D : nullptr;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    bwd_f32_kernel(const __grid_constant__ F32Maps maps, const __grid_constant__ FBParams p) {
    using C = FBCfg<D>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sA = smem;                 // [3] planes of the own S operand
    unsigned char* sR = smem + 3 * C::kTile;  // [kRing]
    __shared__ uint64_t a_full, full[kRing], empty[kRing], s_full, dp_full, ds_full, o_full, o_free, a2_full, meet_bar;
    __shared__ uint64_t drain_bar;
    __shared__ float sL[kBM], sD[kBM];  // the other rows' statistics (dK, dV)
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    int ci = 0;
    while (ci + 1 < p.n_classes && (int)blockIdx.x >= p.c[ci + 1].unit_base) ++ci;
    const FBClass& cl = p.c[ci];
    const FBGroup& G = p.g[cl.group];
    const int kind = cl.kind;
    // units of one head in order split, own tile: neighbours share other tiles in L2
    const int local = (int)blockIdx.x - cl.unit_base;
    const int own = local % cl.n_own;
    const int split = (local / cl.n_own) % cl.n_split;
    const int bh = local / (cl.n_own * cl.n_split);
    const int h = bh % p.H, b = bh / p.H;
    const int u0 = split * cl.n_tiles / cl.n_split, u1 = (split + 1) * cl.n_tiles / cl.n_split;
    const int n = u1 - u0;
    const FBGrad& gr = G.gr[kind == kDq ? 0 : grad_run(G, own)];
    const int own_row = kind == kDq ? G.q_begin + own * kBM : gr.row0 + (own - gr.tile0) * kBM;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        ptx::mbar_init(&a_full, 1);
        for (int s = 0; s < kRing; ++s) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&empty[s], 1);
        }
        ptx::mbar_init(&s_full, 1);
        ptx::mbar_init(&dp_full, 1);
        ptx::mbar_init(&ds_full, 8);
        ptx::mbar_init(&o_full, 1);
        ptx::mbar_init(&o_free, 8);
        ptx::mbar_init(&a2_full, 8);
        ptx::mbar_init(&meet_bar, 8);
        ptx::mbar_init(&drain_bar, 1);
        ptx::fence_mbar_init();
    }
    if (warp == 2) {
        ptx::tmem_alloc(&tmem_base_sh, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tbase = tmem_base_sh;
    volatile int* abort_p = &abort_flag;
    volatile int never = 0;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const bool skip = !planes_hold(p.range);  // the CUDA-core kernels answer instead

    // other tile u: map of K/V (dQ), first row, valid rows
    auto tile_of = [&](int u, int& map, int& row, int& valid) {
        if (kind != kDq) {
            map = 0;
            row = G.q_begin + u * kBM;
            valid = min(kBM, G.q_end - row);
            return;
        }
        int s = 0;
        while (s < G.n_seg - 1 && u >= G.seg[s + 1].tile0) ++s;
        const int kt = u - G.seg[s].tile0;
        map = G.seg[s].map;
        row = G.seg[s].row0 + kt * kBM;
        valid = min(kBM, G.seg[s].len - kt * kBM);
    };

    if (skip) {
    } else if (warp < 4) {
        ptx::setmaxnreg_dec<kCtrlRegs>();
        if (warp == 0) {
            // ============================ TMA producer ============================
            if (lane == 0) {
                bool ok = true;
                const CUtensorMap* ma = kind == kDq ? &maps.q : &maps.k[gr.map];
                ptx::mbar_arrive_expect_tx(&a_full, 3 * C::kTile);
                for (int pl = 0; pl < 3; ++pl)
                    for (int c = 0; c < D / 64; ++c)
                        ptx::tma_load_4d(sA + pl * C::kTile + c * (kBM * 128), ma, &a_full, c * 64, h, own_row,
                                         3 * b + pl);
                int it = 0;  // plane tiles issued
                auto planes = [&](const CUtensorMap* m, int row) {
                    for (int pl = 2; pl >= 0; --pl) {
                        const int st = it % kRing;
                        if (!ptx::mbar_wait_bounded(&empty[st], (uint32_t)(((it / kRing) & 1) ^ 1), abort_p,
                                                    p.wait_limit))
                            return false;
                        ptx::mbar_arrive_expect_tx(&full[st], C::kTile);
                        for (int c = 0; c < D / 64; ++c)
                            ptx::tma_load_4d(sR + st * C::kTile + c * (kBM * 128), m, &full[st], c * 64, h, row,
                                             3 * b + pl);
                        ++it;
                    }
                    return true;
                };
                for (int u = u0; u < u1 && ok; ++u) {
                    int map, row, valid;
                    tile_of(u, map, row, valid);
                    const CUtensorMap* ms = kind == kDq ? &maps.k[map] : &maps.q;
                    ok = planes(ms, row);
                    if (kind != kDv) ok = ok && planes(kind == kDq ? &maps.v[map] : &maps.dout, row);
                    ok = ok && planes(kind == kDv ? &maps.dout : ms, row);
                }
                if (!ok) {
                    // every copy issued lands before the CTA exits
                    ptx::mbar_wait_bounded(&a_full, 0, &never, kWaitLimit);
                    for (int i = (it > kRing ? it - kRing : 0); i < it; ++i)
                        ptx::mbar_wait_bounded(&full[i % kRing], (uint32_t)((i / kRing) & 1), &never, kWaitLimit);
                    atomicOr(p.status, kDevTimeout);
                }
            }
        } else if (warp == 1) {
            // ============================= MMA issuer =============================
            constexpr uint32_t idS = ptx::idesc_bf16(kBM, kBM, false, false);
            constexpr uint32_t idO = ptx::idesc_bf16(kBM, D, false, true);
            constexpr uint64_t kTileDesc = (uint64_t)(C::kTile >> 4);
            const uint64_t a_desc = ptx::sdesc_sw128(ptx::smem_u32(sA), 16, 1024);
            const uint64_t r_desc = ptx::sdesc_sw128(ptx::smem_u32(sR), 16, 1024);
            const uint64_t mn_desc = ptx::sdesc_sw128(ptx::smem_u32(sR), kBM * 128, 1024);
            auto wait_all = [&](uint64_t* bar, uint32_t parity) {
                const bool r = ptx::mbar_wait_bounded(bar, parity, abort_p, p.wait_limit);
                return __all_sync(0xffffffffu, r);
            };
            int it = 0;
            bool ok = wait_all(&a_full, 0);
            if (ok && kind != kDv) ok = wait_all(&a2_full, 0);
            for (int j = 0; j < n && ok; ++j) {
                // S: with the other plane bp the own planes from 2 - bp down to h
                for (int bp = 2; bp >= 0 && ok; --bp, ++it) {
                    const int st = it % kRing;
                    ok = wait_all(&full[st], (uint32_t)((it / kRing) & 1));
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) {
                        const uint64_t bd = r_desc + (uint64_t)st * kTileDesc;
                        for (int ap = 2 - bp; ap >= 0; --ap) {
                            const uint64_t ad = a_desc + (uint64_t)ap * kTileDesc;
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk) {
                                const uint64_t off = (uint64_t)(((kk / 4) * (kBM * 128) + (kk % 4) * 32) >> 4);
                                ptx::mma_ss(tbase, ad + off, bd + off, idS, (bp < 2 || kk > 0) ? 1u : 0u);
                            }
                        }
                        ptx::mma_commit(&empty[st]);
                        if (bp == 0) ptx::mma_commit(&s_full);
                    }
                    __syncwarp();
                }
                if (!ok) break;
                // the previous tile's output has been read: dP takes its columns
                if (j > 0) ok = wait_all(&o_free, (uint32_t)((j - 1) & 1));
                if (kind != kDv)
                    for (int bp = 2; bp >= 0 && ok; --bp, ++it) {
                        const int st = it % kRing;
                        ok = wait_all(&full[st], (uint32_t)((it / kRing) & 1));
                        if (!ok) break;
                        ptx::tc_fence_after();
                        if (ptx::elect_one_sync()) {
                            const uint64_t bd = r_desc + (uint64_t)st * kTileDesc;
                            for (int ap = 2 - bp; ap >= 0; --ap) {
#pragma unroll
                                for (int kk = 0; kk < D / 16; ++kk) {
                                    const uint64_t off = (uint64_t)(((kk / 4) * (kBM * 128) + (kk % 4) * 32) >> 4);
                                    ptx::mma_ts(tbase + kPCol, tbase + kACol + 64 * ap + kk * 8, bd + off, idS,
                                                (bp < 2 || kk > 0) ? 1u : 0u);
                                }
                            }
                            ptx::mma_commit(&empty[st]);
                            if (bp == 0) ptx::mma_commit(&dp_full);
                        }
                        __syncwarp();
                    }
                ok = ok && wait_all(&ds_full, (uint32_t)(j & 1));
                for (int bp = 2; bp >= 0 && ok; --bp, ++it) {
                    const int st = it % kRing;
                    ok = wait_all(&full[st], (uint32_t)((it / kRing) & 1));
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (ptx::elect_one_sync()) {
                        const uint64_t bd = mn_desc + (uint64_t)st * kTileDesc;
                        for (int ap = 2 - bp; ap >= 0; --ap) {
#pragma unroll
                            for (int kk = 0; kk < kBM / 16; ++kk) {
                                const uint32_t half = kk / 4, c = (kk % 4) * 8;
                                const uint32_t a = tbase + c + (ap == 2 ? kLCol + 32 * half : 64 * half + 32 * ap);
                                ptx::mma_ts(tbase + kOutCol, a, bd + (uint64_t)(kk * (2048 >> 4)), idO,
                                            (bp < 2 || kk > 0) ? 1u : 0u);
                            }
                        }
                        ptx::mma_commit(&empty[st]);
                        if (bp == 0) ptx::mma_commit(&o_full);
                    }
                    __syncwarp();
                }
            }
            if (!ok) {
                if (ptx::elect_one_sync()) ptx::mma_commit(&drain_bar);
                __syncwarp();
                ptx::mbar_wait_bounded(&drain_bar, 0, &never, kWaitLimit);
                if (lane == 0) atomicOr(p.status, kDevTimeout);
            }
        }
    } else {
        ptx::setmaxnreg_inc<kSoftmaxRegs>();
        // ============ softmax: one thread per own row and column half ============
        const int half = (warp - 4) / 4, wq = warp % 4;
        const int r = wq * 32 + lane;
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        constexpr int DH = D / 2;  // output columns of this thread
        const uint32_t tS = tbase + 64 * half + lane_off;
        const uint32_t tP = tbase + kPCol + 64 * half + lane_off;
        const uint32_t tL = tbase + kLCol + 32 * half + lane_off;
        const uint32_t tO = tbase + kOutCol + DH * half + lane_off;
        const float sl2 = p.scale_log2;
        float nl = 0.f, nd = 0.f;  // dQ: this row's -lse (log2 units) and -delta
        if (kind == kDq) {
            const int q = own_row + r;
            const size_t rix = ((size_t)b * p.H + h) * p.N + q;
            nl = q < G.q_end ? -p.lse[rix] * kLog2e : -INFINITY;
            nd = q < G.q_end ? -p.delta[rix] : 0.f;
        }
        if (kind != kDv) {
            // the own dP operand (dO or V) into tensor memory, as planes
            const float* src = nullptr;
            if (kind == kDq) {
                const int q = own_row + r;
                if (q < G.q_end) src = p.dout + (((size_t)b * p.N + q) * p.H + h) * D;
            } else {
                const int k = (own - gr.tile0) * kBM + r;
                if (k < gr.len) src = gr.v + b * gr.vbstride + ((size_t)k * p.H + h) * D;
            }
#pragma unroll 1
            for (int c = 0; c < DH / 32; ++c) {
                uint32_t ph[16], pm[16], pl[16];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 x = src ? __ldg(reinterpret_cast<const float4*>(src + DH * half + 32 * c) + e)
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
                    ptx::split_bf16(x.x, x.y, ph[2 * e], pm[2 * e], pl[2 * e]);
                    ptx::split_bf16(x.z, x.w, ph[2 * e + 1], pm[2 * e + 1], pl[2 * e + 1]);
                }
                const uint32_t t = tbase + kACol + DH / 2 * half + 16 * c + lane_off;
                ptx::tmem_st16(t, ph);
                ptx::tmem_st16(t + 64, pm);
                ptx::tmem_st16(t + 128, pl);
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&a2_full);
        }
        float acc[DH];
#pragma unroll
        for (int e = 0; e < DH; ++e) acc[e] = 0.f;
        // The eight softmax warps meet (bounded, unlike a hardware barrier).
        uint32_t meets = 0;
        auto meet = [&]() {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&meet_bar);
            const bool r = ptx::mbar_wait_bounded(&meet_bar, meets & 1u, abort_p, p.wait_limit);
            ++meets;
            return (bool)__all_sync(0xffffffffu, r);
        };
        bool ok = true;
        for (int j = 0; j < n && ok; ++j) {
            int map, row, valid;
            tile_of(u0 + j, map, row, valid);
            if (kind != kDq) {
                // the other rows' statistics: threads 0-127 -lse, 128-255 -delta
                // (every thread has finished the previous tile's: its output
                // could not be ready before)
                const size_t rix = ((size_t)b * p.H + h) * p.N + row + r;
                if (half == 0)
                    sL[r] = r < valid ? -p.lse[rix] * kLog2e : -INFINITY;
                else
                    sD[r] = r < valid ? -p.delta[rix] : 0.f;
                ok = meet();
                if (!ok) break;
            }
            ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&s_full, (uint32_t)(j & 1), abort_p, p.wait_limit));
            if (!ok) break;
            ptx::tc_fence_after();
            float pr[64];
            {
                const int lim = kind == kDq ? valid - 64 * half : 64;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t s[32];
                    ptx::tmem_ld32(tS + 32 * c, s);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        const int x = 32 * c + e;
                        const float off = kind == kDq ? nl : sL[64 * half + x];
                        // context rows past the segment's end: probability 0
                        pr[x] = x < lim ? ex2(fmaf(__uint_as_float(s[e]), sl2, off)) : 0.f;
                    }
                }
            }
            if (kind != kDv) {
                ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&dp_full, (uint32_t)(j & 1), abort_p, p.wait_limit));
                if (!ok) break;
                ptx::tc_fence_after();
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t d[32];
                    ptx::tmem_ld32(tP + 32 * c, d);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        const int x = 32 * c + e;
                        pr[x] *= __uint_as_float(d[e]) + (kind == kDq ? nd : sD[64 * half + x]);
                    }
                }
                // every thread has read its dP: the l planes go into its columns
                ptx::tc_fence_before();
                ok = meet();
                if (!ok) break;
                ptx::tc_fence_after();
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t ph[16], pm[16], pl[16];
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    ptx::split_bf16(pr[32 * c + 2 * e], pr[32 * c + 2 * e + 1], ph[e], pm[e], pl[e]);
                ptx::tmem_st16(tS + 16 * c, ph);
                ptx::tmem_st16(tS + 32 + 16 * c, pm);
                ptx::tmem_st16(tL + 16 * c, pl);
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&ds_full);
            ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&o_full, (uint32_t)(j & 1), abort_p, p.wait_limit));
            if (!ok) break;
            ptx::tc_fence_after();
#pragma unroll
            for (int c = 0; c < DH / 32; ++c) {
                uint32_t o[32];
                ptx::tmem_ld32(tO + 32 * c, o);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[32 * c + e] += __uint_as_float(o[e]);
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&o_free);
        }
        if (ok) {
            float* dst;
            float mul = kind == kDv ? 1.f : p.scale;
            if (cl.n_split > 1) {
                dst = p.partials + (size_t)(cl.slot_base + local) * C::kSlot + r * D;
                mul = 1.f;
            } else {
                dst = out_row<D>(p, cl, own, h, b, r);
            }
            if (dst) {
                float4* d4 = reinterpret_cast<float4*>(dst + DH * half);
#pragma unroll
                for (int e = 0; e < DH / 4; ++e)
                    d4[e] = make_float4(acc[4 * e] * mul, acc[4 * e + 1] * mul, acc[4 * e + 2] * mul,
                                        acc[4 * e + 3] * mul);
            }
        } else if (lane == 0) {
            atomicOr(p.status, kDevTimeout);
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tbase, 512);
    }
}

// Own tiles in several units: the sum of their outputs in unit order. One warp
// per row at a time, eight blocks per own tile.
template <int D>
__global__ void __launch_bounds__(256) bwd_f32_merge_kernel(const __grid_constant__ FBParams p) {
    using C = FBCfg<D>;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (!planes_held(p.range)) return;
    int ci = 0;
    while (ci + 1 < p.n_classes && (p.c[ci].n_split == 1 || (int)blockIdx.x >= p.c[ci + 1].item_base)) ++ci;
    const FBClass& cl = p.c[ci];
    const int item = (int)blockIdx.x - cl.item_base;
    const int own = item % cl.n_own, bh = item / cl.n_own;
    const int h = bh % p.H, b = bh / p.H;
    const float* first = p.partials + (size_t)(cl.slot_base + bh * cl.n_split * cl.n_own + own) * C::kSlot;
    const size_t step = (size_t)cl.n_own * C::kSlot;  // to the tile's next unit
    const int lane = threadIdx.x % 32;
    const float mul = cl.kind == kDv ? 1.f : p.scale;
    constexpr int E = D / 32;
    for (int r = threadIdx.x / 32 + 16 * blockIdx.y; r < 16 * ((int)blockIdx.y + 1); r += 8) {
        float* dst = out_row<D>(p, cl, own, h, b, r);
        if (!dst) break;
        float acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = 0.f;
#pragma unroll 4
        for (int i = 0; i < cl.n_split; ++i) {
            const float* s = first + i * step + r * D + E * lane;
            if (E == 4) {
                const float4 v = __ldcg(reinterpret_cast<const float4*>(s));
                acc[0] += v.x;
                acc[1] += v.y;
                acc[E - 2] += v.z;
                acc[E - 1] += v.w;
            } else {
                const float2 v = __ldcg(reinterpret_cast<const float2*>(s));
                acc[0] += v.x;
                acc[1] += v.y;
            }
        }
        dst += E * lane;
        if (E == 4)
            *reinterpret_cast<float4*>(dst) = make_float4(acc[0] * mul, acc[1] * mul, acc[E - 2] * mul, acc[E - 1] * mul);
        else
            *reinterpret_cast<float2*>(dst) = make_float2(acc[0] * mul, acc[1] * mul);
    }
}

}  // namespace

msf_status launch_bwd_f32_tc(msf_plan_t plan, const BwdCommon& c, const AttnArgs& a, const BwdGroup* bg, float* dq,
                             char* dout_planes, F32Range* range, cudaStream_t st) {
    const Plan& P = *plan;
    auto fail = [](cudaError_t e) {
        set_cuda_error((int)e);
        return MSF_ERR_CUDA;
    };
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return fail(e);
    if (sms > kF32MaxSms) sms = kF32MaxSms;
    // As in the forward, with few keys the CUDA-core kernels are ahead (whole gradient,
    // 12 keys x 64: 12.1 us against 12.4; 4 and 12 keys x 128: 9.1 against 15.8, 16.6
    // against 15.6).
    *range = {};
    if (f32_longest_context(a) <= (P.D == 64 ? 12 : 10)) return MSF_OK;

    SplitParams sp;
    memset(&sp, 0, sizeof(sp));
    F32Maps maps;
    memset(&maps, 0, sizeof(maps));
    sp.words = f32_range_words(P);
    if (!add_context_planes(P, a, sp, maps) || !add_planes(P, sp, kRangeDout, c.dout, c.bstride, dout_planes, P.N, P.N, &maps.dout))
        return fail(cudaErrorInvalidValue);
    FBParams fp;
    memset(&fp, 0, sizeof(fp));
    fp.H = P.H;
    fp.B = P.B;
    fp.N = P.N;
    fp.R = c.R;
    fp.scale = c.scale;
    fp.scale_log2 = c.scale_log2;
    fp.lse = c.lse;
    fp.delta = c.delta;
    fp.dout = (const float*)c.dout;
    fp.dq = dq;
    fp.dk_ctx = c.dk_ctx;
    fp.dv_ctx = c.dv_ctx;
    fp.partials = f32_partials(P);
    fp.status = a.status;
    fp.wait_limit = kWaitLimit;
    const size_t row = (size_t)P.H * P.D * 4;
    for (int gi = 0; gi < a.n_groups; ++gi) {
        const AttnGroup& ag = a.g[gi];
        FBGroup& g = fp.g[gi];
        g.q_begin = ag.q_begin;
        g.q_end = ag.q_end;
        const int n_qt = (ag.q_end - ag.q_begin + kBM - 1) / kBM;
        int tiles = 0;
        g.n_seg = ag.n_seg;
        for (int s = 0; s < ag.n_seg; ++s) {
            const Segment& sg = ag.seg[s];
            const bool pyr = sg.map_id == kMapPyr;
            g.seg[s] = {pyr ? kMapPyr0 + gi : sg.map_id, pyr ? 0 : sg.row0, sg.len, tiles};
            tiles += (sg.len + kBM - 1) / kBM;
        }
        int kt = 0;
        g.n_grad = bg[gi].n_gseg;
        for (int s = 0; s < bg[gi].n_gseg; ++s) {
            const GradSeg& gs = bg[gi].gseg[s];
            const bool pyr = gs.map_id == kMapPyr;
            FBGrad& f = g.gr[s];
            f.v = (const float*)(gs.v + (size_t)gs.row0 * row);
            f.vbstride = gs.bstride / 4;
            // pyramid rows are addressed from the group's pyramid part, the
            // ring from its first slot, the window from token 0
            f.map = pyr ? kMapPyr0 + gi : gs.map_id;
            f.row0 = pyr ? gs.row0 - P.groups[gi].pyr_offset : gs.row0;
            f.len = gs.len;
            f.tile0 = kt;
            f.crow0 = gs.crow0;
            kt += (gs.len + kBM - 1) / kBM;
        }
        if (n_qt == 0) continue;
        fp.c[fp.n_classes++] = {kDq, gi, n_qt, tiles};
        if (kt > 0) {
            fp.c[fp.n_classes++] = {kDk, gi, kt, n_qt};
            fp.c[fp.n_classes++] = {kDv, gi, kt, n_qt};
        }
    }
    // Units per own tile (a dV tile costs what a forward tile does).
    const int HB = P.H * P.B, max_slots = f32_max_slots(P);
    F32Class cls[kMaxF32Classes];
    for (int i = 0; i < fp.n_classes; ++i)
        cls[i] = {(long long)fp.c[i].n_own * HB, fp.c[i].n_tiles, fp.c[i].kind == kDv ? 1.0 : 1.5};
    const int len = f32_unit_tiles(cls, fp.n_classes, P.D, sms, max_slots);
    for (int i = 0; i < fp.n_classes; ++i) fp.c[i].n_split = (fp.c[i].n_tiles + len - 1) / len;
    // Longest units first (a dV tile is two thirds of the others' MMAs).
    auto cost = [](const FBClass& x) { return (double)x.n_tiles / x.n_split * (x.kind == kDv ? 2 : 3); };
    for (int i = 0; i < fp.n_classes; ++i)
        for (int k = i + 1; k < fp.n_classes; ++k)
            if (cost(fp.c[k]) > cost(fp.c[i])) {
                const FBClass t = fp.c[i];
                fp.c[i] = fp.c[k];
                fp.c[k] = t;
            }
    int units = 0, slots = 0, merges = 0;
    for (int i = 0; i < fp.n_classes; ++i) {
        FBClass& cl = fp.c[i];
        cl.unit_base = units;
        cl.slot_base = slots;
        cl.item_base = merges;
        units += cl.n_own * HB * cl.n_split;
        if (cl.n_split > 1) {
            slots += cl.n_own * HB * cl.n_split;
            merges += cl.n_own * HB;
        }
    }
    if (slots > max_slots) return MSF_ERR_STATE;
    if (units == 0) return MSF_OK;
    e = launch_split_planes(sp, c.scale_log2, &fp.range, st);
    if (e != cudaSuccess) return fail(e);
    *range = fp.range;
    const bool d128 = P.D == 128;
    const int smem = d128 ? FBCfg<128>::kSmem : FBCfg<64>::kSmem;
    const void* fn = d128 ? (const void*)bwd_f32_kernel<128> : (const void*)bwd_f32_kernel<64>;
    e = set_smem_attr(fn, smem, -1, kLaunchRegs);
    if (e != cudaSuccess) return fail(e);
    e = d128 ? launch_pdl(bwd_f32_kernel<128>, dim3((unsigned)units), dim3(kThreads), smem, st, maps, fp)
             : launch_pdl(bwd_f32_kernel<64>, dim3((unsigned)units), dim3(kThreads), smem, st, maps, fp);
    if (e == cudaSuccess && merges > 0)
        e = d128 ? launch_pdl(bwd_f32_merge_kernel<128>, dim3((unsigned)merges, 8), dim3(256), 0, st, fp)
                 : launch_pdl(bwd_f32_merge_kernel<64>, dim3((unsigned)merges, 8), dim3(256), 0, st, fp);
    return e == cudaSuccess ? MSF_OK : fail(e);
}

}  // namespace msf
