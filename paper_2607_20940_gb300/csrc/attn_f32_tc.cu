// fp32 MSSA attention on the sm_103a tensor cores.
//
// Every fp32 operand x is held as three bf16 planes h + m + l (h = bf16(x),
// m = bf16(x - h), l = bf16(x - h - m): the differences are exact and the three
// 8-bit significands cover fp32's 24 bits), and a product of two operands as
// the six plane products whose size is above 2^-24 of it:
//   x y = hl + mm + hm + lh + mh + hh   (lm, ml, ll are below fp32's rounding).
// bf16 products are exact and tcgen05 accumulates them in fp32, the small
// terms first, so that only the eight K steps of hh (of a 128-wide
// contraction) add at full size. The accumulators never carry over K/V tiles:
// S is one tile's scores, and each tile's P V is read out and added to the
// running output in fp32 registers. Against 64 bits the result is closer than
// the CUDA-core kernel's on every size tried (480p layer: relative error
// 5.5e-7 against 2.0e-6), and the 480p layer (202.8 GFLOP) takes 0.78 ms
// against 13.9 ms.
//
// split_planes_kernel  reads q and the context's k, v once and writes the
//                      planes [B, 3, rows, H, D] into the workspace.
// mssa_f32_kernel      one unit = one 128-row query tile of one (stream, head,
//                      group) and a range of its 128-row K/V tiles. 384
//                      threads: warp 0 TMA producer (Q's three planes once,
//                      then planes through a 4-deep ring of 128-row tiles),
//                      warp 1 MMA issuer, warp 2 TMEM, warps 4-11 softmax (a
//                      thread per query row and column half).
// merge_f32_kernel     sums the units of a split query tile.
//
// Bound: the tensor pipe, 96 MMAs per 128 x 128 pair tile at D = 128 (six
// times the bf16 kernel's 16), 6144 cycles at 64 per MMA, which a probe that only
// issues them reaches. The softmax
// (exponentials, the three-way split of P, the read-out of O) takes about a
// third of that and runs beside it: S of tile j+1 is issued before P V of
// tile j, into the other S buffer.
// TMEM columns: two S buffers of 192 (128 scores; the planes of P are written
// over them and over 64 more), O from 384.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "attn_f32_tc.h"
#include "attn_tc.h"
#include "f32_range.cuh"
#include "ptx.cuh"
#include "sched.h"

namespace msf {
namespace {

constexpr int kBM = 128;       // query rows and context rows per tile
constexpr int kThreads = 384;  // 12 warps
constexpr int kRing = 4;       // plane tiles in flight
constexpr int kSBuf = 192;     // TMEM columns of one S / P buffer
constexpr int kOCol = 2 * kSBuf;
// 168 registers per thread at launch; the control warpgroup drops to 104 and
// the two softmax warpgroups rise to 192: 4 x 104 + 8 x 192 <= 12 x 168.
constexpr int kLaunchRegs = 168, kCtrlRegs = 104, kSoftmaxRegs = 192;
static_assert(4 * kCtrlRegs + 8 * kSoftmaxRegs <= 12 * kLaunchRegs, "register split");
constexpr long long kWaitLimit = 2000000000LL;  // ~1 s of SM clock

// ------------------------------------------------------------ plane split
__global__ void __launch_bounds__(256) split_planes_kernel(const __grid_constant__ SplitParams p) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    uint32_t codes = 0;
    for (long long i = blockIdx.x * 256 + threadIdx.x; i < p.total; i += gridDim.x * 256) {
        int k = 0;
        while (k + 1 < p.n && i >= p.j[k + 1].base) ++k;
        const SplitJob& J = p.j[k];
        const long long rel = i - J.base;
        const int b = (int)(rel / J.vecs), v = (int)(rel - (long long)b * J.vecs);
        const float4* s = reinterpret_cast<const float4*>(J.src + b * J.src_bstride + 8ll * v);
        const float4 x0 = __ldg(s), x1 = __ldg(s + 1);
        const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
        codes = __vmaxu4(codes, range_code(max(abs_bits4(x0), abs_bits4(x1))) << (8 * J.operand));
        uint32_t h[4], m[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) ptx::split_bf16(x[2 * e], x[2 * e + 1], h[e], m[e], l[e]);
        __nv_bfloat16* d = J.dst + b * J.dst_bstride + 8ll * v;
        *reinterpret_cast<uint4*>(d) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(d + J.dst_plane) = make_uint4(m[0], m[1], m[2], m[3]);
        *reinterpret_cast<uint4*>(d + 2 * J.dst_plane) = make_uint4(l[0], l[1], l[2], l[3]);
    }
    codes = block_codes(codes);
    if (threadIdx.x == 0) p.words[blockIdx.x] = codes;
}

// --------------------------------------------------------------- attention
struct FSeg {
    int map, row0, len, tile0;
};
struct FGroup {
    int q_begin, q_end;
    int n_qt;       // 128-row query tiles
    int n_seg, n_tiles;
    int n_split;    // units per query tile
    int unit_base;  // first unit (block) of the group
    int slot_base;  // first partial slot (n_split > 1)
    FSeg seg[kMaxSeg];
};
struct FParams {
    int H, B, N;
    float scale_log2;
    int n_groups;
    FGroup g[MSF_MAX_GROUPS];  // longest units first
    float* out;
    float* lse;       // optional [B, H, N]
    float* partials;  // [slot]([128][D] output, [128] running max, [128] sum)
    F32Range range;
    unsigned int* status;
    long long wait_limit;
};
template <int D>
struct FCfg {
    static constexpr int kTile = kBM * D * 2;  // one plane of one 128-row tile
    static constexpr int kSmem = (3 + kRing) * kTile + 1024;
    static constexpr int kSlot = kBM * (D + 2);  // floats of a partial slot
};
static_assert(FCfg<128>::kSmem + 2048 <= 227 * 1024, "shared memory of the launch");

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    mssa_f32_kernel(const __grid_constant__ F32Maps maps, const __grid_constant__ FParams p) {
    using C = FCfg<D>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sQ = smem;                // [3] planes h, m, l
    unsigned char* sR = smem + 3 * C::kTile;  // [kRing]
    __shared__ uint64_t q_full, full[kRing], empty[kRing], p_full, o_full, meet_bar, drain_bar;
    // Scores ready, per S buffer: S of tile j + 1 may be ready before a softmax
    // warp has looked for tile j's, so one barrier could run two phases ahead.
    __shared__ uint64_t s_full[2];
    __shared__ float sx[2][kBM];  // row maxima, at the end row sums, of the two column halves
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    int gi = 0;
    while (gi + 1 < p.n_groups && (int)blockIdx.x >= p.g[gi + 1].unit_base) ++gi;
    const FGroup& G = p.g[gi];
    // units of one head in order split, query tile: neighbours share K/V tiles in L2
    const int local = (int)blockIdx.x - G.unit_base;
    const int qt = local % G.n_qt;
    const int split = (local / G.n_qt) % G.n_split;
    const int bh = local / (G.n_qt * G.n_split);
    const int h = bh % p.H, b = bh / p.H;
    const int q_row0 = G.q_begin + qt * kBM;
    const int u0 = split * G.n_tiles / G.n_split, u1 = (split + 1) * G.n_tiles / G.n_split;
    const int n = u1 - u0;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        ptx::mbar_init(&q_full, 1);
        for (int s = 0; s < kRing; ++s) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&empty[s], 1);
        }
        ptx::mbar_init(&s_full[0], 1);
        ptx::mbar_init(&s_full[1], 1);
        ptx::mbar_init(&p_full, 8);
        ptx::mbar_init(&o_full, 1);
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
    const bool skip = !planes_hold(p.range);  // the CUDA-core kernel answers instead

    auto tile_of = [&](int u, int& map, int& row, int& valid) {
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
            ptx::mbar_arrive_expect_tx(&q_full, 3 * C::kTile);
            for (int pl = 0; pl < 3; ++pl)
                for (int c = 0; c < D / 64; ++c)
                    ptx::tma_load_4d(sQ + pl * C::kTile + c * (kBM * 128), &maps.q, &q_full, c * 64, h, q_row0,
                                     3 * b + pl);
            int it = 0;  // plane tiles issued
            // the planes of one K or V tile, smallest first
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
            int map, row, valid;
            tile_of(u0, map, row, valid);
            ok = planes(&maps.k[map], row);
            for (int u = u0; u < u1 && ok; ++u) {
                if (u + 1 < u1) {
                    tile_of(u + 1, map, row, valid);
                    ok = planes(&maps.k[map], row);
                }
                tile_of(u, map, row, valid);
                ok = ok && planes(&maps.v[map], row);
            }
            if (!ok) {
                // every copy issued lands before the CTA exits
                ptx::mbar_wait_bounded(&q_full, 0, &never, kWaitLimit);
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
        const uint64_t q_desc = ptx::sdesc_sw128(ptx::smem_u32(sQ), 16, 1024);
        const uint64_t k_desc = ptx::sdesc_sw128(ptx::smem_u32(sR), 16, 1024);
        const uint64_t v_desc = ptx::sdesc_sw128(ptx::smem_u32(sR), kBM * 128, 1024);
        auto wait_all = [&](uint64_t* bar, uint32_t parity) {
            const bool r = ptx::mbar_wait_bounded(bar, parity, abort_p, p.wait_limit);
            return __all_sync(0xffffffffu, r);
        };
        int it = 0;
        // S = Q K^T of tile j into its buffer. With K's plane kp the planes of Q
        // from 2 - kp down to h: (h; l), (m, h; m), (l, m, h; h).
        auto scores = [&](int j) {
            const uint32_t d = tbase + (uint32_t)((j & 1) * kSBuf);
            for (int kp = 2; kp >= 0; --kp, ++it) {
                const int st = it % kRing;
                if (!wait_all(&full[st], (uint32_t)((it / kRing) & 1))) return false;
                ptx::tc_fence_after();
                if (ptx::elect_one_sync()) {
                    const uint64_t kd = k_desc + (uint64_t)st * kTileDesc;
                    for (int qp = 2 - kp; qp >= 0; --qp) {
                        const uint64_t qd = q_desc + (uint64_t)qp * kTileDesc;
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            const uint64_t off = (uint64_t)(((kk / 4) * (kBM * 128) + (kk % 4) * 32) >> 4);
                            ptx::mma_ss(d, qd + off, kd + off, idS, (kp < 2 || kk > 0) ? 1u : 0u);
                        }
                    }
                    ptx::mma_commit(&empty[st]);
                    if (kp == 0) ptx::mma_commit(&s_full[j & 1]);
                }
                __syncwarp();
            }
            return true;
        };
        bool ok = wait_all(&q_full, 0) && scores(0);
        for (int j = 0; j < n && ok; ++j) {
            if (j + 1 < n) ok = scores(j + 1);
            ok = ok && wait_all(&p_full, (uint32_t)(j & 1));
            // O = P V of tile j alone; p_full also says that the softmax has
            // read O of tile j - 1
            for (int vp = 2; vp >= 0 && ok; --vp, ++it) {
                const int st = it % kRing;
                ok = wait_all(&full[st], (uint32_t)((it / kRing) & 1));
                if (!ok) break;
                ptx::tc_fence_after();
                if (ptx::elect_one_sync()) {
                    const uint64_t vd = v_desc + (uint64_t)st * kTileDesc;
                    const uint32_t a0 = tbase + (uint32_t)((j & 1) * kSBuf);
                    for (int pp = 2 - vp; pp >= 0; --pp) {
#pragma unroll
                        for (int kk = 0; kk < kBM / 16; ++kk) {
                            // plane h, m: columns 64 half + 0 / 32; plane l: 128 + 32 half
                            const uint32_t half = kk / 4, c = (kk % 4) * 8;
                            const uint32_t a = a0 + c + (pp == 2 ? 128 + 32 * half : 64 * half + 32 * pp);
                            ptx::mma_ts(tbase + kOCol, a, vd + (uint64_t)(kk * (2048 >> 4)), idO,
                                        (vp < 2 || kk > 0) ? 1u : 0u);
                        }
                    }
                    ptx::mma_commit(&empty[st]);
                    if (vp == 0) ptx::mma_commit(&o_full);
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
        // ========== softmax: one thread per query row and column half ==========
        const int half = (warp - 4) / 4, wq = warp % 4;
        const int r = wq * 32 + lane;
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        constexpr int DH = D / 2;  // output columns of this thread
        const uint32_t tO = tbase + kOCol + DH * half + lane_off;
        const float sl2 = p.scale_log2;
        float acc[DH];
#pragma unroll
        for (int e = 0; e < DH; ++e) acc[e] = 0.f;
        float m = -INFINITY, l = 0.f;
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
            ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&s_full[j & 1], (uint32_t)((j >> 1) & 1), abort_p, p.wait_limit));
            if (!ok) break;
            ptx::tc_fence_after();
            const uint32_t tS = tbase + (uint32_t)((j & 1) * kSBuf) + 64 * half + lane_off;
            const uint32_t tL = tbase + (uint32_t)((j & 1) * kSBuf) + 128 + 32 * half + lane_off;
            uint32_t s[2][32];
            ptx::tmem_ld32(tS, s[0]);
            ptx::tmem_ld32(tS + 32, s[1]);
            ptx::tmem_wait_ld();
            const int lim = valid - 64 * half;
            if (lim < 64) {
                // context rows past the segment's end: score -inf, probability 0
#pragma unroll
                for (int e = 0; e < 64; ++e)
                    if (e >= lim) s[e >> 5][e & 31] = 0xff800000u;
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int e = 0; e < 64; e += 2)
                mx[(e >> 1) & 3] = ptx::fmax3(mx[(e >> 1) & 3], __uint_as_float(s[e >> 5][e & 31]),
                                              __uint_as_float(s[e >> 5][(e & 31) + 1]));
            const float own = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            // The halves share the row's maximum; both have read their scores
            // when they meet, so P may overwrite them.
            sx[half][r] = own;
            ok = meet();
            if (!ok) break;
            const float m_new = fmaxf(m, fmaxf(own, sx[half ^ 1][r]) * sl2);
            const float corr = ex2(m - m_new);
            m = m_new;
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t ph[16], pm[16], pl[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float p0 = ex2(fmaf(__uint_as_float(s[c][2 * e]), sl2, -m));
                    const float p1 = ex2(fmaf(__uint_as_float(s[c][2 * e + 1]), sl2, -m));
                    sum[(2 * e) & 3] += p0;
                    sum[(2 * e + 1) & 3] += p1;
                    ptx::split_bf16(p0, p1, ph[e], pm[e], pl[e]);
                }
                ptx::tmem_st16(tS + 16 * c, ph);
                ptx::tmem_st16(tS + 32 + 16 * c, pm);
                ptx::tmem_st16(tL + 16 * c, pl);
            }
            l = fmaf(l, corr, (sum[0] + sum[1]) + (sum[2] + sum[3]));
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&p_full);
            ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&o_full, (uint32_t)(j & 1), abort_p, p.wait_limit));
            if (!ok) break;
            ptx::tc_fence_after();
#pragma unroll
            for (int c = 0; c < DH / 32; ++c) {
                uint32_t o[32];
                ptx::tmem_ld32(tO + 32 * c, o);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[32 * c + e] = fmaf(acc[32 * c + e], corr, __uint_as_float(o[e]));
            }
            ptx::tc_fence_before();
        }
        if (ok) {
            sx[half][r] = l;
            ok = meet();
        }
        if (ok) {
            l += sx[half ^ 1][r];
            const int q = q_row0 + r;
            float4* dst = nullptr;
            float mul = 1.f;
            if (G.n_split > 1) {
                float* slot = p.partials + (size_t)(G.slot_base + local) * C::kSlot;
                dst = reinterpret_cast<float4*>(slot + r * D + DH * half);
                if (half == 0) {
                    slot[kBM * D + r] = m;
                    slot[kBM * D + kBM + r] = l;
                }
            } else if (q < G.q_end) {
                dst = reinterpret_cast<float4*>(p.out + (((size_t)b * p.N + q) * p.H + h) * D + DH * half);
                mul = 1.0f / l;
                if (p.lse && half == 0)
                    p.lse[((size_t)b * p.H + h) * p.N + q] = (m + log2f(l)) * 0.6931471805599453f;
            }
            if (dst) {
#pragma unroll
                for (int e = 0; e < DH / 4; ++e)
                    dst[e] = make_float4(acc[4 * e] * mul, acc[4 * e + 1] * mul, acc[4 * e + 2] * mul,
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

// Query tiles in several units: out = sum_i 2^(m_i - M) O_i / sum_i 2^(m_i - M) l_i
// in unit order. One block per query tile, one warp per row at a time.
template <int D>
__global__ void __launch_bounds__(256) merge_f32_kernel(const __grid_constant__ FParams p) {
    using C = FCfg<D>;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (!planes_held(p.range)) return;
    int tile = blockIdx.x, gi = 0;
    for (; gi < p.n_groups; ++gi) {
        const int nt = p.g[gi].n_split > 1 ? p.g[gi].n_qt * p.H * p.B : 0;
        if (tile < nt) break;
        tile -= nt;
    }
    if (gi >= p.n_groups) return;
    const FGroup& G = p.g[gi];
    const int qt = tile % G.n_qt, bh = tile / G.n_qt;
    const int h = bh % p.H, b = bh / p.H;
    const float* first = p.partials + (size_t)(G.slot_base + bh * G.n_split * G.n_qt + qt) * C::kSlot;
    const size_t step = (size_t)G.n_qt * C::kSlot;  // to the tile's next unit
    const int lane = threadIdx.x % 32;
    constexpr int E = D / 32;
    for (int r = threadIdx.x / 32 + 16 * blockIdx.y; r < 16 * (blockIdx.y + 1); r += 8) {
        const int q = G.q_begin + qt * kBM + r;
        if (q >= G.q_end) break;
        // The units' maxima and sums by lanes, 32 at a time, so that a row costs
        // two round trips to L2 and not two per unit.
        float M = -INFINITY;
        for (int i0 = 0; i0 < G.n_split; i0 += 32) {
            const int i = i0 + lane;
            M = fmaxf(M, i < G.n_split ? __ldcg(first + i * step + kBM * D + r) : -INFINITY);
        }
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, x));
        float L = 0.f, acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = 0.f;
        for (int i0 = 0; i0 < G.n_split; i0 += 32) {
            const int i = i0 + lane, n = min(32, G.n_split - i0);
            const float w_own = i < G.n_split ? ex2(__ldcg(first + i * step + kBM * D + r) - M) : 0.f;
            const float l_own = i < G.n_split ? __ldcg(first + i * step + kBM * D + kBM + r) : 0.f;
#pragma unroll 4
            for (int k = 0; k < n; ++k) {
                const float* s = first + (size_t)(i0 + k) * step + r * D;
                const float w = __shfl_sync(0xffffffffu, w_own, k);
                L = fmaf(w, __shfl_sync(0xffffffffu, l_own, k), L);
                if (E == 4) {
                    const float4 v = __ldcg(reinterpret_cast<const float4*>(s) + lane);
                    acc[0] = fmaf(w, v.x, acc[0]);
                    acc[1] = fmaf(w, v.y, acc[1]);
                    acc[E - 2] = fmaf(w, v.z, acc[E - 2]);
                    acc[E - 1] = fmaf(w, v.w, acc[E - 1]);
                } else {
                    const float2 v = __ldcg(reinterpret_cast<const float2*>(s) + lane);
                    acc[0] = fmaf(w, v.x, acc[0]);
                    acc[1] = fmaf(w, v.y, acc[1]);
                }
            }
        }
        const float inv = 1.0f / L;
        float* dst = p.out + (((size_t)b * p.N + q) * p.H + h) * D + E * lane;
        if (E == 4)
            *reinterpret_cast<float4*>(dst) = make_float4(acc[0] * inv, acc[1] * inv, acc[E - 2] * inv, acc[E - 1] * inv);
        else
            *reinterpret_cast<float2*>(dst) = make_float2(acc[0] * inv, acc[1] * inv);
        if (p.lse && lane == 0)
            p.lse[((size_t)b * p.H + h) * p.N + q] = (M + log2f(L)) * 0.6931471805599453f;
    }
}

// ---------------------------------------------------------------- host side

}  // namespace


// The limit with the earliest estimated end: the units placed longest first on
// the least loaded SM, a unit costing 2 tiles besides its own (the resident
// planes, the pipeline's start, the read-out; D = 64 tiles take half as long:
// 4) and 0.7 more if it writes a partial result, and the merge. Tried: no
// split, one to six units per SM, and the longest that starts all at once.
// Against one split rule (as many rounds as sqrt(tiles per SM / 4)): 480p
// forward 833 -> 775 us, gradient of a small window (1008 tokens) 127 -> 86.
int f32_unit_tiles(const F32Class* c, int n, int D, int sms, int max_slots) {
    double total = 0;
    int longest = 1;
    for (int i = 0; i < n; ++i) {
        total += c[i].items * c[i].n_tiles * c[i].weight;
        longest = c[i].n_tiles > longest ? c[i].n_tiles : longest;
    }
    const double own = D == 64 ? 4.0 : 2.0;
    auto estimate = [&](int len) -> double {
        WorkUnits u[kMaxF32Classes];
        long long slots = 0;
        for (int i = 0; i < n; ++i) {
            const int ns = (c[i].n_tiles + len - 1) / len;
            u[i] = {(double)((c[i].n_tiles + ns - 1) / ns) * c[i].weight + own + (ns > 1 ? 0.7 : 0.0), c[i].items * ns};
            if (ns > 1) slots += u[i].n;
        }
        if (slots > max_slots) return 1e30;
        return lpt_end(u, n, sms) + (slots > 0 ? 1.0 + 0.006 * (double)slots : 0.0);
    };
    int best = longest;
    double least = estimate(longest);
    auto try_len = [&](int len) {
        len = len < 1 ? 1 : len;
        if (len >= longest) return;
        const double e = estimate(len);
        if (e < least) {
            least = e;
            best = len;
        }
    };
    for (int k = 1; k <= kF32MaxRounds; ++k) try_len((int)ceil(total / sms / k));
    // all at once: the shortest limit whose units fit the SMs
    for (int lo = 1, hi = longest; lo < hi;) {
        const int mid = (lo + hi) / 2;
        long long units = 0;
        for (int i = 0; i < n; ++i) units += c[i].items * ((c[i].n_tiles + mid - 1) / mid);
        if (units <= sms)
            hi = mid;
        else
            lo = mid + 1;
        if (lo >= hi) try_len(hi);
    }
    return best;
}

int f32_longest_context(const AttnArgs& a) {
    int longest = 0;
    for (int gi = 0; gi < a.n_groups; ++gi) {
        int n = 0;
        for (int s = 0; s < a.g[gi].n_seg; ++s) n += a.g[gi].seg[s].len;
        longest = n > longest ? n : longest;
    }
    return longest;
}

bool add_planes(const Plan& P, SplitParams& sp, int operand, const void* src, long long src_bstride_bytes, char* dst,
                int alloc, int rows, CUtensorMap* m) {
    const long long rowe = (long long)P.H * P.D;
    SplitJob& j = sp.j[sp.n++];
    j.src = (const float*)src;
    j.dst = (__nv_bfloat16*)dst;
    j.src_bstride = src_bstride_bytes / 4;
    j.dst_plane = alloc * rowe;
    j.dst_bstride = 3 * j.dst_plane;
    j.vecs = (int)(rows * rowe / 8);
    j.operand = operand;
    j.base = sp.total;
    sp.total += (long long)j.vecs * P.B;
    return encode_rows(m, dst, P.D, P.H, rows, 3 * P.B, j.dst_plane * 2);
}

bool add_context_planes(const Plan& P, const AttnArgs& a, SplitParams& sp, F32Maps& maps) {
    const size_t rowe = (size_t)P.H * P.D;
    if (!add_planes(P, sp, kRangeQ, a.q, a.q_bstride, f32_planes(P, kF32Q, 0), P.N, P.N, &maps.q)) return false;
    bool done[kNumMaps] = {false};
    for (int gi = 0; gi < a.n_groups; ++gi)
        for (int s = 0; s < a.g[gi].n_seg; ++s) {
            const Segment& sg = a.g[gi].seg[s];
            const bool pyr = sg.map_id == kMapPyr;
            const int map = pyr ? kMapPyr0 + gi : sg.map_id;
            if (done[map]) continue;
            done[map] = true;
            // rows that the segment's tensor holds: a group's part of the
            // pyramid, the live slots of the ring, else all of it
            const int part = pyr ? kF32Pyr : map == kMapSink ? kF32Sink : map == kMapHist ? kF32Ring : kF32Win;
            const int rows = pyr || map == kMapHist ? sg.len : sg.rows_total;
            const size_t off = pyr ? (size_t)3 * P.B * P.groups[gi].pyr_offset * rowe * 2 : 0;
            const int alloc = pyr ? P.groups[gi].pyr_cap : f32_part_rows(P, part);
            const size_t so = pyr ? (size_t)sg.row0 * rowe * 4 : 0;
            if (!add_planes(P, sp, kRangeK, sg.k + so, sg.bstride, f32_planes(P, part, 0) + off, alloc, rows,
                            &maps.k[map]) ||
                !add_planes(P, sp, kRangeV, sg.v + so, sg.bstride, f32_planes(P, part, 1) + off, alloc, rows,
                            &maps.v[map]))
                return false;
        }
    return true;
}

cudaError_t launch_split_planes(const SplitParams& sp, float scale_log2, F32Range* range, cudaStream_t st) {
    const long long want = (sp.total + 255) / 256;
    range->words = sp.words;
    range->answer = sp.words + kF32SplitBlocks;
    range->n = want < kF32SplitBlocks ? (int)want : kF32SplitBlocks;
    frexpf(scale_log2, &range->scale_exp);
    return launch_pdl(split_planes_kernel, dim3((unsigned)range->n), dim3(256), 0, st, sp);
}

msf_status launch_attn_f32_tc(msf_plan_t plan, const AttnArgs& a, cudaStream_t st) {
    const Plan& P = *plan;
    auto fail = [](cudaError_t e) {
        set_cuda_error((int)e);
        return MSF_ERR_CUDA;
    };
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return fail(e);
    if (sms > kF32MaxSms) sms = kF32MaxSms;
    // So few keys that the CUDA-core kernel is done before the planes are written
    // (24 keys x 64: 8.5 us against 8.9; 12 and 24 keys x 128: 7.1 against 10.4, 12.6
    // against 10.8).
    if (f32_longest_context(a) <= (P.D == 64 ? 24 : 18)) {
        e = launch_attn_simt(a, false, st);
        return e == cudaSuccess ? MSF_OK : fail(e);
    }
    SplitParams sp;
    memset(&sp, 0, sizeof(sp));
    F32Maps maps;
    memset(&maps, 0, sizeof(maps));
    FParams fp;
    memset(&fp, 0, sizeof(fp));
    sp.words = f32_range_words(P);
    if (!add_context_planes(P, a, sp, maps)) return fail(cudaErrorInvalidValue);
    fp.n_groups = a.n_groups;
    for (int gi = 0; gi < a.n_groups; ++gi) {
        const AttnGroup& ag = a.g[gi];
        FGroup& g = fp.g[gi];
        g.q_begin = ag.q_begin;
        g.q_end = ag.q_end;
        g.n_qt = (ag.q_end - ag.q_begin + kBM - 1) / kBM;
        g.n_seg = ag.n_seg;
        for (int s = 0; s < ag.n_seg; ++s) {
            const Segment& sg = ag.seg[s];
            FSeg& fs = g.seg[s];
            const bool pyr = sg.map_id == kMapPyr;
            fs.map = pyr ? kMapPyr0 + gi : sg.map_id;
            fs.row0 = pyr ? 0 : sg.row0;
            fs.len = sg.len;
            fs.tile0 = g.n_tiles;
            g.n_tiles += (sg.len + kBM - 1) / kBM;
        }
    }
    fp.H = P.H;
    fp.B = P.B;
    fp.N = P.N;
    fp.scale_log2 = a.scale_log2;
    fp.out = (float*)a.out;
    fp.lse = a.lse;
    fp.partials = f32_partials(P);
    fp.status = a.status;
    fp.wait_limit = kWaitLimit;
    F32Class cls[MSF_MAX_GROUPS];
    for (int i = 0; i < fp.n_groups; ++i) cls[i] = {(long long)fp.g[i].n_qt * P.H * P.B, fp.g[i].n_tiles, 1.0};
    const int len = f32_unit_tiles(cls, fp.n_groups, P.D, sms, f32_max_slots(P));
    for (int i = 0; i < fp.n_groups; ++i) fp.g[i].n_split = (fp.g[i].n_tiles + len - 1) / len;
    // longest units first
    for (int i = 0; i < fp.n_groups; ++i)
        for (int k = i + 1; k < fp.n_groups; ++k)
            if (fp.g[k].n_tiles * fp.g[i].n_split > fp.g[i].n_tiles * fp.g[k].n_split) {
                const FGroup t = fp.g[i];
                fp.g[i] = fp.g[k];
                fp.g[k] = t;
            }
    int units = 0, slots = 0, merges = 0;
    for (int i = 0; i < fp.n_groups; ++i) {
        FGroup& g = fp.g[i];
        const int items = g.n_qt * P.H * P.B;
        g.unit_base = units;
        g.slot_base = slots;
        units += items * g.n_split;
        if (g.n_split > 1) {
            slots += items * g.n_split;
            merges += items;
        }
    }
    if (units == 0) return MSF_OK;
    if (slots > f32_max_slots(P)) return MSF_ERR_STATE;
    e = launch_split_planes(sp, a.scale_log2, &fp.range, st);
    if (e != cudaSuccess) return fail(e);
    const bool d128 = P.D == 128;
    const int smem = d128 ? FCfg<128>::kSmem : FCfg<64>::kSmem < 120 * 1024 ? 120 * 1024 : FCfg<64>::kSmem;
    const void* fn = d128 ? (const void*)mssa_f32_kernel<128> : (const void*)mssa_f32_kernel<64>;
    e = set_smem_attr(fn, smem, -1, kLaunchRegs);
    if (e != cudaSuccess) return fail(e);
    const dim3 grid((unsigned)units);
    e = d128 ? launch_pdl(mssa_f32_kernel<128>, grid, dim3(kThreads), smem, st, maps, fp)
             : launch_pdl(mssa_f32_kernel<64>, grid, dim3(kThreads), smem, st, maps, fp);
    if (e == cudaSuccess && merges > 0)
        e = d128 ? launch_pdl(merge_f32_kernel<128>, dim3((unsigned)merges, 8), dim3(256), 0, st, fp)
                 : launch_pdl(merge_f32_kernel<64>, dim3((unsigned)merges, 8), dim3(256), 0, st, fp);
    if (e != cudaSuccess) return fail(e);
    AttnArgs fallback = a;
    fallback.unless = fp.range;
    e = launch_attn_simt(fallback, false, st);
    return e == cudaSuccess ? MSF_OK : fail(e);
}

}  // namespace msf
