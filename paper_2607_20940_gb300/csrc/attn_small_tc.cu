// MSSA attention of small calls on the sm_103a tensor cores (bf16 operands,
// fp32 softmax and accumulation; the arithmetic of attn_tc.cu).
//
// Work: one 128-row query tile of one (stream, head, group) per thread-block
// cluster; the tile's 128-row K/V tiles are split over the cluster's CTAs, and
// inside a CTA over two softmax warpgroups (even and odd tiles), each with its
// own scores, running max, sum and output. Every warpgroup leaves its partial
// result in shared memory, and after a cluster barrier each CTA sums its share
// of the rows over distributed shared memory in a fixed order.
//
// Bound: latency. With few query blocks the persistent kernel's stream-K split
// cuts each into pieces of two or three tiles that meet again in global memory
// (a partial write, an atomic and a batch of L2 loads: ~7 us, more than the
// tiles), and its 256-row blocks leave half of the SMs without work.
//
// Roles (384 threads): warp 0 TMA producer (Q once, then K and V through two
// 3-deep rings), warp 1 MMA issuer, warp 2 TMEM, warps 4-7 softmax of the even
// tiles, warps 8-11 of the odd ones (one thread per query row).
// TMEM columns: S0 [0,128) S1 [128,256) O0 [256,256+D) O1 [384,384+D).
// At 168 registers ptxas spills 8 bytes (stored once, 40 loaded).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <type_traits>

#include "attn_small_tc.h"
#include "ptx.cuh"
#include "sched.h"

namespace msf {
namespace {

constexpr int kBM = 128;       // query rows and context rows per tile
constexpr int kThreads = 384;  // 12 warps
constexpr int kRing = 3;       // K and V tiles in flight
constexpr int kMaxCluster = 8;
constexpr long long kWaitLimit = 2000000000LL;  // ~1 s of SM clock
// 168 registers per thread at launch; the control warpgroup drops to 120 and
// the two softmax warpgroups rise to 192: 4 x 120 + 8 x 192 <= 12 x 168.
constexpr int kLaunchRegs = 168, kCtrlRegs = 120, kSoftmaxRegs = 192;
static_assert(4 * kCtrlRegs + 8 * kSoftmaxRegs <= 12 * kLaunchRegs, "register split");

struct SmallParams {
    int H, B, N;
    float scale_log2;
    int n_groups;
    int item_base[MSF_MAX_GROUPS];  // first query tile of a group, over all streams and heads
    int n_qt[MSF_MAX_GROUPS];
    TcGroup g[MSF_MAX_GROUPS];
    __nv_bfloat16* out;
    float* lse;  // optional [B, H, N]
    unsigned int* status;
    long long wait_limit;
};

template <int D>
struct SCfg {
    static constexpr int kTile = kBM * D * 2;
    static constexpr int kRow = D + 4;  // floats of a staged row (the padding spreads the banks)
    static constexpr int kPart = kBM * kRow * 4;
    static constexpr int kUsed = (1 + 2 * kRing) * kTile + 1024;
    static constexpr int kSmem = kUsed > 120 * 1024 ? kUsed : 120 * 1024;  // one CTA per SM (512 TMEM columns)
};
static_assert(2 * SCfg<128>::kPart + kBM * 16 <= SCfg<128>::kSmem - 1024 &&
                  2 * SCfg<64>::kPart + kBM * 16 <= SCfg<64>::kSmem - 1024,
              "the partial results fit the tiles' space");
static_assert(SCfg<128>::kSmem + 1024 <= 227 * 1024, "shared memory of the launch");

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    mssa_small_kernel(const __grid_constant__ TcMaps maps, const __grid_constant__ SmallParams p, int cluster) {
    using C = SCfg<D>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sQ = smem;
    unsigned char* sK = smem + C::kTile;                // [kRing]
    unsigned char* sV = smem + (1 + kRing) * C::kTile;  // [kRing]
    float* part = reinterpret_cast<float*>(smem);       // [2][128][kRow] once every MMA is done
    __shared__ uint64_t q_full, k_full[kRing], k_empty[kRing], v_full[kRing], v_empty[kRing];
    __shared__ uint64_t s_full[2], p_full[2], o_full;
    float(*ml)[4] = reinterpret_cast<float(*)[4]>(smem + 2 * C::kPart);  // per row: max, sum of warpgroup 0, of 1
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int item = (int)blockIdx.x / cluster, rank = (int)blockIdx.x % cluster;
    int gi = 0;
    while (gi + 1 < p.n_groups && item >= p.item_base[gi + 1]) ++gi;
    const TcGroup& G = p.g[gi];
    const int local = item - p.item_base[gi];
    const int qt = local % p.n_qt[gi];
    const int h = (local / p.n_qt[gi]) % p.H, b = local / (p.n_qt[gi] * p.H);
    const int q_row0 = G.q_begin + qt * kBM;
    const int u0 = rank * G.n_tiles / cluster;
    const int n = (rank + 1) * G.n_tiles / cluster - u0;  // 0 when the context has fewer tiles than CTAs

    if (threadIdx.x == 0) {
        abort_flag = 0;
        ptx::mbar_init(&q_full, 1);
        for (int s = 0; s < kRing; ++s) {
            ptx::mbar_init(&k_full[s], 1);
            ptx::mbar_init(&k_empty[s], 1);
            ptx::mbar_init(&v_full[s], 1);
            ptx::mbar_init(&v_empty[s], 1);
        }
        for (int t = 0; t < 2; ++t) {
            ptx::mbar_init(&s_full[t], 1);
            ptx::mbar_init(&p_full[t], 4);
        }
        ptx::mbar_init(&o_full, 1);
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

    // segment map, first row and valid rows of K/V tile u
    auto tile_of = [&](int u, int& map, int& row, int& valid) {
        int s = 0;
        while (s < G.n_seg - 1 && u >= G.seg[s + 1].tile0) ++s;
        const int kt = u - G.seg[s].tile0;
        map = G.seg[s].map;
        row = G.seg[s].row0 + kt * kBM;
        valid = min(kBM, G.seg[s].len - kt * kBM);
    };
    auto load = [&](unsigned char* dst, const CUtensorMap* m, uint64_t* bar, int row) {
        for (int c = 0; c < D / 64; ++c) ptx::tma_load_4d(dst + c * (kBM * 128), m, bar, c * 64, h, row, b);
    };

    bool ok = true;
    if (warp < 4) {
        ptx::setmaxnreg_dec<kCtrlRegs>();
        if (warp == 0 && n > 0) {
            // ============================ TMA producer ============================
            if (lane == 0) {
                ptx::mbar_arrive_expect_tx(&q_full, C::kTile);
                load(sQ, &maps.q, &q_full, q_row0);
                int nk = 0, nv = 0;
                for (int v = 0; v < n; ++v) {
                    int map, row, valid;
                    tile_of(u0 + v, map, row, valid);
                    const int st = v % kRing;
                    const uint32_t par = (uint32_t)(((v / kRing) & 1) ^ 1);
                    if (!ptx::mbar_wait_bounded(&k_empty[st], par, abort_p, p.wait_limit)) {
                        ok = false;
                        break;
                    }
                    ptx::mbar_arrive_expect_tx(&k_full[st], C::kTile);
                    load(sK + st * C::kTile, &maps.k[map], &k_full[st], row);
                    ++nk;
                    if (!ptx::mbar_wait_bounded(&v_empty[st], par, abort_p, p.wait_limit)) {
                        ok = false;
                        break;
                    }
                    ptx::mbar_arrive_expect_tx(&v_full[st], C::kTile);
                    load(sV + st * C::kTile, &maps.v[map], &v_full[st], row);
                    ++nv;
                }
                if (!ok) {
                    // every copy issued lands before the space is used again
                    ptx::mbar_wait_bounded(&q_full, 0, &never, kWaitLimit);
                    for (int i = (nk > kRing ? nk - kRing : 0); i < nk; ++i)
                        ptx::mbar_wait_bounded(&k_full[i % kRing], (uint32_t)((i / kRing) & 1), &never, kWaitLimit);
                    for (int i = (nv > kRing ? nv - kRing : 0); i < nv; ++i)
                        ptx::mbar_wait_bounded(&v_full[i % kRing], (uint32_t)((i / kRing) & 1), &never, kWaitLimit);
                    atomicOr(p.status, kDevTimeout);
                }
            }
        } else if (warp == 1 && n > 0) {
            // ============================= MMA issuer =============================
            constexpr uint32_t idS = ptx::idesc_bf16(kBM, kBM, false, false);
            constexpr uint32_t idO = ptx::idesc_bf16(kBM, D, false, true);
            constexpr uint64_t kTileDesc = (uint64_t)(C::kTile >> 4);
            const uint64_t q_desc = ptx::sdesc_sw128(ptx::smem_u32(sQ), 16, 1024);
            const uint64_t k_desc = ptx::sdesc_sw128(ptx::smem_u32(sK), 16, 1024);
            const uint64_t v_desc = ptx::sdesc_sw128(ptx::smem_u32(sV), kBM * 128, 1024);
            auto wait_all = [&](uint64_t* bar, uint32_t parity) {
                const bool r = ptx::mbar_wait_bounded(bar, parity, abort_p, p.wait_limit);
                return __all_sync(0xffffffffu, r);
            };
            auto scores = [&](int v) {  // S_t = Q K_v^T, t = v & 1
                const int st = v % kRing;
                if (!wait_all(&k_full[st], (uint32_t)((v / kRing) & 1))) return false;
                ptx::tc_fence_after();
                if (ptx::elect_one_sync()) {
                    const uint64_t kd = k_desc + (uint64_t)st * kTileDesc;
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint64_t off = (uint64_t)(((kk / 4) * (kBM * 128) + (kk % 4) * 32) >> 4);
                        ptx::mma_ss(tbase + (v & 1) * 128, q_desc + off, kd + off, idS, kk > 0 ? 1u : 0u);
                    }
                    ptx::mma_commit(&k_empty[st]);
                    ptx::mma_commit(&s_full[v & 1]);  // also covers P V of tile v - 2
                }
                __syncwarp();
                return true;
            };
            ok = wait_all(&q_full, 0) && scores(0);
            if (ok && n > 1) ok = scores(1);
            for (int v = 0; v < n && ok; ++v) {
                const int st = v % kRing, t = v & 1;
                ok = wait_all(&v_full[st], (uint32_t)((v / kRing) & 1)) && wait_all(&p_full[t], (uint32_t)((v >> 1) & 1));
                if (!ok) break;
                ptx::tc_fence_after();
                if (ptx::elect_one_sync()) {
                    const uint64_t vd = v_desc + (uint64_t)st * kTileDesc;
#pragma unroll
                    for (int kk = 0; kk < kBM / 16; ++kk)
                        ptx::mma_ts(tbase + 256 + t * 128, tbase + t * 128 + kk * 8, vd + (uint64_t)(kk * (2048 >> 4)),
                                    idO, (v > 1 || kk > 0) ? 1u : 0u);
                    ptx::mma_commit(&v_empty[st]);
                }
                __syncwarp();
                if (v + 2 < n) ok = scores(v + 2);
            }
            // also after an abort: every MMA is done when o_full completes
            if (ptx::elect_one_sync()) ptx::mma_commit(&o_full);
            __syncwarp();
            if (!ok && lane == 0) atomicOr(p.status, kDevTimeout);
        }
        __syncwarp();
        ptx::cluster_sync();  // the partial results are staged (below)
    } else {
        ptx::setmaxnreg_inc<kSoftmaxRegs>();
        // =================== softmax: one thread per query row ===================
        const int t = (warp - 4) / 4, wq = warp % 4;
        const int r = wq * 32 + lane;
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        const uint32_t tS = tbase + t * 128 + lane_off, tO = tbase + 256 + t * 128 + lane_off;
        const float sl2 = p.scale_log2;
        float m_used = -INFINITY, l = 0.f;
        int j = 0;  // this warpgroup's tiles done
        for (int v = t; v < n; v += 2, ++j) {
            int map, row, valid;
            tile_of(u0 + v, map, row, valid);
            ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&s_full[t], (uint32_t)(j & 1), abort_p, p.wait_limit));
            if (!ok) break;
            ptx::tc_fence_after();
            uint32_t s[4][32];
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) ptx::tmem_ld32(tS + 32 * q4, s[q4]);
            ptx::tmem_wait_ld();
            if (valid < kBM) {
                // rows past the segment's end: score -inf, probability 0
#pragma unroll
                for (int c = 0; c < 128; ++c)
                    if (c >= valid) s[c >> 5][c & 31] = 0xff800000u;
            }
            // The running maximum may lag the row's, as in the persistent
            // kernel: it changes only a power of two common to P, O and l, and
            // is brought up to date when a tile's sum passes 2^32.
            auto tile_max = [&]() -> float {
                float mx[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) mx[e] = -INFINITY;
#pragma unroll
                for (int c = 0; c < 128; c += 2)
                    mx[(c >> 1) & 7] = ptx::fmax3(mx[(c >> 1) & 7], __uint_as_float(s[c >> 5][c & 31]),
                                                  __uint_as_float(s[c >> 5][(c & 31) + 1]));
                return fmaxf(ptx::fmax3(mx[0], mx[1], mx[2]),
                             fmaxf(ptx::fmax3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7]))) * sl2;
            };
            if (j == 0) m_used = tile_max();
            uint64_t sum2[2];
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                const float nm = -m_used;
                const uint64_t sl2x2 = ptx::f2_pack(sl2, sl2), nmx2 = ptx::f2_pack(nm, nm);
                sum2[0] = sum2[1] = ptx::f2_pack(0.f, 0.f);
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    uint32_t pk[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const uint64_t arg = ptx::f2_fma(
                            ptx::f2_pack(__uint_as_float(s[q4][2 * c]), __uint_as_float(s[q4][2 * c + 1])), sl2x2, nmx2);
                        float a0, a1;
                        ptx::f2_unpack(arg, a0, a1);
                        const float p0 = ex2(a0), p1 = ex2(a1);
                        sum2[c & 1] = ptx::f2_add(sum2[c & 1], ptx::f2_pack(p0, p1));
                        pk[c] = ptx::pack_bf16(p0, p1);
                    }
                    ptx::tmem_st16(tS + 16 * q4, pk);
                }
                if (pass == 1) break;
                float a0, a1, b0, b1;
                ptx::f2_unpack(sum2[0], a0, a1);
                ptx::f2_unpack(sum2[1], b0, b1);
                const float tile_sum = (a0 + a1) + (b0 + b1);
                if (!__any_sync(0xffffffffu, !(tile_sum <= 4294967296.0f))) break;
                // O_t holds every P V up to this warpgroup's last tile (the
                // commit of these scores covers it).
                const float m_new = fmaxf(m_used, tile_max());
                const float f = ex2(m_used - m_new);
                l *= f;
                m_used = m_new;
                if (j > 0) {
#pragma unroll 1
                    for (int c = 0; c < D / 16; ++c) {
                        uint32_t o[16];
                        ptx::tmem_ld16(tO + c * 16, o);
                        ptx::tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * f);
                        ptx::tmem_st16(tO + c * 16, o);
                    }
                }
                ptx::tmem_wait_st();  // P of the first pass is overwritten after this
            }
            {
                float a0, a1, b0, b1;
                ptx::f2_unpack(sum2[0], a0, a1);
                ptx::f2_unpack(sum2[1], b0, b1);
                l += (a0 + a1) + (b0 + b1);
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&p_full[t]);
        }
        // ---- this warpgroup's partial result into the tiles' space
        if (n > 0) ok = ok && ptx::mbar_wait_bounded(&o_full, 0, abort_p, p.wait_limit);
        ok = __all_sync(0xffffffffu, ok);
        ptx::tc_fence_after();
        if (ok) {
            *reinterpret_cast<float2*>(&ml[r][2 * t]) = make_float2(m_used, l);
            float4* dst = reinterpret_cast<float4*>(part + (size_t)t * kBM * C::kRow + r * C::kRow);
            uint32_t o[D / 32][32];
            if (j > 0) {
#pragma unroll
                for (int c = 0; c < D / 32; ++c) ptx::tmem_ld32(tO + 32 * c, o[c]);
                ptx::tmem_wait_ld();
            } else {  // no tile: weight 0
#pragma unroll
                for (int c = 0; c < D / 32; ++c)
#pragma unroll
                    for (int e = 0; e < 32; ++e) o[c][e] = 0u;
            }
#pragma unroll
            for (int c = 0; c < D / 32; ++c)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    dst[8 * c + e] = make_float4(__uint_as_float(o[c][4 * e]), __uint_as_float(o[c][4 * e + 1]),
                                                 __uint_as_float(o[c][4 * e + 2]), __uint_as_float(o[c][4 * e + 3]));
        } else if (lane == 0) {
            atomicOr(p.status, kDevTimeout);
        }
        // Every thread of every CTA of the cluster: the partial results are
        // staged. (The sums stay in this branch, whose registers they need.)
        __syncwarp();
        ptx::tc_fence_before();
        ptx::cluster_sync();
        // ---- rows [rank * R, rank * R + R): the 2 * cluster partial results in
        // order of CTA and warpgroup
        const int R = kBM / cluster;
        constexpr int kVec = D / 4;  // float4 per row
        for (int x = (int)threadIdx.x - 128; x < R * kVec; x += 256) {
            const int row = rank * R + x / kVec, c4 = x % kVec;
            const int q = q_row0 + row;
            if (q >= G.q_end) continue;
            float M, L = 0.f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            auto add = [&](const float4& w, const float4& o0, const float4& o1) {  // w: max, sum, max, sum
                const float a = ex2(w.x - M), c = ex2(w.z - M);
                L = fmaf(c, w.w, fmaf(a, w.y, L));
                acc.x = fmaf(c, o1.x, fmaf(a, o0.x, acc.x));
                acc.y = fmaf(c, o1.y, fmaf(a, o0.y, acc.y));
                acc.z = fmaf(c, o1.z, fmaf(a, o0.z, acc.z));
                acc.w = fmaf(c, o1.w, fmaf(a, o0.w, acc.w));
            };
            const float* p0 = part + row * C::kRow + 4 * c4;
            const float* p1 = p0 + kBM * C::kRow;
            if (cluster == 1) {
                const float4 w = *reinterpret_cast<const float4*>(&ml[row][0]);
                M = fmaxf(w.x, w.z);
                add(w, *reinterpret_cast<const float4*>(p0), *reinterpret_cast<const float4*>(p1));
            } else {
                // Everything this thread needs of every CTA is asked for at once.
                auto sum = [&](auto size) {
                    constexpr int kC = decltype(size)::value;
                    float4 w[kC], o0[kC], o1[kC];
#pragma unroll
                    for (int k = 0; k < kC; ++k) {
                        w[k] = ptx::ld_cluster_f4(&ml[row][0], (uint32_t)k);
                        o0[k] = ptx::ld_cluster_f4(p0, (uint32_t)k);
                        o1[k] = ptx::ld_cluster_f4(p1, (uint32_t)k);
                    }
                    M = -INFINITY;
#pragma unroll
                    for (int k = 0; k < kC; ++k) M = ptx::fmax3(M, w[k].x, w[k].z);
#pragma unroll
                    for (int k = 0; k < kC; ++k) add(w[k], o0[k], o1[k]);
                };
                if (cluster == 2)
                    sum(std::integral_constant<int, 2>{});
                else if (cluster == 4)
                    sum(std::integral_constant<int, 4>{});
                else
                    sum(std::integral_constant<int, kMaxCluster>{});
            }
            const float inv = 1.0f / L;
            *reinterpret_cast<uint2*>(p.out + (((size_t)b * p.N + q) * p.H + h) * D + 4 * c4) =
                make_uint2(ptx::pack_bf16(acc.x * inv, acc.y * inv), ptx::pack_bf16(acc.z * inv, acc.w * inv));
            if (p.lse && c4 == 0)
                p.lse[((size_t)b * p.H + h) * p.N + q] = (M + log2f(L)) * 0.6931471805599453f;
        }
    }
    // No CTA leaves while another may still read its shared memory.
    ptx::cluster_sync();
    if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tbase, 512);
    }
}

}  // namespace

// The rule: the estimate of this kernel's end (its clusters placed longest
// first; clusters of four and eight leave some SMs of a GPC over) against the
// persistent kernel's. Microseconds fitted on a GB300 over 660 drawn windows of
// 0.01 to 600 GFLOP, each timed in every form that it can take: a start and a step
// of two K/V tiles (median 1.02 of the measured time, 0.95 to 1.2 for nine of ten of
// 500 others). 8 heads x 64,
// 24 tiles, cluster 2: 14.2 us against 20.1 of the even split; one query tile a
// head, 32 tiles, cluster 8: 13.3 against 58.2; 96 query tiles of 49 K/V tiles: 50
// against 38.4, which the estimates tell apart. More than one round has to win by a
// tenth; of two sizes that end together the larger is taken (one pair of tiles: 9.2
// us on one CTA, 8.6 on two).
int attn_small_cluster(const TcGroup* g, int n_groups, int H, int B, int D, int sms, double persistent_us) {
    long long items = 0;  // 128-row query tiles
    int longest = 0;
    for (int i = 0; i < n_groups; ++i) {
        const int nq = g[i].q_end - g[i].q_begin;
        items += (long long)((nq + kBM - 1) / kBM) * H * B;
        longest = g[i].n_tiles > longest ? g[i].n_tiles : longest;
    }
    if (items > 2 * sms) return 0;
    const double step = D == 64 ? 1.34 : 1.67;
    double best = persistent_us;
    int cluster = 0;
    for (int c = 1; c <= kMaxCluster && (c == 1 || c <= longest); c *= 2) {
        const int places = (c <= 2 ? sms : sms * 5 / 6) / c;
        if (c > 1 && items > places) break;
        const double start = D == 64 ? (c == 8 ? 7.1 : 5.7) : (c == 8 ? 9.8 : 7.7);
        WorkUnits u[MSF_MAX_GROUPS];
        for (int i = 0; i < n_groups; ++i)
            u[i] = {start + step * ((g[i].n_tiles + 2 * c - 1) / (2 * c)),
                    (long long)((g[i].q_end - g[i].q_begin + kBM - 1) / kBM) * H * B};
        const double t = lpt_end(u, n_groups, places) * (items > places ? 1.1 : 1.0);
        if (t < best || (cluster > 0 && t == best)) {
            best = t;
            cluster = c;
        }
    }
    return cluster;
}

cudaError_t launch_attn_small(const TcMaps& maps, const TcGroup* g, int n_groups, const Plan& P, const AttnArgs& a,
                              int cluster, cudaStream_t st) {
    SmallParams p;
    memset(&p, 0, sizeof(p));
    p.H = P.H;
    p.B = P.B;
    p.N = P.N;
    p.scale_log2 = a.scale_log2;
    p.n_groups = n_groups;
    int items = 0;
    for (int i = 0; i < n_groups; ++i) {
        p.g[i] = g[i];
        p.item_base[i] = items;
        p.n_qt[i] = (g[i].q_end - g[i].q_begin + kBM - 1) / kBM;
        items += p.n_qt[i] * P.H * P.B;
    }
    p.out = (__nv_bfloat16*)a.out;
    p.lse = a.lse;
    p.status = a.status;
    p.wait_limit = kWaitLimit;
    const bool d128 = P.D == 128;
    const int smem = d128 ? SCfg<128>::kSmem : SCfg<64>::kSmem;
    const void* fn = d128 ? (const void*)mssa_small_kernel<128> : (const void*)mssa_small_kernel<64>;
    cudaError_t e = set_smem_attr(fn, smem, -1, kLaunchRegs);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(items * cluster));
    const dim3 cl((unsigned)cluster, 1, 1);
    return d128 ? launch_pdl_cluster(mssa_small_kernel<128>, grid, dim3(kThreads), smem, st, cl, maps, p, cluster)
                : launch_pdl_cluster(mssa_small_kernel<64>, grid, dim3(kThreads), smem, st, cl, maps, p, cluster);
}

}  // namespace msf
