// fp32 GEMM C[m, n] = sum_k A[m, k] B[n, k] on the sm_103a tensor cores, for
// the patch embedding and de-embedding of fp32 plans.
//
// Operands become three bf16 planes and a product six plane products, as in
// the fp32 attention (attn_f32_tc.cu); here the split happens on the way into
// shared memory, and the five small products have an accumulator of their own,
// so that rounding at full size happens only in the four hh steps of each
// 64-wide K chunk. A 128 x BN tile's K chunks are split over a thread-block
// cluster; the CTAs' sums meet in distributed shared memory in a fixed order.
// A CTA that reads operands that the planes cannot hold (f32_range.h) redoes its
// share with fp32 FMAs.
//
// Bound: at K = 64 (the fine tier) the fp32 output's writes, at the
// de-embedding's K = E latency, with the split's integer and FMA work (about
// eight instructions per element) beside the MMAs: 256 threads load a chunk's
// fp32 rows while the chunk before is multiplied, and two CTAs share an SM.
// 480p layer: the five embeddings 149 -> 31 us, the head's de-embedding
// 251 -> 10.4 us against the CUDA-core kernel (64 x 64 tiles, one launch a state).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <string.h>

#include "f32_range.cuh"
#include "gemm_f32_tc.h"
#include "ptx.cuh"

namespace msf {
namespace {

constexpr int kThreads = 256;
constexpr int kBM = 128;
constexpr int kPlane = 128 * 128;  // bytes of one plane chunk: 128 rows x 64 bf16, swizzled
constexpr int kMaxSplits = 8;
constexpr long long kWaitLimit = 2000000000LL;

struct F32Problem {
    const float* A;
    const float* B;
    float* C;
    int M, N, K;
    long long lda, ldb, ldc, a_bstride, c_bstride;
    int tile_base, m_tiles;
};
struct F32GemmParams {
    F32Problem g[kMaxGemmF32];
    int n, splits;
    unsigned int* status;
    // scatter into the latent (P > 0)
    int P, gw, Wl;
    long long plane;  // Hl * Wl
};

template <int BN>
struct GCfg {
    static constexpr int kB = BN * 128;  // bytes of one plane chunk of B
    static constexpr int kStage = 3 * (kPlane + kB);
    static constexpr int kRow = BN + 4;  // floats of a staged row (the padding spreads the banks)
    static constexpr int kPart = kBM * kRow * 4;
    static constexpr int kSmem = (kStage > kPart ? kStage : kPart) + 1024;
};

// Byte offset of elements (row, k..k+3) of a plane chunk in the 128-byte swizzle.
__device__ __forceinline__ uint32_t swz4(int row, int k) {
    return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((((k >> 3) ^ (row & 7)) << 4) | ((k & 4) << 1)));
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 2) gemm_f32_kernel(const __grid_constant__ F32GemmParams p) {
    using C = GCfg<BN>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sA = smem;               // [3] planes h, m, l
    unsigned char* sB = smem + 3 * kPlane;  // [3]
    float* part = reinterpret_cast<float*>(smem);
    __shared__ uint64_t mma_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int tile = (int)blockIdx.x, split = (int)blockIdx.y, b = blockIdx.z;
    int gi = 0;
    while (gi + 1 < p.n && tile >= p.g[gi + 1].tile_base) ++gi;
    const F32Problem& g = p.g[gi];
    const int m0 = (tile - g.tile_base) % g.m_tiles * kBM, n0 = (tile - g.tile_base) / g.m_tiles * BN;
    const int chunks = (g.K + 63) / 64;
    const int c0 = split * chunks / p.splits, c1 = (split + 1) * chunks / p.splits;

    if (tid == 0) {
        abort_flag = 0;
        ptx::mbar_init(&mma_bar, 1);
        ptx::fence_mbar_init();
    }
    if (warp == 0) {
        ptx::tmem_alloc(&tmem_base_sh, 2 * BN);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tbase = tmem_base_sh;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();

    // Sixteen threads per 64-wide row chunk, four columns each: rows tid / 16 + 16 i.
    constexpr int RA = kBM / 16, RB = BN / 16;
    const int k4 = 4 * (tid % 16), r0 = tid / 16;
    const float* A = g.A + b * g.a_bstride;
    float4 xa[RA], xb[RB];
    auto load = [&](int c) {
        const int k = 64 * c + k4;
#pragma unroll
        for (int i = 0; i < RA; ++i) {
            const int m = m0 + r0 + 16 * i;
            xa[i] = m < g.M && k < g.K ? __ldg(reinterpret_cast<const float4*>(A + m * g.lda + k))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int n = n0 + r0 + 16 * i;
            xb[i] = n < g.N && k < g.K ? __ldg(reinterpret_cast<const float4*>(g.B + n * g.ldb + k))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    bool ok = true;
    uint32_t code_a = 0, code_b = 0;
    auto put = [&](unsigned char* dst, int plane_bytes, int row, const float4& x, uint32_t& code) {
        uint2 h, m, l;
        ptx::split_bf16(x.x, x.y, h.x, m.x, l.x);
        ptx::split_bf16(x.z, x.w, h.y, m.y, l.y);
        code = max(code, range_code(abs_bits4(x)));
        const uint32_t o = swz4(row, k4);
        *reinterpret_cast<uint2*>(dst + o) = h;
        *reinterpret_cast<uint2*>(dst + plane_bytes + o) = m;
        *reinterpret_cast<uint2*>(dst + 2 * plane_bytes + o) = l;
    };
    if (c0 < c1) load(c0);
    for (int c = c0; c < c1; ++c) {
        // the chunk before has been multiplied: its space is free
        if (c > c0) ok = ok && ptx::mbar_wait_bounded(&mma_bar, (uint32_t)((c - c0 - 1) & 1), &abort_flag, kWaitLimit);
#pragma unroll
        for (int i = 0; i < RA; ++i) put(sA, kPlane, r0 + 16 * i, xa[i], code_a);
#pragma unroll
        for (int i = 0; i < RB; ++i) put(sB, C::kB, r0 + 16 * i, xb[i], code_b);
        ptx::fence_proxy_async_smem();
        __syncthreads();
        if (warp == 0) {
            ptx::tc_fence_after();
            if (ptx::elect_one_sync()) {
                constexpr uint32_t idesc = ptx::idesc_bf16(kBM, BN, false, false);
                const uint64_t ad = ptx::sdesc_sw128(ptx::smem_u32(sA), 16, 1024);
                const uint64_t bd = ptx::sdesc_sw128(ptx::smem_u32(sB), 16, 1024);
                const bool first = c == c0;
                // hl, mm, lh, hm, mh into the small accumulator, hh into its own
                const int pa[6] = {0, 1, 2, 0, 1, 0}, pb[6] = {2, 1, 0, 1, 0, 0};
#pragma unroll
                for (int x = 0; x < 6; ++x)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        ptx::mma_ss(tbase + (x < 5 ? BN : 0), ad + (uint64_t)((pa[x] * kPlane) >> 4) + (uint64_t)(2 * kk),
                                    bd + (uint64_t)((pb[x] * C::kB) >> 4) + (uint64_t)(2 * kk), idesc,
                                    (first && kk == 0 && (x == 0 || x == 5)) ? 0u : 1u);
                ptx::mma_commit(&mma_bar);
            }
            __syncwarp();
        }
        if (c + 1 < c1) load(c + 1);
    }
    if (c0 < c1) ok = ok && ptx::mbar_wait_bounded(&mma_bar, (uint32_t)((c1 - c0 - 1) & 1), &abort_flag, kWaitLimit);
    if (!ok && lane == 0) atomicOr(p.status, kDevTimeout);
    const uint32_t codes = block_codes(code_a | code_b << 8);
    const bool redo = !range_holds_gemm(codes & 255u, codes >> 8);
    ptx::tc_fence_after();
    // ---- this CTA's share of the sums into shared memory
    if (redo) {
        for (int e = tid; e < kBM * BN; e += kThreads) {
            const int m = m0 + e / BN, n = n0 + e % BN;
            float acc = 0.f;
            if (m < g.M && n < g.N)
                for (int k = 64 * c0; k < min(64 * c1, g.K); ++k)
                    acc = fmaf(__ldg(A + m * g.lda + k), __ldg(g.B + n * g.ldb + k), acc);
            part[(e / BN) * C::kRow + e % BN] = acc;
        }
    } else {
        const int half = warp / 4, row = (warp % 4) * 32 + lane;
        const uint32_t t = tbase + ((uint32_t)((warp % 4) * 32) << 16) + half * (BN / 2);
#pragma unroll
        for (int c = 0; c < BN / 64; ++c) {
            uint32_t hh[32], lo[32];
            if (c0 < c1) {
                ptx::tmem_ld32(t + 32 * c, hh);
                ptx::tmem_ld32(t + BN + 32 * c, lo);
                ptx::tmem_wait_ld();
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) hh[e] = lo[e] = 0u;
            }
            float4* d = reinterpret_cast<float4*>(part + row * C::kRow + half * (BN / 2) + 32 * c);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                d[e] = make_float4(__uint_as_float(hh[4 * e]) + __uint_as_float(lo[4 * e]),
                                   __uint_as_float(hh[4 * e + 1]) + __uint_as_float(lo[4 * e + 1]),
                                   __uint_as_float(hh[4 * e + 2]) + __uint_as_float(lo[4 * e + 2]),
                                   __uint_as_float(hh[4 * e + 3]) + __uint_as_float(lo[4 * e + 3]));
        }
    }
    ptx::tc_fence_before();
    ptx::cluster_sync();
    // ---- rows [split * R, split * R + R) of the tile, summed in split order
    const int R = kBM / p.splits;
    auto sum4 = [&](const float* src) {
        if (p.splits == 1) return *reinterpret_cast<const float4*>(src);
        float4 v[kMaxSplits];
#pragma unroll
        for (int s = 0; s < kMaxSplits; ++s)
            if (s < p.splits) v[s] = ptx::ld_cluster_f4(src, (uint32_t)s);
        float4 a = v[0];
#pragma unroll
        for (int s = 1; s < kMaxSplits; ++s)
            if (s < p.splits) {
                a.x += v[s].x;
                a.y += v[s].y;
                a.z += v[s].z;
                a.w += v[s].w;
            }
        return a;
    };
    // Four features of a token from n on, into the latent from its first pixel.
    const int P = p.P, PP = P * P;
    auto scatter = [&](float* lat, int n, const float4& a) {
        auto at = [&](int f) { return lat + (f / PP) * p.plane + (long long)(f % PP / P) * p.Wl + f % P; };
        if (P % 4 == 0) {
            *reinterpret_cast<float4*>(at(n)) = a;
        } else if (P % 2 == 0) {
            *reinterpret_cast<float2*>(at(n)) = make_float2(a.x, a.y);
            *reinterpret_cast<float2*>(at(n + 2)) = make_float2(a.z, a.w);
        } else {
            *at(n) = a.x;
            *at(n + 1) = a.y;
            *at(n + 2) = a.z;
            *at(n + 3) = a.w;
        }
    };
    auto pixel = [&](int m) {
        return g.C + b * g.c_bstride + (long long)(P * (m / p.gw)) * p.Wl + (long long)P * (m % p.gw);
    };
    if (P == 0 || p.splits > 2) {
        for (int x = tid; x < R * (BN / 4); x += kThreads) {
            const int row = split * R + x / (BN / 4), n = n0 + 4 * (x % (BN / 4)), m = m0 + row;
            if (m >= g.M || n >= g.N) continue;
            const float4 a = sum4(part + row * C::kRow + n - n0);
            if (P == 0)
                *reinterpret_cast<float4*>(g.C + b * g.c_bstride + m * g.ldc + n) = a;
            else
                scatter(pixel(m), n, a);
        }
    } else if (m0 + split * R + tid % R < g.M) {
        // The sums of one or two CTAs into the latent, a token per thread: neighbouring
        // tokens' pixels of a feature run lie side by side there, while a row's features
        // go to a line each (one chunk, 96 tokens of patch edge 4: 17.2 us and 7.3).
        // From four CTAs on the loads of the others' shared memory, a row's features in
        // a run, weigh more (144 tokens, 8 chunks: 8.5 us as above, 9.6 this way).
        const int row = split * R + tid % R;
        float* lat = pixel(m0 + row);
        for (int c = 4 * (tid / R); c < BN && n0 + c < g.N; c += 4 * (kThreads / R))
            scatter(lat, n0 + c, sum4(part + row * C::kRow + c));
    }
    // No CTA leaves while another may still read its shared memory.
    ptx::cluster_sync();
    if (warp == 0) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tbase, 2 * BN);
    }
}

}  // namespace

bool gemm_f32_tc_supported(const GemmArgs& g) {
    return g.M > 0 && g.N > 0 && g.K > 0 && g.K % 4 == 0 && g.N % 4 == 0 && g.lda % 4 == 0 && g.ldb % 4 == 0 &&
           g.ldc % 4 == 0 && g.a_bstride % 4 == 0 && g.c_bstride % 4 == 0 &&
           (((uintptr_t)g.A | (uintptr_t)g.B | (uintptr_t)g.C) & 15) == 0;
}

cudaError_t launch_gemm_f32_tc(const GemmArgs* a, int n, int batch, unsigned int* status, cudaStream_t st,
                               const MspShape* scatter, int P) {
    F32GemmParams p;
    memset(&p, 0, sizeof(p));
    int widest = 0, deepest = 0;
    for (int i = 0; i < n; ++i) {
        widest = a[i].N > widest ? a[i].N : widest;
        deepest = a[i].K > deepest ? a[i].K : deepest;
    }
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const int chunks = (deepest + 63) / 64;
    // Tiles of 64 columns where those of 128 would leave SMs idle and have little to
    // multiply (36 tokens, K = 64, N = 256: 10.5 -> 7.2 us).
    long long wide = 0;
    for (int i = 0; i < n; ++i) wide += (long long)((a[i].M + kBM - 1) / kBM) * ((a[i].N + 127) / 128) * batch;
    const int bn = widest <= 64 || (chunks <= 2 && wide <= sms) ? 64 : 128;
    int tiles = 0;
    for (int i = 0; i < n; ++i) {
        F32Problem& g = p.g[i];
        g = {(const float*)a[i].A, (const float*)a[i].B, (float*)a[i].C, a[i].M, a[i].N, a[i].K,
             a[i].lda, a[i].ldb, a[i].ldc, a[i].a_bstride, a[i].c_bstride, tiles, (a[i].M + kBM - 1) / kBM};
        tiles += g.m_tiles * ((a[i].N + bn - 1) / bn);
    }
    p.n = n;
    p.status = status;
    if (scatter) {
        p.P = P;
        p.gw = scatter->Wl / P;
        p.Wl = scatter->Wl;
        p.plane = (long long)scatter->Hl * scatter->Wl;
    }
    // At most eight chunks (32 steps at full size) per CTA where the cluster
    // allows it, and more CTAs while the tiles leave half of the SMs idle.
    int s = 1;
    while (s < kMaxSplits && (chunks > 8 * s || ((long long)tiles * batch * s < sms && chunks >= 4 * s))) s *= 2;
    p.splits = s;
    const void* fn = bn == 64 ? (const void*)gemm_f32_kernel<64> : (const void*)gemm_f32_kernel<128>;
    const int smem = bn == 64 ? GCfg<64>::kSmem : GCfg<128>::kSmem;
    e = set_smem_attr(fn, smem, 100);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)tiles, (unsigned)s, (unsigned)batch);
    return bn == 64 ? launch_pdl_cluster(gemm_f32_kernel<64>, grid, dim3(kThreads), smem, st, dim3(1, s, 1), p)
                    : launch_pdl_cluster(gemm_f32_kernel<128>, grid, dim3(kThreads), smem, st, dim3(1, s, 1), p);
}

}  // namespace msf
