// Fused Multi-Scale Patchification kernels on the sm_103a tensor cores
// (Sec. 3.2: a latent state of scale s_l is cut into patches of edge
// P = patch * s_l; Eq. 3 token counts; feature order (c, dy, dx)).
//
// msp_embed_kernel    patchify + tier embedding in one pass. The A operand
//                     (raw patch vectors, K = C*P^2) is gathered from the
//                     latent straight into 128-byte-swizzled shared memory by
//                     four warps, B (the tier's [E, K] weight) arrives by TMA,
//                     and the accumulator is written once as bf16 tokens.
//
// msp_deembed_kernel  de-embedding + unpatchify of one window position,
//                     split-K over a thread-block cluster and reduced over
//                     distributed shared memory (see its section below).
//
// Roles (256 threads): warp 0 TMA producer, warp 1 MMA issuer (one elected
// lane of the converged warp), warp 2 TMEM allocation, warps 4-7 gather and
// epilogue. Every wait is bounded and winds down through the status word.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <string.h>

#include "gemm_tc.h"
#include "kernels.h"
#include "msp_tc.h"
#include "pool.cuh"
#include "ptx.cuh"
#include "sched.h"

namespace msf {

namespace {

constexpr int kThreads = 256;
constexpr long long kWaitLimit = 2000000000LL;
constexpr int kChunkA = 128 * 128;  // 128 rows x 64 bf16 (one K chunk), swizzled
constexpr int kEmbedBN = 256;
constexpr int kLoraBN = 192;  // columns of a tile with an adapter: 64 of the 256 hold the codes
constexpr int kEmbedStages = 2;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encoder() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)ptr;
    }
    return fn;
}

bool encode_2d(CUtensorMap* m, const void* base, int inner, int outer, long long stride_bytes,
               int box_inner, int box_outer) {
    EncodeTiledFn enc = encoder();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    cuuint64_t strides[1] = {(cuuint64_t)stride_bytes};
    cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_outer};
    cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Byte offset of bf16 element (row, k) inside one 128-row x 64-column K chunk
// in the 128-byte swizzle layout the tensor core and TMA use: rows are 128
// bytes, eight rows form a 1024-byte atom, and the 16-byte unit index is
// XOR-ed with the row's position in its atom.
__device__ __forceinline__ uint32_t swz_offset(int row, int k) {
    const int byte = k * 2;
    return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + (((byte >> 4) ^ (row & 7)) << 4) + (byte & 15));
}

// ----------------------------------------------------------------- embedding

// Features [64 kc, 64 kc + 64) of one token row in (c, dy, dx) order: 64 / P
// runs of P pixels, each run one row segment of one channel. The loads and the
// stores are apart, so a row's next chunk can be in flight while the current
// one waits for its stage.
template <int P, typename V>
__device__ __forceinline__ void load_chunk(V (&v)[64 / P], const __nv_bfloat16* base, size_t plane, int Wl,
                                           int kc, bool valid) {
#pragma unroll
    for (int g = 0; g < 64 / P; ++g) {
        const int f0 = kc * 64 + g * P;
        const int c = f0 / (P * P), dy = (f0 % (P * P)) / P;
        if (valid)
            v[g] = __ldg(reinterpret_cast<const V*>(base + c * plane + (size_t)dy * Wl));
        else
            memset(&v[g], 0, sizeof(V));
    }
}
template <int P, typename V>
__device__ __forceinline__ void store_chunk(unsigned char* dst, const V (&v)[64 / P], int r) {
#pragma unroll
    for (int g = 0; g < 64 / P; ++g) *reinterpret_cast<V*>(dst + swz_offset(r, g * P)) = v[g];
}

// Every K chunk of one token row into the A ring, each chunk's loads issued
// before the wait for the previous chunk's stage, so that the L2 round trips
// of consecutive chunks overlap. Returns false if a wait gave up.
template <int P, typename V>
__device__ __forceinline__ bool gather_row(unsigned char* sA, uint64_t* a_full, uint64_t* a_empty,
                                           const __nv_bfloat16* base, size_t plane, int Wl, int r, int nk,
                                           bool valid, volatile int* abort_p) {
    V cur[64 / P], nxt[64 / P];
    load_chunk<P, V>(cur, base, plane, Wl, 0, valid);
    for (int kc = 0; kc < nk; ++kc) {
        if (kc + 1 < nk) load_chunk<P, V>(nxt, base, plane, Wl, kc + 1, valid);
        const int st = kc % kEmbedStages;
        const uint32_t ph = (uint32_t)((kc / kEmbedStages) & 1);
        const bool ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&a_empty[st], ph ^ 1u, abort_p, kWaitLimit));
        if (!ok) return false;
        store_chunk<P, V>(sA + st * kChunkA, cur, r);
        ptx::fence_proxy_async_smem();  // the tensor core reads through the async proxy
        ptx::mbar_arrive(&a_full[st]);
#pragma unroll
        for (int g = 0; g < 64 / P; ++g) cur[g] = nxt[g];
    }
    return true;
}

struct EmbedRun {
    int tile_base;  // first CTA of this run in blockIdx.x
    int m_tiles;
    int M;          // tokens of the run (per stream)
    int l0;         // first state of the run
    int n_l;        // tokens per state
    int gw;         // tokens per grid row (Wl / P)
    int P;          // patch edge in latent pixels
    int K;          // C * P * P
    int tok_off;    // first token row of the run in the output
    int lora;       // 1: one more K chunk (LoRA codes x up projection), 192-column tiles
    float scale;    // LoRA scale
    int pool_base;  // first pyramid task of this run's tiles, and tasks of each
    int pool_per;   // thread of their two idle warps (0: none)
};
struct EmbedParams {
    int n_runs;
    EmbedRun run[kMaxGemmProblems];
    int T, C, Hl, Wl, E;
    int n_embed_tiles;  // CTAs [0, n_embed_tiles) of a stream embed; the rest pool
    int pool_ctas;      // CTAs per stream that run the pyramid jobs (0: none)
    int pool_tasks;     // vector-pair tasks per pyramid job
    int pool_first;     // first task of those CTAs (the tiles' idle warps run the others)
    const __nv_bfloat16* latent;  // [B, T, C, Hl, Wl]
    __nv_bfloat16* tokens;        // [B, N, E]
    long long tok_bstride;        // elements
    unsigned int* status;
};
struct EmbedMaps {
    CUtensorMap w[kMaxGemmProblems];    // [E, K] weight of each run: dims {K, E}
    CUtensorMap out[kMaxGemmProblems];  // the run's tokens: dims {E, M, B}, rows past M clipped
};
struct LoraMaps {
    CUtensorMap down[kMaxGemmProblems];  // LoRA down projection [r, K]: dims {K, r}
    CUtensorMap up[kMaxGemmProblems];    // LoRA up projection [E, r]: dims {r, E}
};
struct NoLora {};

// 128 tokens x 256 embedding columns per CTA (one N=256 MMA per K step, half
// the gathers of 128-column tiles); two CTAs per SM (97 KB of shared memory
// each), so the 480p window's 210 tiles run in one wave on 152 SMs.
//
// kLora (its own instantiation, with the adapters' maps): a run with an adapter
// has 192-column tiles; each K chunk is also multiplied by the down projection
// into the 64 accumulator columns left, the gathering warps round those codes
// (scaled, once) into one more A chunk, and the last K chunk is codes x up
// projection. Every column tile of a token tile computes the codes again, which
// costs a 64-wide MMA per K step; a launch of their own cost 4.8 us (480p).
//
// kShare (its own instantiation): the tiles' idle warps pool. Compiled into the
// plain kernel, that code alone made an attention behind a launch without
// pyramid jobs end 1.5 us later (117.8 -> 119.3 us).
template <bool kLora, bool kShare, class Lora>
__global__ void __launch_bounds__(kThreads, 2)
    msp_embed_kernel(const __grid_constant__ EmbedMaps maps, const __grid_constant__ EmbedParams p,
                     const __grid_constant__ PoolBatch pool, const __grid_constant__ Lora lmaps) {
    if (!kLora && (int)blockIdx.x >= p.n_embed_tiles) {
        // ---- K/V pyramid jobs in the CTAs after the embedding tiles (the
        // longest tiles, those of the runs with the most K chunks, come
        // first): the same per-thread pooling as pool_kernel, one task per
        // thread. The two parts read and write disjoint buffers; the block
        // scheduler starts these CTAs in the slots the embedding leaves free
        // and, as its short tiles finish, in theirs.
        ptx::grid_dep_wait();
        ptx::grid_dep_launch();
        const int stride = p.pool_ctas * kThreads;
        const int total = pool.n * p.pool_tasks;
        for (int t = p.pool_first + ((int)blockIdx.x - p.n_embed_tiles) * kThreads + (int)threadIdx.x; t < total;
             t += stride)
            pool_task<__nv_bfloat16>(pool, t / p.pool_tasks, blockIdx.z, t % p.pool_tasks);
        return;
    }
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sA = smem;                                   // [stage][chunk]
    unsigned char* sB = smem + kEmbedStages * kChunkA;          // [stage][BN rows x 128 B]
    constexpr int kBBytes = kEmbedBN * 128;
    __shared__ uint64_t a_full[kEmbedStages], a_empty[kEmbedStages];
    __shared__ uint64_t b_full[kEmbedStages], b_empty[kEmbedStages], acc_full, codes_full;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int tile = (int)blockIdx.x;
    int ri = 0;
    while (ri < p.n_runs - 1 && tile >= p.run[ri + 1].tile_base) ++ri;
    const EmbedRun& R = p.run[ri];
    const int local = tile - R.tile_base;
    const int mt = local % R.m_tiles, nt = local / R.m_tiles;
    const int b = blockIdx.z;
    const int nk_patch = R.K / 64;      // chunks gathered from the latent
    const bool lora = kLora && R.lora;
    const int nk = nk_patch + (lora ? 1 : 0);   // plus the LoRA chunk
    const int bn = lora ? kLoraBN : kEmbedBN;   // output columns of this tile

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < kEmbedStages; ++s) {
            ptx::mbar_init(&a_full[s], 128);  // one arrival per gathering thread
            ptx::mbar_init(&a_empty[s], 1);
            ptx::mbar_init(&b_full[s], 1);
            ptx::mbar_init(&b_empty[s], 1);
        }
        ptx::mbar_init(&acc_full, 1);
        ptx::mbar_init(&codes_full, 1);
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&maps.w[ri]);
    }
    if (warp == 2) {
        ptx::tmem_alloc(&tmem_base_sh, kEmbedBN);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tbase = tmem_base_sh;
    volatile int* abort_p = &abort_flag;
    volatile int never = 0;
    ptx::grid_dep_wait();  // the latent and weights written before are visible
    ptx::grid_dep_launch();

    if (warp == 0) {
        if (lane == 0) {
            int issued = 0;
            bool ok = true;
            for (int kc = 0; kc < nk; ++kc) {
                const int st = kc % kEmbedStages;
                const uint32_t ph = (uint32_t)((kc / kEmbedStages) & 1);
                if (!ptx::mbar_wait_bounded(&b_empty[st], ph ^ 1u, abort_p, kWaitLimit)) {
                    ok = false;
                    break;
                }
                // a LoRA run's patch chunk: 192 rows of the weight, then the 64
                // (zero past the rank) of the down projection
                ptx::mbar_arrive_expect_tx(&b_full[st], lora && kc == nk_patch ? kLoraBN * 128 : kBBytes);
                if constexpr (kLora) {
                    if (kc == nk_patch)
                        ptx::tma_load_2d(sB + st * kBBytes, &lmaps.up[ri], &b_full[st], 0, nt * bn);
                    else
                        ptx::tma_load_2d(sB + st * kBBytes, &maps.w[ri], &b_full[st], kc * 64, nt * bn);
                    if (lora && kc < nk_patch)
                        ptx::tma_load_2d(sB + st * kBBytes + kLoraBN * 128, &lmaps.down[ri], &b_full[st], kc * 64, 0);
                } else {
                    ptx::tma_load_2d(sB + st * kBBytes, &maps.w[ri], &b_full[st], kc * 64, nt * bn);
                }
                ++issued;
            }
            if (!ok) {
                for (int kc = (issued > kEmbedStages ? issued - kEmbedStages : 0); kc < issued; ++kc)
                    ptx::mbar_wait_bounded(&b_full[kc % kEmbedStages],
                                           (uint32_t)((kc / kEmbedStages) & 1), &never, kWaitLimit);
                atomicOr(p.status, kDevTimeout);
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc =
            lora ? ptx::idesc_bf16(128, kLoraBN, false, false) : ptx::idesc_bf16(128, kEmbedBN, false, false);
        constexpr uint32_t id_codes = ptx::idesc_bf16(128, 64, false, false);
        const uint64_t a_desc = ptx::sdesc_sw128(ptx::smem_u32(sA), 16, 1024);
        const uint64_t b_desc = ptx::sdesc_sw128(ptx::smem_u32(sB), 16, 1024);
        bool ok = true;
        for (int kc = 0; kc < nk && ok; ++kc) {
            const int st = kc % kEmbedStages;
            const uint32_t ph = (uint32_t)((kc / kEmbedStages) & 1);
            const bool ra = ptx::mbar_wait_bounded(&a_full[st], ph, abort_p, kWaitLimit);
            const bool rb = ra && ptx::mbar_wait_bounded(&b_full[st], ph, abort_p, kWaitLimit);
            ok = __all_sync(0xffffffffu, rb);
            if (!ok) break;
            ptx::tc_fence_after();
            if (ptx::elect_one_sync()) {
                const uint64_t ad = a_desc + (uint64_t)(st * (kChunkA >> 4));
                const uint64_t bd = b_desc + (uint64_t)(st * (kBBytes >> 4));
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    ptx::mma_ss(tbase, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc,
                                (kc > 0 || kk > 0) ? 1u : 0u);
                if (lora && kc < nk_patch) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        ptx::mma_ss(tbase + kLoraBN, ad + (uint64_t)(kk * 2),
                                    bd + (uint64_t)((kLoraBN * 128) >> 4) + (uint64_t)(kk * 2), id_codes,
                                    (kc > 0 || kk > 0) ? 1u : 0u);
                    if (kc + 1 == nk_patch) ptx::mma_commit(&codes_full);
                }
                ptx::mma_commit(&a_empty[st]);
                ptx::mma_commit(&b_empty[st]);
            }
            __syncwarp();
        }
        if (ptx::elect_one_sync()) ptx::mma_commit(&acc_full);  // also after an abort: drains the MMAs
        __syncwarp();
        if (!ok && lane == 0) atomicOr(p.status, kDevTimeout);
    } else if (warp < 4) {
        // ---- warps 2 and 3: this tile's share of the pyramid jobs
        if constexpr (kShare) {
            const int total = pool.n * p.pool_tasks;
            int t = R.pool_base + local * 64 * R.pool_per + (int)threadIdx.x - 64;
            for (int k = 0; k < R.pool_per && t < total; ++k, t += 64)
                pool_task<__nv_bfloat16>(pool, t / p.pool_tasks, blockIdx.z, t % p.pool_tasks);
        }
    } else {
        // ---- gather: one token row per thread
        const int r = (warp - 4) * 32 + lane;
        const int m = mt * 128 + r;
        const bool valid = m < R.M;
        const int P = R.P;
        const __nv_bfloat16* base = p.latent;
        if (valid) {
            const int l = R.l0 + m / R.n_l;
            const int loc = m % R.n_l;
            const int i = loc / R.gw, jj = loc % R.gw;
            base = p.latent + ((size_t)b * p.T + l) * p.C * p.Hl * p.Wl + (size_t)(P * i) * p.Wl + P * jj;
        }
        const size_t plane = (size_t)p.Hl * p.Wl;
        bool ok = true;
        if (P == 2) {
            ok = gather_row<2, uint32_t>(sA, a_full, a_empty, base, plane, p.Wl, r, nk_patch, valid, abort_p);
        } else if (P == 4) {
            ok = gather_row<4, uint2>(sA, a_full, a_empty, base, plane, p.Wl, r, nk_patch, valid, abort_p);
        } else if (P == 8) {
            ok = gather_row<8, uint4>(sA, a_full, a_empty, base, plane, p.Wl, r, nk_patch, valid, abort_p);
        } else for (int kc = 0; kc < nk_patch; ++kc) {
            const int st = kc % kEmbedStages;
            const uint32_t ph = (uint32_t)((kc / kEmbedStages) & 1);
            ok = ptx::mbar_wait_bounded(&a_empty[st], ph ^ 1u, abort_p, kWaitLimit);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            unsigned char* dst = sA + st * kChunkA;
            {
                for (int g = 0; g < 64 / P; ++g) {
                    const int f0 = kc * 64 + g * P;
                    const int c = f0 / (P * P), dy = (f0 % (P * P)) / P;
                    const __nv_bfloat16* src = base + c * plane + (size_t)dy * p.Wl;
                    for (int x = 0; x < P; ++x)
                        *reinterpret_cast<__nv_bfloat16*>(dst + swz_offset(r, g * P + x)) =
                            valid ? src[x] : __float2bfloat16(0.f);
                }
            }
            ptx::fence_proxy_async_smem();  // the tensor core reads through the async proxy
            ptx::mbar_arrive(&a_full[st]);
        }
        if (ok && lora) {
            // ---- LoRA chunk: this row's codes, scaled and rounded once
            const int st = nk_patch % kEmbedStages;
            const uint32_t ph = (uint32_t)((nk_patch / kEmbedStages) & 1);
            ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&codes_full, 0, abort_p, kWaitLimit) &&
                                             ptx::mbar_wait_bounded(&a_empty[st], ph ^ 1u, abort_p, kWaitLimit));
            if (ok) {
                ptx::tc_fence_after();
                const uint32_t taddr = tbase + kLoraBN + ((uint32_t)((warp - 4) * 32) << 16);
                unsigned char* dst = sA + st * kChunkA;
                const float sc = R.scale;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t v[32];
                    ptx::tmem_ld32(taddr + 32 * c, v);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        *reinterpret_cast<uint4*>(dst + swz_offset(r, 32 * c + 8 * e)) = make_uint4(
                            ptx::pack_bf16(sc * __uint_as_float(v[8 * e]), sc * __uint_as_float(v[8 * e + 1])),
                            ptx::pack_bf16(sc * __uint_as_float(v[8 * e + 2]), sc * __uint_as_float(v[8 * e + 3])),
                            ptx::pack_bf16(sc * __uint_as_float(v[8 * e + 4]), sc * __uint_as_float(v[8 * e + 5])),
                            ptx::pack_bf16(sc * __uint_as_float(v[8 * e + 6]), sc * __uint_as_float(v[8 * e + 7])));
                }
                ptx::tc_fence_before();
                ptx::fence_proxy_async_smem();
                ptx::mbar_arrive(&a_full[st]);
            }
        }
        // ---- epilogue: bf16 tile staged in the (now idle) A and B stages in
        // the 128-byte swizzle layout, then TMA stores of 128 rows x 64 columns.
        ok = ok && ptx::mbar_wait_bounded(&acc_full, 0, abort_p, kWaitLimit);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            ptx::tc_fence_after();
            const uint32_t taddr = tbase + ((uint32_t)((warp - 4) * 32) << 16);
#pragma unroll 1
            for (int c = 0; c < bn / 32; ++c) {
                uint32_t v[32];
                ptx::tmem_ld32(taddr + c * 32, v);
                ptx::tmem_wait_ld();
                unsigned char* stage = sA + (c / 2) * kChunkA;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    *reinterpret_cast<uint4*>(stage + swz_offset(r, (c % 2) * 32 + 8 * e)) =
                        make_uint4(ptx::pack_bf16(__uint_as_float(v[8 * e]), __uint_as_float(v[8 * e + 1])),
                                   ptx::pack_bf16(__uint_as_float(v[8 * e + 2]), __uint_as_float(v[8 * e + 3])),
                                   ptx::pack_bf16(__uint_as_float(v[8 * e + 4]), __uint_as_float(v[8 * e + 5])),
                                   ptx::pack_bf16(__uint_as_float(v[8 * e + 6]), __uint_as_float(v[8 * e + 7])));
            }
            ptx::fence_proxy_async_smem();
        }
        // The four epilogue warps meet before one thread stores the tile.
        ok = ptx::named_bar_and(1, 128, ok);
        if (ok && warp == 4 && lane == 0) {
            for (int h = 0; h < bn / 64 && nt * bn + h * 64 < p.E; ++h)
                ptx::tma_store_3d(&maps.out[ri], sA + h * kChunkA, nt * bn + h * 64, mt * 128, b);
            ptx::bulk_commit();
            ptx::bulk_wait_read_all();
        }
        if (!ok && lane == 0) atomicOr(p.status, kDevTimeout);
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tbase, kEmbedBN);
    }
}


// ------------------------------------------------------------ de-embedding
//
// msp_deembed_kernel: de-embedding + unpatchify of one window position. The
// K = E contraction is split over the S CTAs of a thread-block cluster
// (S <= 8 divides 128). Each CTA leaves its fp32 partial 128 x 64 tile in its
// own shared memory; after a cluster barrier CTA r sums rows [r*128/S,
// (r+1)*128/S) of all S partials in split order over distributed shared
// memory, rounds once to bf16 and scatters them into the latent layout
// [B, C, Hl, Wl]. No partial sums go through global memory and no second
// kernel is needed.

constexpr int kDeBN = 64;
constexpr int kDeStages = 4;
constexpr int kDeTierStages = 3;
constexpr int kDeMaxSplits = 8;  // cluster size along the split (portable limit)
constexpr int kDePartStride = kDeBN + 4;  // floats per staged row (padding spreads the banks)

struct DeembedParams {
    int M;              // tokens of the position (per stream)
    int K;              // embedding width E
    int nk_all;         // K chunks: E / 64 token chunks, then the latent residual's
    int m_tiles;
    int splits;         // cluster size along y
    int P, gw, C, Hl, Wl;
    int tok_row0;       // first token row of the position
    __nv_bfloat16* latent;  // [B, C, Hl, Wl]
    unsigned int* status;
};
// The tier's extras of one position.
struct DeembedTierParams {
    int rank;                     // of the adapter, 0: none
    float scale;                  // LoRA scale
    const __nv_bfloat16* up;      // LoRA up projection [F, rank]
    const __nv_bfloat16* latent;  // the position's input latent of stream 0 (residual)
    long long latent_bstride;     // elements
};
struct NoTier {};
struct DeembedMaps {
    CUtensorMap a;     // tokens {E, rows, B}
    CUtensorMap b;     // W_out {E, F}
    CUtensorMap down;  // LoRA down projection [r, E]: {E, r}
    CUtensorMap res;   // latent residual [F, F]: {F, F}
};

// One token row of the residual's K chunks c0, c0 + step, ... (n of them) into
// the ring as chunk uses k0, k0 + 1, ...: each chunk's loads go out before the
// wait for its stage (`go`: the producer, which follows every use of a stage,
// says that it is free). Returns false if a wait gave up.
template <int P, typename V, int kStages>
__device__ __forceinline__ bool gather_residual(unsigned char* ring, int stage_bytes, uint64_t* a_full, uint64_t* go,
                                                const __nv_bfloat16* base, size_t plane, int Wl, int r, int c0, int step,
                                                int n, int k0, bool valid, volatile int* abort_p) {
    V cur[64 / P];
    for (int i = 0; i < n; ++i) {
        load_chunk<P, V>(cur, base, plane, Wl, c0 + i * step, valid);
        const int st = (k0 + i) % kStages;
        if (!__all_sync(0xffffffffu, ptx::mbar_wait_bounded(&go[st], (uint32_t)((i / kStages) & 1), abort_p, kWaitLimit)))
            return false;
        store_chunk<P, V>(ring + st * stage_bytes, cur, r);
        ptx::fence_proxy_async_smem();
        ptx::mbar_arrive(&a_full[st]);
    }
    return true;
}

// kTier (its own instantiation): each token chunk is also multiplied by the
// LoRA down projection into a second accumulator, the residual's K chunks are
// gathered from the input latent, and the CTA that sums a row adds
// up x bf16(scale * codes) to it in fp32. (The codes, the raw patch vectors and
// the sum were three launches.)
template <bool kTier, class Tier>
__global__ void __launch_bounds__(kThreads, kTier ? 2 : 1)
    msp_deembed_kernel(const __grid_constant__ DeembedMaps maps, const __grid_constant__ DeembedParams p,
                       const __grid_constant__ Tier tier) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    constexpr int kBBytes = kDeBN * 128;
    constexpr int kStageBytes = kChunkA + (kTier ? 2 : 1) * kBBytes;  // tokens, W_out, down projection
    float* part = reinterpret_cast<float*>(smem);  // reuses the ring once every MMA is done
    float* cpart = part + 128 * kDePartStride;     // kTier: this split's codes
    // kTier: then the up projection of the tile's features transposed
    // [rank][kDePartStride], and the summed codes of this CTA's rows
    float* up_s = cpart + 128 * kDePartStride;
    float* code_s = up_s + 64 * kDePartStride;
    constexpr int kStages = kTier ? kDeTierStages : kDeStages;
    __shared__ uint64_t full[kStages], empty[kStages], go[kStages], a_full[kStages], acc_full;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int tile = blockIdx.x;
    const int mt = tile % p.m_tiles, nt = tile / p.m_tiles;
    const int split = (int)ptx::cluster_rank();
    const int b = blockIdx.z;
    const int nk_all = p.nk_all;
    const int nk_tok = p.K / 64;
    // Chunks of this split: a contiguous run, or (kTier) every splits-th one, so
    // that the gathered residual chunks, which come last, spread over the CTAs.
    const int step = kTier ? p.splits : 1;
    const int kc0 = kTier ? split : (int)((long long)split * nk_all / p.splits);
    const int nk = kTier ? (nk_all - split + step - 1) / step
                         : (int)((long long)(split + 1) * nk_all / p.splits) - kc0;
    const int n_tok = kTier ? min(max((nk_tok - split + step - 1) / step, 0), nk) : nk;  // token chunks, then residual
    bool lora = false;
    if constexpr (kTier) lora = tier.rank > 0;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < kStages; ++s) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&empty[s], 1);
            if constexpr (kTier) {
                ptx::mbar_init(&go[s], 1);
                ptx::mbar_init(&a_full[s], 128);  // residual chunks: one arrival per gathering thread
            }
        }
        ptx::mbar_init(&acc_full, 1);
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&maps.a);  // before the wait for the previous launch: 0.2 us behind an attention
        ptx::prefetch_tmap(&maps.b);
    }
    if (warp == 2) {
        ptx::tmem_alloc(&tmem_base_sh, kTier ? 2 * kDeBN : kDeBN);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tbase = tmem_base_sh;
    volatile int* abort_p = &abort_flag;
    volatile int never = 0;
    ptx::grid_dep_wait();  // the tokens written by the attention kernel are visible
    ptx::grid_dep_launch();

    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            int issued = 0;
            for (int kc = 0; kc < nk; ++kc) {
                const int st = kc % kStages;
                const uint32_t ph = (uint32_t)((kc / kStages) & 1);
                if (!ptx::mbar_wait_bounded(&empty[st], ph ^ 1u, abort_p, kWaitLimit)) {
                    ok = false;
                    break;
                }
                unsigned char* sa = smem + st * kStageBytes;
                const int g = kc0 + kc * step;
                if (!kTier || kc < n_tok) {
                    ptx::mbar_arrive_expect_tx(&full[st], kChunkA + (lora ? 2 : 1) * kBBytes);
                    ptx::tma_load_3d(sa, &maps.a, &full[st], g * 64, p.tok_row0 + mt * 128, b);
                    ptx::tma_load_2d(sa + kChunkA, &maps.b, &full[st], g * 64, nt * kDeBN);
                    if (lora) ptx::tma_load_2d(sa + kChunkA + kBBytes, &maps.down, &full[st], g * 64, 0);
                } else {
                    ptx::mbar_arrive(&go[st]);
                    ptx::mbar_arrive_expect_tx(&full[st], kBBytes);
                    ptx::tma_load_2d(sa + kChunkA, &maps.res, &full[st], (g - nk_tok) * 64, nt * kDeBN);
                }
                ++issued;
            }
            if (!ok) {
                for (int kc = (issued > kStages ? issued - kStages : 0); kc < issued; ++kc)
                    ptx::mbar_wait_bounded(&full[kc % kStages], (uint32_t)((kc / kStages) & 1), &never,
                                           kWaitLimit);
                atomicOr(p.status, kDevTimeout);
            }
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = ptx::idesc_bf16(128, kDeBN, false, false);
        const uint64_t desc0 = ptx::sdesc_sw128(ptx::smem_u32(smem), 16, 1024);
        for (int kc = 0; kc < nk && ok; ++kc) {
            const int st = kc % kStages;
            const uint32_t ph = (uint32_t)((kc / kStages) & 1);
            bool rf = ptx::mbar_wait_bounded(&full[st], ph, abort_p, kWaitLimit);
            if (kTier && kc >= n_tok)  // the residual's use of this stage, counted from its first chunk
                rf = rf && ptx::mbar_wait_bounded(&a_full[st], (uint32_t)(((kc - n_tok) / kStages) & 1), abort_p,
                                                  kWaitLimit);
            ok = __all_sync(0xffffffffu, rf);
            if (!ok) break;
            ptx::tc_fence_after();
            if (ptx::elect_one_sync()) {
                const uint64_t ad = desc0 + (uint64_t)(st * (kStageBytes >> 4));
                const uint64_t bd = ad + (uint64_t)(kChunkA >> 4);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    ptx::mma_ss(tbase, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc,
                                (kc > 0 || kk > 0) ? 1u : 0u);
                if (lora && kc < n_tok) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        ptx::mma_ss(tbase + kDeBN, ad + (uint64_t)(kk * 2),
                                    bd + (uint64_t)(kBBytes >> 4) + (uint64_t)(kk * 2), idesc,
                                    (kc > 0 || kk > 0) ? 1u : 0u);
                }
                ptx::mma_commit(&empty[st]);
            }
            __syncwarp();
        }
        if (ptx::elect_one_sync()) ptx::mma_commit(&acc_full);  // also after an abort: drains the MMAs
        __syncwarp();
        if (!ok && lane == 0) atomicOr(p.status, kDevTimeout);
    } else if (warp >= 4) {
        const int r = (warp - 4) * 32 + lane;
        if constexpr (kTier) {
            // ---- residual chunks: one token row of raw patch vectors per thread
            if (n_tok < nk) {
                const int m = mt * 128 + r;
                const bool valid = m < p.M;
                const __nv_bfloat16* base =
                    tier.latent + b * tier.latent_bstride +
                    (valid ? (size_t)(p.P * (m / p.gw)) * p.Wl + (size_t)p.P * (m % p.gw) : 0);
                const size_t plane = (size_t)p.Hl * p.Wl;
                const int c0 = kc0 + n_tok * step - nk_tok, n = nk - n_tok;
                if (p.P == 2)
                    ok = gather_residual<2, uint32_t, kStages>(smem, kStageBytes, a_full, go, base, plane, p.Wl, r, c0,
                                                               step, n, n_tok, valid, abort_p);
                else if (p.P == 4)
                    ok = gather_residual<4, uint2, kStages>(smem, kStageBytes, a_full, go, base, plane, p.Wl, r, c0,
                                                            step, n, n_tok, valid, abort_p);
                else if (p.P == 8)
                    ok = gather_residual<8, uint4, kStages>(smem, kStageBytes, a_full, go, base, plane, p.Wl, r, c0,
                                                            step, n, n_tok, valid, abort_p);
                else
                    for (int i = 0; i < n && ok; ++i) {  // any other patch edge, pixel by pixel
                        const int st = (n_tok + i) % kStages;
                        ok = __all_sync(0xffffffffu,
                                        ptx::mbar_wait_bounded(&go[st], (uint32_t)((i / kStages) & 1), abort_p, kWaitLimit));
                        if (!ok) break;
                        for (int x = 0; x < 64; ++x) {
                            const int f = (c0 + i * step) * 64 + x, PP = p.P * p.P;
                            *reinterpret_cast<__nv_bfloat16*>(smem + st * kStageBytes + swz_offset(r, x)) =
                                valid ? base[f / PP * plane + (size_t)(f % PP / p.P) * p.Wl + f % p.P]
                                      : __float2bfloat16(0.f);
                        }
                        ptx::fence_proxy_async_smem();
                        ptx::mbar_arrive(&a_full[st]);
                    }
            }
        }
        // ---- this split's partial tile into shared memory (row-major, padded rows)
        ok = ok && __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&acc_full, 0, abort_p, kWaitLimit));
        if (ok) {
            ptx::tc_fence_after();
            const uint32_t taddr = tbase + ((uint32_t)((warp - 4) * 32) << 16);
            auto stage = [&](uint32_t t, float* dst, bool any) {
                uint32_t vb[kDeBN / 32][32];
                if (any) {
#pragma unroll
                    for (int c = 0; c < kDeBN / 32; ++c) ptx::tmem_ld32(t + c * 32, vb[c]);
                    ptx::tmem_wait_ld();
                } else {
#pragma unroll
                    for (int c = 0; c < kDeBN / 32; ++c)
#pragma unroll
                        for (int e = 0; e < 32; ++e) vb[c][e] = 0u;
                }
#pragma unroll
                for (int c = 0; c < kDeBN / 32; ++c) {
                    const uint32_t* v = vb[c];
                    float4* d4 = reinterpret_cast<float4*>(dst + r * kDePartStride + c * 32);
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        d4[e] = make_float4(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1]),
                                            __uint_as_float(v[4 * e + 2]), __uint_as_float(v[4 * e + 3]));
                }
            };
            stage(taddr, part, true);
            if (lora) stage(taddr + kDeBN, cpart, n_tok > 0);
        } else if (lane == 0) {
            atomicOr(p.status, kDevTimeout);
        }
    } else if constexpr (kTier) {
        // ---- warps 2 and 3: the up projection's rows of the tile's 64
        // features, loaded early and put into the ring's space at its end
        if (lora) {
            const int f = (warp - 2) * 32 + lane;
            const uint4* src = reinterpret_cast<const uint4*>(tier.up + (size_t)(nt * kDeBN + f) * tier.rank);
            uint4 u[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) u[x] = 8 * x < tier.rank ? __ldg(src + x) : make_uint4(0u, 0u, 0u, 0u);
            if (ptx::mbar_wait_bounded(&acc_full, 0, abort_p, kWaitLimit)) {
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    const uint32_t w[4] = {u[x].x, u[x].y, u[x].z, u[x].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        up_s[(8 * x + 2 * e) * kDePartStride + f] = __uint_as_float(w[e] << 16);
                        up_s[(8 * x + 2 * e + 1) * kDePartStride + f] = __uint_as_float(w[e] & 0xffff0000u);
                    }
                }
            }
        }
    }
    // Every thread of every CTA of the cluster: partials are staged.
    __syncwarp();
    ptx::tc_fence_before();
    ptx::cluster_sync();
    const int R = 128 / p.splits;  // rows [split * R, split * R + R) of the tile are this CTA's
    // All splits' partials requested before the first add (remote
    // shared-memory loads are independent), summed in split order.
    auto sum4 = [&](const float* src) {
        float4 v[kDeMaxSplits];
#pragma unroll
        for (int sp = 0; sp < kDeMaxSplits; ++sp)
            v[sp] = sp < p.splits ? ptx::ld_cluster_f4(src, (uint32_t)sp) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int sp = 0; sp < kDeMaxSplits; ++sp) {
            acc.x += v[sp].x;
            acc.y += v[sp].y;
            acc.z += v[sp].z;
            acc.w += v[sp].w;
        }
        return acc;
    };
    const int per_row = kDeBN / 4;  // float4 per row
    if constexpr (kTier) {
        if (lora) {
            // the rows' codes: summed, scaled, rounded once to bf16
            for (int q = threadIdx.x; q < R * per_row; q += kThreads) {
                const int row = q / per_row, c4 = q % per_row;
                const float4 a = sum4(cpart + (split * R + row) * kDePartStride + 4 * c4);
                const uint32_t lo = ptx::pack_bf16(tier.scale * a.x, tier.scale * a.y);
                const uint32_t hi = ptx::pack_bf16(tier.scale * a.z, tier.scale * a.w);
                *reinterpret_cast<float4*>(code_s + row * kDePartStride + 4 * c4) =
                    make_float4(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u),
                                __uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
            }
            __syncthreads();
        }
    }
    {
        // ---- sum the S partials in split order, add the adapter, round once,
        // scatter into the latent
        const int P = p.P, PP = P * P;
        const size_t plane = (size_t)p.Hl * p.Wl;
        for (int q = threadIdx.x; q < R * per_row; q += kThreads) {
            const int row = split * R + q / per_row;
            const int c4 = q % per_row;
            const int m = mt * 128 + row;
            float4 acc = sum4(part + row * kDePartStride + 4 * c4);
            if constexpr (kTier) {
                const float* code = code_s + (q / per_row) * kDePartStride;
#pragma unroll 8
                for (int k = 0; k < tier.rank; ++k) {  // a multiple of 8
                    const float4 u = *reinterpret_cast<const float4*>(up_s + k * kDePartStride + 4 * c4);
                    const float c = code[k];
                    acc.x = fmaf(c, u.x, acc.x);
                    acc.y = fmaf(c, u.y, acc.y);
                    acc.z = fmaf(c, u.z, acc.z);
                    acc.w = fmaf(c, u.w, acc.w);
                }
            }
            if (m < p.M) {
                const int i = m / p.gw, jj = m % p.gw;
                __nv_bfloat16* lat =
                    p.latent + (size_t)b * p.C * plane + (size_t)(P * i) * p.Wl + (size_t)P * jj;
                const float vals[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int f = nt * kDeBN + 4 * c4 + e;
                    const int ch = f / PP, dy = (f % PP) / P, dx = f % P;
                    lat[(size_t)ch * plane + (size_t)dy * p.Wl + dx] = __float2bfloat16_rn(vals[e]);
                }
            }
        }
    }
    // No CTA leaves while another may still read its shared memory.
    ptx::cluster_sync();
    __syncthreads();
    if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tbase, kTier ? 2 * kDeBN : kDeBN);
    }
}

constexpr int kDeSmem = kDeStages * (kChunkA + kDeBN * 128) + 1024;
// With an adapter or residual: three stages, then two partial tiles, the up
// projection and 128 / splits rows of codes in their space, so that two CTAs
// share an SM (a 480p coarse state has 16 clusters of eight CTAs, and with one
// CTA per SM only 15 of them ran at once: 21.7 us).
constexpr int de_tier_smem(int splits) {
    const int ring = kDeTierStages * (kChunkA + 2 * kDeBN * 128);
    const int sums = (128 + 128 + 64 + 128 / splits) * kDePartStride * 4;
    return (ring > sums ? ring : sums) + 1024;
}
static_assert(128 * kDePartStride * 4 <= kDeStages * (kChunkA + kDeBN * 128), "partial tile fits the ring");


constexpr int kEmbedSmem = kEmbedStages * (kChunkA + kEmbedBN * 128) + 1024;

}  // namespace

bool msp_embed_supported(const MspEmbedRun* runs, int n, int E) {
    if (n < 1 || n > kMaxGemmProblems || E % 64 != 0 || E <= 0) return false;
    for (int i = 0; i < n; ++i) {
        const MspEmbedRun& r = runs[i];
        if (r.K % 64 != 0 || r.P < 1 || 64 % r.P != 0 || ((uintptr_t)r.w & 15) || r.M <= 0) return false;
        if (r.lora_up && (r.rank < 8 || r.rank > 64 || r.rank % 8 != 0 || !r.lora_down ||
                          ((uintptr_t)r.lora_up & 15) || ((uintptr_t)r.lora_down & 15)))
            return false;
    }
    return true;
}

cudaError_t launch_msp_embed(const MspEmbedRun* runs, int n, const MspShape& sh, int E, const void* latent,
                             void* tokens, long long tok_bstride, int batch, unsigned int* status,
                             cudaStream_t st, const PoolBatch* pool) {
    EmbedMaps maps;
    memset(&maps, 0, sizeof(maps));
    LoraMaps lmaps;
    bool lora = false;
    EmbedParams p;
    memset(&p, 0, sizeof(p));
    int tiles = 0;
    for (int i = 0; i < n; ++i) {
        const MspEmbedRun& r = runs[i];
        const int bn = r.lora_up ? kLoraBN : kEmbedBN;
        if (!encode_2d(&maps.w[i], r.w, r.K, E, (long long)r.K * 2, 64, bn)) return cudaErrorInvalidValue;
        if (r.lora_up) {
            lora = true;
            if (!encode_2d(&lmaps.up[i], r.lora_up, r.rank, E, (long long)r.rank * 2, 64, bn) ||
                !encode_2d(&lmaps.down[i], r.lora_down, r.K, r.rank, (long long)r.K * 2, 64, 64))
                return cudaErrorInvalidValue;
        }
        {
            EncodeTiledFn enc = encoder();
            cuuint64_t dims[3] = {(cuuint64_t)E, (cuuint64_t)r.M, (cuuint64_t)batch};
            cuuint64_t strides[2] = {(cuuint64_t)E * 2, (cuuint64_t)tok_bstride * 2};
            cuuint32_t box[3] = {64, 128, 1};
            cuuint32_t es[3] = {1, 1, 1};
            if (!enc || enc(&maps.out[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                            (char*)tokens + (size_t)r.tok_off * E * 2, dims, strides, box, es,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
        }
        EmbedRun& R = p.run[i];
        R.tile_base = tiles;
        R.m_tiles = (r.M + 127) / 128;
        R.M = r.M;
        R.l0 = r.l0;
        R.n_l = r.n_l;
        R.gw = r.gw;
        R.P = r.P;
        R.K = r.K;
        R.tok_off = r.tok_off;
        R.lora = r.lora_up ? 1 : 0;
        R.scale = r.lora_scale;
        tiles += R.m_tiles * ((E + bn - 1) / bn);
    }
    p.n_runs = n;
    p.T = sh.T;
    p.C = sh.C;
    p.Hl = sh.Hl;
    p.Wl = sh.Wl;
    p.E = E;
    p.latent = (const __nv_bfloat16*)latent;
    p.tokens = (__nv_bfloat16*)tokens;
    p.tok_bstride = tok_bstride;
    p.status = status;
    if (lora && pool && pool->n > 0) return cudaErrorInvalidValue;  // no caller pools beside adapters
    p.n_embed_tiles = tiles;
    PoolBatch pb;
    if (pool && pool->n > 0) {
        pb = *pool;
        int max_n = 0;
        for (int k = 0; k < pb.n; ++k) max_n = pb.j[k].out_n > max_n ? pb.j[k].out_n : max_n;
        p.pool_tasks = max_n * (pb.row_vecs / 2);
        const long long total = (long long)pb.n * p.pool_tasks;
        auto share_of = [&](int one, int more) {
            long long x = 0;
            for (int i = 0; i < n; ++i)
                x += 64ll * (p.run[i].K <= 64 ? one : more) * ((i + 1 < n ? p.run[i + 1].tile_base : tiles) - p.run[i].tile_base);
            return x;
        };
        int sms = 0;
        const cudaError_t e = device_sms(&sms);
        if (e != cudaSuccess) return e;
        const IdleTasks idle = idle_tasks(batch * (tiles + (total + kThreads - 1) / kThreads), sms, total,
                                          share_of(2, 4), share_of(1, 3));
        for (int i = 0; i < n && idle.one > 0; ++i) {
            EmbedRun& R = p.run[i];
            R.pool_base = p.pool_first;
            R.pool_per = R.K <= 64 ? idle.one : idle.more;
            p.pool_first += 64 * R.pool_per * ((i + 1 < n ? p.run[i + 1].tile_base : tiles) - R.tile_base);
        }
        p.pool_ctas = (int)((total - p.pool_first + kThreads - 1) / kThreads);
    } else {
        memset(&pb, 0, sizeof(pb));
    }
    const bool share = p.pool_first > 0;
    const void* fn = lora    ? (const void*)msp_embed_kernel<true, false, LoraMaps>
                     : share ? (const void*)msp_embed_kernel<false, true, NoLora>
                             : (const void*)msp_embed_kernel<false, false, NoLora>;
    cudaError_t e = set_smem_attr(fn, kEmbedSmem, 100);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(tiles + p.pool_ctas), 1, (unsigned)batch);
    if (lora)
        return launch_pdl(msp_embed_kernel<true, false, LoraMaps>, grid, dim3(kThreads), kEmbedSmem, st, maps, p, pb,
                          lmaps);
    return share ? launch_pdl(msp_embed_kernel<false, true, NoLora>, grid, dim3(kThreads), kEmbedSmem, st, maps, p, pb,
                              NoLora{})
                 : launch_pdl(msp_embed_kernel<false, false, NoLora>, grid, dim3(kThreads), kEmbedSmem, st, maps, p,
                              pb, NoLora{});
}


bool msp_deembed_supported(int M, int F, int E) {
    return M > 0 && F % kDeBN == 0 && E % 64 == 0 && E >= 64;
}

cudaError_t launch_msp_deembed(const void* tokens, long long tok_bstride_elems, int tok_rows, int tok_row0,
                               const void* w_out, int M, int F, int E, const MspShape& sh, int P, void* latent,
                               int batch, unsigned int* status, cudaStream_t st, const DeembedTier* tier) {
    DeembedMaps maps;
    memset(&maps, 0, sizeof(maps));
    EncodeTiledFn enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    {
        cuuint64_t dims[3] = {(cuuint64_t)E, (cuuint64_t)tok_rows, (cuuint64_t)batch};
        cuuint64_t strides[2] = {(cuuint64_t)E * 2, (cuuint64_t)tok_bstride_elems * 2};
        cuuint32_t box[3] = {64, 128, 1};
        cuuint32_t es[3] = {1, 1, 1};
        if (enc(&maps.a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(tokens), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    if (!encode_2d(&maps.b, w_out, E, F, (long long)E * 2, 64, kDeBN)) return cudaErrorInvalidValue;
    const bool lora = tier && tier->up;
    const bool res = tier && tier->residual;
    if (lora && !encode_2d(&maps.down, tier->down, E, tier->rank, (long long)E * 2, 64, kDeBN))
        return cudaErrorInvalidValue;
    if (res && !encode_2d(&maps.res, tier->residual, F, F, (long long)F * 2, 64, kDeBN)) return cudaErrorInvalidValue;
    const int nk_all = E / 64 + (res ? F / 64 : 0);
    // Splits (the cluster size) by the number of clusters, as measured. Launches
    // in a row favour one wave: E 1536, eight / four / two / one: 13 tiles 5.6 /
    // 6.5 / 9.6 / 15.0 us, 26 8.0 / 6.7 / 9.8 / 15.1, 52 14.6 / 9.1 / 10.0 / 15.3, 111
    // 27.3 / 17.8 / 13.7 / 15.5. Behind an attention launch, whose CTAs do not end
    // together, the shorter chain of eight is still ahead at two waves (whole
    // step, eight / four / two): 18 tiles 42.5 / 44.2 / 48.0 us, 26 161.8 / 163.2 /
    // 168.0, 39 118.7 / 116.7 / 119.6, 52 113.9 / 109.6 / 113.2, 78 161.5 / 155.6 /
    // 153.9, two and one from 156 on within 1 %. With extras, the tiers of a window
    // in turn (eight / four / two / one): 16 tiles 61.3 / 57.2 / 69.9 / 100.4 us, 32
    // 75.8 / 77.6 / 83.0 / 113.9, 48 111.8 / 90.2 / 91.6 / 123.3, 64 124.2 / 97.6 /
    // 109.1 / 131.5, 80 155.3 / 129.5 / 122.7 / 139.8, and from there on two (160
    // 266.8 / 213.7 / 200.1 / 238.1: one CTA's gather and sums are too long a
    // chain). Each split keeps at least one K chunk.
    const int clusters = (M + 127) / 128 * (F / kDeBN) * batch;
    const bool extras = lora || res;
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    int splits = clusters <= (extras ? 15 : 30) ? 8 : clusters <= 72 ? 4 : extras || clusters <= sms ? 2 : 1;
    while (splits > 1 && splits > nk_all) splits /= 2;
    DeembedParams p;
    memset(&p, 0, sizeof(p));
    p.M = M;
    p.K = E;
    p.nk_all = nk_all;
    p.m_tiles = (M + 127) / 128;
    p.splits = splits;
    p.P = P;
    p.gw = sh.Wl / P;
    p.C = sh.C;
    p.Hl = sh.Hl;
    p.Wl = sh.Wl;
    p.tok_row0 = tok_row0;
    p.latent = (__nv_bfloat16*)latent;
    p.status = status;
    const dim3 grid((unsigned)(p.m_tiles * (F / kDeBN)), (unsigned)splits, (unsigned)batch);
    const dim3 cluster(1, (unsigned)splits, 1);
    if (lora || res) {
        DeembedTierParams tp;
        memset(&tp, 0, sizeof(tp));
        tp.rank = lora ? tier->rank : 0;
        tp.scale = tier->scale;
        tp.up = (const __nv_bfloat16*)tier->up;
        tp.latent = (const __nv_bfloat16*)tier->latent;
        tp.latent_bstride = tier->latent_bstride;
        e = set_smem_attr((const void*)msp_deembed_kernel<true, DeembedTierParams>, de_tier_smem(1), 100);
        if (e != cudaSuccess) return e;
        return launch_pdl_cluster(msp_deembed_kernel<true, DeembedTierParams>, grid, dim3(kThreads),
                                  de_tier_smem(splits), st, cluster, maps, p, tp);
    }
    e = set_smem_attr((const void*)msp_deembed_kernel<false, NoTier>, kDeSmem);
    if (e != cudaSuccess) return e;
    return launch_pdl_cluster(msp_deembed_kernel<false, NoTier>, grid, dim3(kThreads), kDeSmem, st, cluster, maps, p,
                              NoTier{});
}

}  // namespace msf
