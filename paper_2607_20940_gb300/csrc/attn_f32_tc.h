// fp32 MSSA attention on the tensor cores (three bf16 planes per fp32 value).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "attn_tc.h"
#include "f32_range.h"
#include "internal.h"
#include "kernels.h"

namespace msf {

// ---- the operands' planes (attn_f32_tc.cu)
struct SplitJob {
    const float* src;    // stream 0
    __nv_bfloat16* dst;  // stream 0, plane 0
    long long src_bstride, dst_bstride, dst_plane;  // elements
    int vecs;            // 8-element vectors per stream
    int operand;         // kRangeQ, ..
    long long base;      // first vector of the job (all streams) in the launch
};
constexpr int kMaxSplitJobs = 2 + 2 * (3 + MSF_MAX_GROUPS);
struct SplitParams {
    SplitJob j[kMaxSplitJobs];
    int n;
    long long total;
    unsigned int* words;  // one word of range codes per block (f32_range.h)
};
struct F32Maps {
    CUtensorMap q, dout;
    CUtensorMap k[kNumMaps];
    CUtensorMap v[kNumMaps];
};
// Keys of the longest context.
int f32_longest_context(const AttnArgs& a);
// Add the first `rows` rows per stream of a [B, .., H, D] fp32 tensor as planes
// [B, 3, alloc, H, D] at `dst` to the split, and encode their tensor map.
bool add_planes(const Plan& P, SplitParams& sp, int operand, const void* src, long long src_bstride_bytes, char* dst,
                int alloc, int rows, CUtensorMap* m);
// q and the k, v of every context segment of `a`, in the workspace's planes.
bool add_context_planes(const Plan& P, const AttnArgs& a, SplitParams& sp, F32Maps& maps);
// Write the planes and the range words, which *range then names.
cudaError_t launch_split_planes(const SplitParams& sp, float scale_log2, F32Range* range, cudaStream_t st);
// A class of equal own tiles (query tiles of a group, gradient rows of one) and
// the other tiles each walks; `weight`: the cost of one, K/V tile = 1.
constexpr int kMaxF32Classes = 3 * MSF_MAX_GROUPS;
struct F32Class {
    long long items;
    int n_tiles;
    double weight;
};
// The most tiles a unit of work may have (a tile of more is split evenly over
// several units, with a partial slot each): see the definition.
int f32_unit_tiles(const F32Class* c, int n, int D, int sms, int max_slots);

// The fp32 attention of `a` (a plan with fp32 tensors, workspace bound): the
// operands split into bf16 planes, the tensor-core kernel, the merge of split
// query tiles, and the CUDA-core kernel, which runs only where the planes
// cannot hold an operand (a value that is not finite or not below 2^127).
msf_status launch_attn_f32_tc(msf_plan_t plan, const AttnArgs& a, cudaStream_t st);

}  // namespace msf
