// Tensor-core MSSA backward (tcgen05 + TMA) launcher interface.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"
#include "kernels.h"

namespace msf {

struct BwdTcInput {
    const AttnArgs* a;    // the forward's context segments (q = the forward's q)
    const BwdGroup* g;    // per group (same order as a->g): rows that receive gradients
    const void* q;        // [B, N, H, D] bf16
    const void* dout;     // [B, N, H, D] bf16
    const float* lse;     // [B, H, N]
    const float* delta;   // [B, H, N]
    void* dq;             // [B, N, H, D] bf16, written
    float* dk_ctx;        // [B, R, H, D] fp32 context-row gradients, written
    float* dv_ctx;
    int R;
};

// dq (bf16) for every query (one launch), and the key/value gradients of
// every group's window-derived context rows (one launch).
msf_status launch_bwd_tc(msf_plan_t plan, const BwdTcInput& in, cudaStream_t st);

// What such a launch does on a device with `sms` SMs (host only).
struct BwdRoute {
    int items;
    int placed;  // 1: placed lists, 0: rounds of alternating direction
};
void bwd_route(const Plan& P, const AttnArgs& a, const BwdGroup* bg, int sms, BwdRoute* out);

// fp32 plans (attn_bwd_f32_tc.cu): dq and the context-row gradients on the
// tensor cores from three bf16 planes per value; dout_planes is scratch of
// f32_part_bytes(kF32Q). *range receives what says whether the CUDA-core
// kernels have to answer instead (no condition: nothing was launched here).
msf_status launch_bwd_f32_tc(msf_plan_t plan, const BwdCommon& c, const AttnArgs& a, const BwdGroup* bg, float* dq,
                             char* dout_planes, F32Range* range, cudaStream_t st);

}  // namespace msf
