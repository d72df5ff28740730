// fp32 MSSA attention on the tensor cores (three bf16 planes per fp32 value).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"
#include "kernels.h"

namespace msf {

// The fp32 attention of `a` (a plan with fp32 tensors, workspace bound): the
// operands split into bf16 planes, the tensor-core kernel, the merge of split
// query tiles, and the CUDA-core kernel, which runs only where the planes
// cannot hold an operand (a value that is not finite or not below 2^127).
msf_status launch_attn_f32_tc(msf_plan_t plan, const AttnArgs& a, cudaStream_t st);

}  // namespace msf
