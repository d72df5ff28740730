// fp32 projections on the tensor cores (three bf16 planes per value).
#pragma once

#include <cuda_runtime.h>

#include "kernels.h"

namespace msf {

constexpr int kMaxGemmF32 = MSF_MAX_STATES;

// Whether the kernel takes this fp32 problem: C = A B^T with vectors of four
// along K and N.
bool gemm_f32_tc_supported(const GemmArgs& g);
// n such problems in one launch. `scatter` (one problem): its rows are the
// tokens of one state of patch edge `P`, and the result goes to the latent
// [B, C, Hl, Wl] at g->C instead of rows.
cudaError_t launch_gemm_f32_tc(const GemmArgs* g, int n, int batch, unsigned int* status, cudaStream_t st,
                               const MspShape* scatter = nullptr, int P = 0);

}  // namespace msf
