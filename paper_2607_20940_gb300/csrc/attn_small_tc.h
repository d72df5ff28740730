// Tensor-core MSSA attention of small calls: one query tile per cluster.
#pragma once

#include <cuda_runtime.h>

#include "attn_tc.h"
#include "internal.h"
#include "kernels.h"

namespace msf {

// Cluster size that the small-call kernel takes for these groups, 0 = the
// persistent kernel is the better one (see the definition).
// persistent_us: the estimated end of the persistent kernel.
int attn_small_cluster(const TcGroup* g, int n_groups, int H, int B, int D, int sms, double persistent_us);
cudaError_t launch_attn_small(const TcMaps& maps, const TcGroup* g, int n_groups, const Plan& P, const AttnArgs& a,
                              int cluster, cudaStream_t st);

}  // namespace msf
