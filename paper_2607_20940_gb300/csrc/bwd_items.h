// Bookkeeping of the persistent bf16 backward's items (attn_bwd_tc.cu), free of
// CUDA so that the host can run it too.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MSF_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MSF_HOST_DEVICE inline
#endif

namespace msf {

// The barrier that says that a CTA's k-th item is done, and the parity of its
// phase there. A parity wait can tell a phase only from the one before it, and
// item k - 1 may be done by the time the producer, about to load item k, asks for
// item k - 2: on one barrier "both done" would look like "neither done". With a
// barrier per item parity, item k is the next to complete on the one asked, and
// it has not been loaded yet.
constexpr int kDoneBars = 2;
MSF_HOST_DEVICE int done_bar(int k) { return k & 1; }
MSF_HOST_DEVICE uint32_t done_parity(int k) { return (uint32_t)((k >> 1) & 1); }

}  // namespace msf
