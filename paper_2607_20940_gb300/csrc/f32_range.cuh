// Device side of f32_range.h.
#pragma once

#include <cuda_runtime.h>

#include "f32_range.h"

namespace msf {

// The largest codes, byte by byte, over the warp.
__device__ __forceinline__ uint32_t warp_codes(uint32_t m) {
    uint32_t r = 0;
#pragma unroll
    for (int i = 0; i < 32; i += 8) r |= __reduce_max_sync(0xffffffffu, (m >> i) & 255u) << i;
    return r;
}

// Over every thread of the block (whole warps, all of them calling, once per kernel).
__device__ __forceinline__ uint32_t block_codes(uint32_t m) {
    __shared__ uint32_t of_warp[32];
    m = warp_codes(m);
    const int lane = threadIdx.x % 32;
    if (lane == 0) of_warp[threadIdx.x / 32] = m;
    __syncthreads();
    return warp_codes(lane < (int)blockDim.x / 32 ? of_warp[lane] : 0u);
}

// Whether the planes hold the operands of this call, from the split's words (every
// thread of the block); leaves the answer for the kernels behind this one.
__device__ __forceinline__ bool planes_hold(const F32Range& r) {
    uint32_t m = 0;
    for (int i = threadIdx.x; i < r.n; i += blockDim.x) m = __vmaxu4(m, __ldcg(r.words + i));
    const bool holds = range_holds(block_codes(m), r.scale_exp);
    if (blockIdx.x == 0 && threadIdx.x == 0) *r.answer = holds ? 1u : 0u;
    return holds;
}
// The same from the answer.
__device__ __forceinline__ bool planes_held(const F32Range& r) { return __ldcg(r.answer) != 0; }

// The largest magnitude of four values, as bits.
__device__ __forceinline__ uint32_t abs_bits4(const float4& x) {
    const uint32_t a = __float_as_uint(x.x) & 0x7fffffffu, b = __float_as_uint(x.y) & 0x7fffffffu;
    const uint32_t c = __float_as_uint(x.z) & 0x7fffffffu, d = __float_as_uint(x.w) & 0x7fffffffu;
    return max(max(a, b), max(c, d));
}

}  // namespace msf
