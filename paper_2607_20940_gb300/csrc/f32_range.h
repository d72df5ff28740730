// Which fp32 operands the tensor-core paths take (three bf16 planes per value,
// see attn_f32_tc.cu); the others go to the CUDA-core kernels. Free of CUDA so
// that the host can run the rule too.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MSF_RANGE_FN __host__ __device__ __forceinline__
#else
#define MSF_RANGE_FN inline
#endif

namespace msf {

// A value's planes miss it by 2^-25 of itself, or by bf16's smallest normal
// number, 2^-126, whichever is more. Values are judged in the vectors that a
// thread splits (eight neighbours along the head, four along a GEMM's K): a
// vector that is not all zeros has to reach 2^-96, which makes that 2^-30 of its
// largest value. The largest value of an operand bounds its products and sums.
constexpr int kRangeBias = 127;
constexpr int kRangeLeast = kRangeBias - 96;  // exponent field of a vector's largest value
constexpr uint32_t kRangeBad = 255;

// The range code of a vector whose largest magnitude has these bits: 0 for all
// zeros, the exponent field, or kRangeBad where the planes cannot hold it (below
// the bound; not finite, or 2^127 and more, which can round to infinity). The
// code of several vectors is their largest.
MSF_RANGE_FN uint32_t range_code(uint32_t abs_bits) {
    const uint32_t e = abs_bits >> 23;
    return abs_bits == 0 ? 0u : e < (uint32_t)kRangeLeast || e >= 254u ? kRangeBad : e;
}

// Sums of products of operands with these codes: largest terms between 2^lo and
// 2^hi (any, if one operand is all zeros). Above 2^-100 the smallest plane products
// are normal numbers; the upper bounds keep plane products, whose signs differ from
// the sum's, and the sums finite.
MSF_RANGE_FN bool range_product(int a, int b, int lo, int hi) {
    const int s = a + b - 2 * kRangeBias;
    return a == 0 || b == 0 || (s >= lo && s <= hi);
}

// The attention's operands, a code per byte.
enum : int { kRangeQ = 0, kRangeK = 1, kRangeV = 2, kRangeDout = 3 };

// Whether the planes hold a call: q and k, v, and dout in a gradient (0 in a
// forward pass). `scale_exp`: exponent of the softmax scale in log2 units.
//   S = q k      sums of 128: below 2^(116 + 9), also after the scale
//   P v, P^T dO  probabilities up to 1, up to 2^24 keys: below 2^(96 + 26)
//   dP = dO v    above 2^-70, so that dS = P (dP - delta) keeps its planes with
//                probabilities down to 2^-26
//   dS k, dS q   the sums of three
MSF_RANGE_FN bool range_holds(uint32_t codes, int scale_exp) {
    const int q = codes & 255, k = (codes >> 8) & 255, v = (codes >> 16) & 255, g = codes >> 24;
    if (q == 255 || k == 255 || v == 255 || g == 255) return false;
    if (!range_product(q, k, -100, scale_exp > 0 ? 116 - scale_exp : 116)) return false;
    if (v > kRangeBias + 96 || g > kRangeBias + 96) return false;
    if (g == 0 || v == 0) return true;
    if (!range_product(g, v, -70, 80)) return false;
    const int ds = g + v - kRangeBias;  // code of dP
    return (q == 0 || range_product(ds, q, -80, 80)) && (k == 0 || range_product(ds, k, -80, 80));
}

// A GEMM's operands (up to 2^16 products a sum).
MSF_RANGE_FN bool range_holds_gemm(uint32_t a, uint32_t b) {
    return a != kRangeBad && b != kRangeBad && range_product((int)a, (int)b, -100, 105);
}

// What the plane split found in a call's operands: one word of codes per block.
struct F32Range {
    unsigned int* words;  // NULL: no condition
    int n;
    int scale_exp;
    // The kernel after the split leaves its answer here (1: the planes hold) for the
    // ones behind it.
    unsigned int* answer;
};

}  // namespace msf
