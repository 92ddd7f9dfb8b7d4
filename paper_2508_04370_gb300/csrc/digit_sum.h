// Integer recombination of the sliced update's accumulators (host and device;
// no arithmetic here leaves the range of its type).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define IPM_DIGIT_FN __host__ __device__ __forceinline__
#else
#define IPM_DIGIT_FN inline
#endif

namespace ipm {
namespace sliced {

// Bits of the float 1.5 * 2^23: an integer |a| < 2^22 added to that float in FP32
// leaves the bits kIntBias + a.
constexpr uint32_t kIntBias = 0x4B400000u;

// 128 a + b (below 2^30) from the biased bits of a and b.  The biased bits times
// 128 pass 2^32, so the biases cancel modulo 2^32, in unsigned arithmetic: in int the
// product overflows, and a compiler may then carry it in 64 bits and keep what
// should have wrapped.
IPM_DIGIT_FN int32_t digit_pair(uint32_t a, uint32_t b) {
    return (int32_t)(a * 128u + b - 129u * kIntBias);
}

// T 2^-8 for T = sum_d S_d 2^(7 (7 - d)), rounded down, in two halves so that four
// accumulators are held at a time: first the pairs 128 S_4 + S_5 and
// 128 S_6 + S_7, then, added to that, 128 S_0 + S_1 and 128 S_2 + S_3.  With
// |S_d| <= 2^21.4 below 2^62.5.
IPM_DIGIT_FN int64_t digit_low(int32_t s45, int32_t s67) { return (int64_t)s45 * 64 + (s67 >> 8); }
IPM_DIGIT_FN int64_t digit_sum(int64_t low, int32_t s01, int32_t s23) {
    return low + (int64_t)s23 * (int64_t(1) << 20) + (int64_t)s01 * (int64_t(1) << 34);
}

}  // namespace sliced
}  // namespace ipm
