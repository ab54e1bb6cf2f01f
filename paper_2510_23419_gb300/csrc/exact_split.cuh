// exact_split.cuh -- FP64-accurate sums of FP32 couplings at FP32 speed.  With u = 2^e at least the largest
// magnitude, a coupling is split into multiples of 2^-17 u, of 2^-35 u and of 2^-53 u by adding and subtracting a
// constant whose last place is that step; sums of 64 of any one part are exact in FP32.  What has no such split (of
// N(0,1) draws one in 600 into two parts, one in 10^8 into three) the caller sums whole and at full accuracy.
#pragma once

#include <cmath>
#include <cstdint>
#include <limits>

namespace pb {

constexpr float kSplit1 = 96.0f;             // 1.5 2^6: last place 2^-17
constexpr float kSplit2 = 0.0003662109375f;  // 1.5 2^-12: last place 2^-35
constexpr float kSplit3 = 1.5f / (1 << 30);  // 1.5 2^-30: last place 2^-53

// u for couplings of magnitude up to amax; infinity where the constants or the sums would leave the FP32 range, which
// makes the splits refuse every coupling.
inline float split_unit(float amax)
{
    int e = 0;
    if (amax > 0.0f) std::frexp(amax, &e);  // amax <= 2^e
    return e >= -90 && e <= 120 ? std::ldexp(1.0f, e) : std::numeric_limits<float>::infinity();
}

#ifdef __CUDACC__
// The part of x that is a multiple of the last place of k (u times a constant above); x - part is exact.
__device__ __forceinline__ float split_part(float x, float k) { return __fadd_rn(__fadd_rn(x, k), -k); }

// x = q1 + q2 exactly, or false (and q1, q2 unspecified).
__device__ __forceinline__ bool split_exact(float x, float u, float& q1, float& q2)
{
    q1 = split_part(x, kSplit1 * u);
    const float x1 = __fadd_rn(x, -q1);
    q2 = split_part(x1, kSplit2 * u);
    return q2 == x1;
}
// x = q1 + q2 + q3 exactly, or false.
__device__ __forceinline__ bool split_exact(float x, float u, float& q1, float& q2, float& q3)
{
    q1 = split_part(x, kSplit1 * u);
    const float x1 = __fadd_rn(x, -q1);
    q2 = split_part(x1, kSplit2 * u);
    const float x2 = __fadd_rn(x1, -q2);
    q3 = split_part(x2, kSplit3 * u);
    return q3 == x2;
}
#endif

}  // namespace pb
