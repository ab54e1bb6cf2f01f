// exact_split.cuh -- sums of FP32 couplings without rounding in FP32: x in [-1, 1] is
// split into multiples of 2^-17, multiples of 2^-35 and the rest by adding and
// subtracting a constant whose last place is that step.
#pragma once

namespace pb {

constexpr float kSplit1 = 96.0f;           // 1.5 2^6: last place 2^-17
constexpr float kSplit2 = 0.0003662109375f;  // 1.5 2^-12: last place 2^-35

}  // namespace pb
