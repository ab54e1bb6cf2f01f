// ea_philox.cuh -- Philox4x32-10 with the round keys in registers and the first
// round's products of counter words 1..3 hoisted, for kernels that draw many
// words whose counters differ in word 0 only (the EA resident tiles).
#pragma once

#include "pb_common.h"

namespace pb {

struct RoundKeys {
    uint32_t k0[10], k1[10];
};

__device__ __forceinline__ RoundKeys round_keys(uint32_t key0, uint32_t key1)
{
    RoundKeys k;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        k.k0[r] = key0 + (uint32_t)r * kPhiloxWeylA;
        k.k1[r] = key1 + (uint32_t)r * kPhiloxWeylB;
    }
    return k;
}

// First-round terms that do not depend on counter word 0.
struct PhiloxPre {
    uint32_t n0, n1, x3;
};

__device__ __forceinline__ PhiloxPre philox_pre(uint32_t c1, uint32_t c2, uint32_t c3, const RoundKeys& k)
{
    uint32_t hB, lB;
    mulhilo32(kPhiloxMulB, c2, hB, lB);
    return PhiloxPre{hB ^ c1 ^ k.k0[0], lB, c3 ^ k.k1[0]};
}

// Philox4x32-10 of counter (c0, c1, c2, c3), with (c1, c2, c3) folded into `p`.
__device__ __forceinline__ U4 philox_c0(uint32_t c0, const PhiloxPre& p, const RoundKeys& k)
{
    uint32_t hA, lA;
    mulhilo32(kPhiloxMulA, c0, hA, lA);
    uint32_t x0 = p.n0, x1 = p.n1, x2 = hA ^ p.x3, x3 = lA;
#pragma unroll
    for (int r = 1; r < 10; ++r) {
        uint32_t hA2, lA2, hB2, lB2;
        mulhilo32(kPhiloxMulA, x0, hA2, lA2);
        mulhilo32(kPhiloxMulB, x2, hB2, lB2);
        const uint32_t y0 = hB2 ^ x1 ^ k.k0[r];
        const uint32_t y2 = hA2 ^ x3 ^ k.k1[r];
        x0 = y0;
        x1 = lB2;
        x2 = y2;
        x3 = lA2;
    }
    return U4{x0, x1, x2, x3};
}

}  // namespace pb
