// bit_count.cuh -- population counts over several words (products of +-1 vectors
// kept one bit per element: a . b = n - 2 popc(a ^ b)).
#pragma once

#include "pb_common.h"

namespace pb {

// Full adder of three words, bit by bit: sum s, carry c.
__device__ __forceinline__ void csa(uint32_t a, uint32_t b, uint32_t d, uint32_t& s, uint32_t& c)
{
    s = a ^ b ^ d;
    c = (a & b) | (d & (a | b));
}
// Seven words as bit counts o + 2 t + 4 f.
__device__ __forceinline__ void csa7(const uint32_t* x, uint32_t& o, uint32_t& t, uint32_t& f)
{
    uint32_t s1, c1, s2, c2, c3;
    csa(x[0], x[1], x[2], s1, c1);
    csa(x[3], x[4], x[5], s2, c2);
    csa(s1, s2, x[6], o, c3);
    csa(c1, c2, c3, t, f);
}

// Set bits of NW words x, carry-save compressed: four population counts (which run at
// a quarter of the other instructions' rate) for eight words, five for sixteen.
template <int NW>
__device__ __forceinline__ int popc_words(const uint32_t (&x)[NW])
{
    if constexpr (NW == 8) {
        uint32_t o, t, f;
        csa7(x, o, t, f);
        return __popc(o) + __popc(x[7]) + 2 * __popc(t) + 4 * __popc(f);
    } else if constexpr (NW == 16) {
        uint32_t o1, t1, f1, o2, t2, f2, o, t, f, c, e;
        csa7(x, o1, t1, f1);
        csa7(x + 7, o2, t2, f2);
        csa(o1, o2, x[14], o, c);
        csa(t1, t2, c, t, c);
        csa(f1, f2, c, f, e);
        return __popc(o) + __popc(x[15]) + 2 * __popc(t) + 4 * __popc(f) + 8 * __popc(e);
    } else {
        int t = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) t += __popc(x[w]);
        return t;
    }
}

}  // namespace pb
