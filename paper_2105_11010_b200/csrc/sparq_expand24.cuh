// A group of four activations -> the six pairs a 2:4 pattern can select, transformed (Sections 4, 5.3).
#pragma once

#include "sparq_common.cuh"

namespace sparq {

// x: the group's bytes; o0..o2: T2 of the pairs (0,1) (0,2) | (0,3) (1,2) | (1,3) (2,3).
// Every value is either its own bSPARQ result or, beside a zero, its wider window, whatever the
// pair: both are computed once per activation and then copied and selected per pair.
template <int XN, bool RND>
__device__ __forceinline__ void expand_group(uint32_t x, const XformDev &d, uint32_t &o0, uint32_t &o1, uint32_t &o2)
{
    uint32_t q, l;
    window_and_lone<XN, RND>(x, d, q, l);
    const uint32_t nz = ((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x;          // bit 7 of each byte: byte != 0
    auto word = [&](uint32_t pick, uint32_t partner) {                   // partner: the pair's other index, | 8
        const uint32_t m = prmt(nz, nz, partner);
        return (prmt(q, q, pick) & m) | (prmt(l, l, pick) & ~m);
    };
    o0 = word(0x2010u, 0x8A89u);
    o1 = word(0x2130u, 0x9A8Bu);
    o2 = word(0x3231u, 0xAB9Bu);
}

}  // namespace sparq
