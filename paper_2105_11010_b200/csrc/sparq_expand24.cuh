// A group of four activations -> the six pairs a 2:4 pattern can select, transformed (Sections 4, 5.3).
#pragma once

#include "sparq_common.cuh"

namespace sparq {

// x: the group's bytes; o0..o2: T2 of the pairs (0,1) (0,2) | (0,3) (1,2) | (1,3) (2,3).
// Every value is either its own bSPARQ result or, beside a zero, its wider window, whatever the
// pair: both are computed once per activation and then copied and selected per pair.
// XN as in xform_fused: 4 = n = 4 with all placements, 8 = another full set, 0 = any set.
template <int XN, bool RND>
__device__ __forceinline__ void expand_group(uint32_t x, const XformDev &d, uint32_t &o0, uint32_t &o1, uint32_t &o2)
{
    const uint32_t q = xform_fused<SPARQ_MODE_BSPARQ, XN, RND>(x, d);
    uint32_t l = x;                                   // beside a zero: the whole byte for n = 4
    if (XN != 4 && d.n != 4) {
        if (XN == 8) {
            const uint32_t k1024 = 0x64006400u;
            const uint32_t lo = h2_sub(prmt(x, 0x64646464u, 0x4140u), k1024), hi = h2_sub(prmt(x, 0x64646464u, 0x4342u), k1024);
            l = prmt(h2_add(h2_min((lo + d.l_add) & d.l_mask, d.l_sat), k1024),
                     h2_add(h2_min((hi + d.l_add) & d.l_mask, d.l_sat), k1024), 0x6420u);
        } else {
            l = apply_mask<RND>(x, drop_mask<0, false>(x, 2 * d.n, 0u), 2 * d.n);
        }
    }
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
