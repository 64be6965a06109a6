// morton.cuh -- the domain cube and the 63-bit Morton keys (paper Sect. 2,
// "Sorting of the particles along a Space Filling Curve (Morton)").
//
// The cube corner is the per-axis minimum and its side S the smallest power
// of two strictly greater than the largest extent, so that the quantisation
//   q_d = floor((x_d - mn_d) * 2^21 / S)
// is exact as (int)(__fsub_rd(x_d, mn_d) * (2^21 / S)): the round-down
// subtraction never exceeds the exact difference and floor(v 2^21/S)*S/2^21
// is itself a float <= v, so both floors agree; the multiply by a power of
// two is exact.
#pragma once
#include "common.cuh"

namespace bonsai {

// Smallest power of two strictly greater than the exact difference hi - lo.
__device__ __forceinline__ float pow2_above_diff(float hi, float lo) {
    float e_rd = __fsub_rd(hi, lo), e_ru = __fsub_ru(hi, lo);
    if (!(e_ru > 0.f)) return 0.f;
    int ex;
    float m = frexpf(e_ru, &ex);           // e_ru = m 2^ex, m in [0.5, 1)
    if (e_rd == e_ru) return ldexpf(1.f, ex);          // exact: 2^(floor(log2 e) + 1)
    return (m == 0.5f) ? e_ru : ldexpf(1.f, ex);       // inexact: smallest pow2 >= e_ru
}

// Domain of a system from its bounding box (dom: orderable-int min xyz, max
// xyz): corner mn, side S; returns 2^21 / S.
__device__ __forceinline__ float domain_of(const int *dom, float (&mn)[3], float &side) {
    float S = 0x1p-64f;
    for (int d = 0; d < 3; d++) {
        const float lo = ord2f(dom[d]), hi = ord2f(dom[3 + d]);
        mn[d] = lo;
        S = fmaxf(S, pow2_above_diff(hi, lo));
    }
    int ex;
    frexpf(S, &ex);                        // S = 2^(ex-1)
    side = S;
    return ldexpf(1.f, KEY_BITS_PER_AXIS - (ex - 1));
}

// Spread the low 21 bits of v to every third bit (bit b -> bit 3b).
__device__ __forceinline__ unsigned long long spread3(unsigned v) {
    unsigned long long x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x001f00000000ffffull;
    x = (x | (x << 16)) & 0x001f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// Key of a position in the cube dm = (mn xyz, 2^21 / S).
__device__ __forceinline__ unsigned long long morton_key(const float4 q, const float4 dm) {
    const unsigned qmax = (1u << KEY_BITS_PER_AXIS) - 1u;
    const unsigned qx = min((unsigned)(__fsub_rd(q.x, dm.x) * dm.w), qmax);
    const unsigned qy = min((unsigned)(__fsub_rd(q.y, dm.y) * dm.w), qmax);
    const unsigned qz = min((unsigned)(__fsub_rd(q.z, dm.z) * dm.w), qmax);
    return spread3(qx) | (spread3(qy) << 1) | (spread3(qz) << 2);
}

}  // namespace bonsai
