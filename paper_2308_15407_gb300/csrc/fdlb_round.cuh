// Stochastic rounding of FP32 storage (why: see the update kernel).
#pragma once
#include <stdint.h>

namespace fdlb {

// base + inc stored as a float, in expectation exactly: the sum's truncation t, or the next float away
// from zero with probability rem/gap, rem = base + inc - t (TwoSum), to 2^-25 of the gap: 24 random bits
// j, j + 1/2 compared with 2^24 rem/gap, all products exact.  Truncated, the gap beyond t is t's own
// last place at powers of two and down to the subnormals alike, and sums of either sign mirror each other.
// 15 instructions and no branch (2048 mixed instances: update 651 us per launch, 655 with the uniform
// number below).  (Rounding to nearest first makes the neighbour and its distance
// depend on the sign of the remainder and on whether the value is a power of two: 25 instructions and a
// branch.  Adding a uniform number of (-gap/2, gap/2) to the rounded sum, 15 instructions, holds a
// value that creeps up through a power of two, whose lower neighbour is half as far.)
__device__ __forceinline__ float sr_add(float base, float inc, uint32_t bits) {
    const float t = __fadd_rz(base, inc);
    const float bb = __fsub_rn(t, base);
    const float rem = __fadd_rn(__fsub_rn(base, __fsub_rn(t, bb)), __fsub_rn(inc, bb));
    const float next = __uint_as_float(__float_as_uint(t) + 1u);
    const float gap = __fsub_rn(fabsf(next), fabsf(t));
    const float j = __uint2float_rn(bits >> 8);
    return __fmul_rn(j, gap) < __fmaf_rn(gap, -0.5f, __fmul_rn(fabsf(rem), 0x1p24f)) ? next : t;
}

}  // namespace fdlb
