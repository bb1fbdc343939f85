// nls_pivot.cuh -- the CTA tilings' reciprocal of a pivot.
#pragma once

#include "nls_common.cuh"

namespace nls {

// The reciprocal that the multipliers take; ok becomes false where the pivot
// is zero, an infinity or a NaN.  FP32: the hardware approximation, whose error is
// inside the FP32 LU's own rounding.  It flushes subnormal numbers, and with them
// the reciprocals of pivots above 2^126 (whose multipliers would be zero), so the
// pivot is scaled by 2^-64 (from 2 on) or 2^64 into the middle of the range and the
// result by the same factor: exact, one logical operation and two products.  (A
// branch to the rounded reciprocal: 2.5% more on the Bratu n = 64..128 set.)  FP64:
// the rounded one.
NLS_DI float pivot_reciprocal(float x, bool &ok)
{
    const uint32_t m = mag_bits(x);
    if (m == 0u || m >= INF32_BITS) ok = false;
    const float s = __uint_as_float((__float_as_uint(x) & 0x40000000u) ^ 0x5f800000u);
    return pivot_rcp(x * s) * s;
}
NLS_DI double pivot_reciprocal(double x, bool &ok)
{
    const uint64_t m = mag_bits(x);
    if (m == 0u || m >= INF64_BITS) ok = false;
    return rcp(x);
}

} // namespace nls
