// A quotient by a divisor whose inverse is known.
#pragma once

// n / det from the correctly rounded inverse of det: the quotient corrected by
// its residual (Markstein 1990), one multiplication and two fused multiply-adds
// in place of a division.  Equal to the division for numerators and quotients
// that are zero (of either sign) or between 2^-99 and 2^100 in size, where the
// residual is a normal number; smaller ones are within a unit of their last place
// and 2^-149.  An infinite numerator, which leaves no residual, gives no number
// where the division gives infinity; a solver that has come to one is lost either
// way, and a test for it costs the refinement 2.8 % (668 -> 687 us on 1024 x 436).
__device__ __forceinline__ float quotient(float n, float det, float inv) {
    const float q = n * inv;
    return __fmaf_rn(__fmaf_rn(-q, det, n), inv, q);
}
