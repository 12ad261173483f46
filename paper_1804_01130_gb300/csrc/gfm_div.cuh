// Exact quotients by a divisor whose inverse is known (device only).
#pragma once

namespace gfm {

namespace {

// a / b correctly rounded from inv = RN(1 / b): one Newton step on the
// quotient with an exact remainder (Markstein, IBM J. Res. Dev. 34, 1990), for
// |a| far from under- and overflow and a normal b whose significand is not
// all ones; the caller passes inv = 0 when b is not.  Three instructions of
// the FP64 pipe instead of a divide's ten or so.
__device__ __forceinline__ double div_known(double a, double b, double inv)
{
    const int e = (__double2hiint(a) >> 20) & 0x7ff;
    if (inv == 0.0 || e < 0x100 || e > 0x6ff) return a / b;
    const double q = a * inv;
    return fma(fma(-q, b, a), inv, q);
}

}  // namespace

}  // namespace gfm
