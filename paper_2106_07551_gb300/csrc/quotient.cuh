// fp64 division from a reciprocal that is at hand.
#pragma once

#include <cmath>
#include <cstring>

namespace malib {

// b / a from inv = 1 / a, correctly rounded, so that equal rationals tie (times the
// reciprocal alone, 49 / 49 and 1 / 1 give different doubles). q = b inv is within an
// ulp of the quotient; Markstein's correction step (IBM J. Res. Dev. 34 (1), 1990) adds
// its exact remainder times the reciprocal. Two FMAs where a second division costs 450
// cycles on this part: one linear program of 100 x 100, 346 -> 330 us. Outside 2^-500
// .. 2^500 the remainder could fall below fp64's range: a division there (the exponents
// are compared as integers; fp64 comparisons are as slow as its sums).
__host__ __device__ __forceinline__ double quotient(double b, double a, double inv) {
    const auto bits = [](double v) {
#ifdef __CUDA_ARCH__
        return (unsigned long long)__double_as_longlong(v);
#else
        unsigned long long u;
        std::memcpy(&u, &v, 8);
        return u;
#endif
    };
    const auto near_one = [&](double v) { return ((unsigned)(bits(v) >> 32) & 0x7fffffffu) - 0x20b00000u < 0x3e800000u; };
    const double q = b * inv;
    if (!near_one(a) || !(near_one(q) || bits(b) == 0ull)) return b / a;
    return fma(fma(-q, a, b), inv, q);
}

}  // namespace malib
