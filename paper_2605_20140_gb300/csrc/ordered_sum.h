// Sums in the order of the array, to the bit, without adding one by one.
// The state's reference mass and the offset of the v transform are sums of the
// input in array order; their rounding enters every later step, so a faster way to
// them has to give the same bits.
#pragma once

#include <float.h>
#include <math.h>
#include <stdint.h>

namespace sipf {

// ((m + m) + m) + ... with n terms, m > 0 finite, each addition rounded to
// nearest.  While the running sum stays in one binade its spacing u is fixed,
// so every addition rounds m to the same multiple d of u (unless m lies
// halfway between two, where the even neighbour alternates) and t additions
// give acc + t d, a multiple of u below the binade's end and so exact.  About
// one round per binade instead of n dependent additions.
inline double ordered_sum_of_equal(double m, int64_t n) {
    double acc = 0.0;
    while (n > 0) {
        const double next = acc + m;
        if (!isfinite(next)) return next;
        --n;
        if (acc > 0.0 && n > 0) {
            const double end = ldexp(1.0, ilogb(acc) + 1);   // acc lies in [end/2, end)
            const double d = next - acc;                      // exact: both are multiples of u
            // m - d is exact (|m - d| <= u/2, both multiples of m's spacing or finer)
            const bool tie = fabs(m - d) == 0.5 * ldexp(1.0, ilogb(acc) - 52);
            if (!tie && d > 0.0 && next < end) {
                // steps that certainly stay below end (m <= d + u/2 < 2 d + u), and below
                // the largest number in the topmost binade, whose end is not one
                const double room = (isfinite(end) ? end : DBL_MAX) - next;
                int64_t t = static_cast<int64_t>(room / d) - 3;
                if (t > n) t = n;
                if (t > 0) {
                    acc = next + static_cast<double>(t) * d;
                    n -= t;
                    continue;
                }
            }
        }
        acc = next;
    }
    return acc;
}

// Whether a sum of n values, each a multiple of 2^low and at most max_abs in
// magnitude, is exact in float64 in every order: all partial sums are multiples of 2^low
// below n max_abs, which fits when that is at most 2^(53 + low).
inline bool any_order_exact(int64_t n, double max_abs, int low) {
    return static_cast<double>(n) * max_abs <= ldexp(1.0, 53 + (low < 900 ? low : 900));
}

}  // namespace sipf
