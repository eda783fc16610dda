// Upper bounds on prime counts, which size the device buffers that a generated
// range of primes goes to (host code).
#pragma once
#include <math.h>
#include <stdint.h>

#include <algorithm>

namespace cs {

// pi(x) bounds of P. Dusart (2010): x/ln x (1 + 1/ln x + 2/ln^2 x) <= pi(x) for
// x >= 88789 and pi(x) <= x/ln x (1 + 1/ln x + 2.51/ln^2 x) for x >= 355991.
inline double pi_upper(double x) {
    if (x < 355991.0) return x < 2 ? 0 : 1.26 * x / log(x) + 16;   // Rosser-Schoenfeld for small x
    const double l = log(x);
    return x / l * (1 + 1 / l + 2.51 / (l * l));
}
inline double pi_lower(double x) {
    if (x < 355991.0) return 0;
    const double l = log(x);
    return x / l * (1 + 1 / l + 2 / (l * l));
}

// Entries for the primes of (lo, hi]: the smaller of pi(hi) - pi(lo) and the
// bound 2y / log y of any interval of length y (Montgomery and Vaughan, "The
// large sieve", Mathematika 20, 1973), plus slack.  The first is within a few
// percent of the count near the origin, where a chunk of 2^27 numbers holds half
// of what the second allows (7.6e6 primes from 65,536 on against 1.43e7), and
// still the smaller one at 1e11 (8.6e6).
inline uint64_t primes_between_bound(uint64_t lo, uint64_t hi) {
    const double c = pi_upper((double)hi) - pi_lower((double)lo);
    const double mv = hi - lo >= 64 ? 2.0 * (double)(hi - lo) / log((double)(hi - lo)) : 64.0;
    return (uint64_t)(std::min(c, mv) * 1.01) + 4096;
}

}  // namespace cs
