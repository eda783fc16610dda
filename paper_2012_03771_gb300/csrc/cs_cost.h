// Estimated device time of one sieve (host code), for ordering the instances of a
// batch and for the priority level of a server's request.
#pragma once
#include <math.h>
#include <stdint.h>

#include <algorithm>

namespace cs {

// Picoseconds on one GB300: 6 for a (row, small prime) pair of the tile sieve; 1.25
// for each of a prime's hits over all m (the walk visits the classes of m that can
// be rows and stores a third of its visits); per large prime 40 for generation,
// preparation and walk and 0.4 for every limb of K, or 28 for the walk from a residue
// cache; 15 us of launches per chunk and 80 us for the rest.  Within a quarter of
// the measured time above half a millisecond (0.56 ms to 0.89 s, with and without
// caches), within 40% below.
inline double sieve_cost_ps(uint64_t M_c, uint64_t M_inc, uint64_t S, uint64_t P, uint64_t T, uint64_t L, uint64_t n_limb,
                            uint64_t n_chunks, bool cached) {
    auto pi = [](double x) {
        const double l = log(x);
        return x < 3 ? 0.0 : x / l * (1 + 1 / l + 2 / (l * l));
    };
    const double Ld = (double)std::max<uint64_t>(L, 2), Td = (double)T;
    const double small = (double)M_c * std::max(0.0, pi(std::min(Td, Ld)) - pi((double)P));
    double hits = 0, large = 0;
    if (L > T && T > 2) {
        hits = (double)M_inc * (double)S * log(log(Ld) / log(Td));
        large = pi(Ld) - pi(Td);
    }
    const double per_prime = cached ? 28.0 : 40.0 + 0.4 * (double)n_limb;
    return small * 6.0 + hits * 1.25 + large * per_prime + 15e6 * (double)n_chunks + 80e6;
}

}  // namespace cs
