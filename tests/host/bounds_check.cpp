// Host build of the prime-count bounds that size device buffers
// (cs_prime_bounds.h): reads "lo hi" lines, prints the entries for (lo, hi].
#include <cstdio>
#include "../../paper_2012_03771_gb300/csrc/cs_prime_bounds.h"

int main() {
    unsigned long long lo, hi;
    while (scanf("%llu %llu", &lo, &hi) == 2) printf("%llu\n", (unsigned long long)cs::primes_between_bound(lo, hi));
    return 0;
}
