// Host build of the sieve's cost estimate (csrc/cs_cost.h): reads "M_c M_inc S P T
// L limbs chunks cached" lines, prints picoseconds.
#include <cstdio>

#include "../../paper_2012_03771_gb300/csrc/cs_cost.h"

int main() {
    unsigned long long M_c, M_inc, S, P, T, L, limbs, chunks, cached;
    while (scanf("%llu %llu %llu %llu %llu %llu %llu %llu %llu", &M_c, &M_inc, &S, &P, &T, &L, &limbs, &chunks, &cached) == 9)
        printf("%.0f\n", cs::sieve_cost_ps(M_c, M_inc, S, P, T, L, limbs, chunks, cached != 0));
    return 0;
}
