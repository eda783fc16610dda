// Host build of the rule for the light chunks' form (csrc/cs_classes.h): reads
// "M_inc S Q" lines, prints the prime from which every m is tried.
#include <cstdio>

#include "../../paper_2012_03771_gb300/csrc/cs_classes.h"

int main() {
    unsigned long long M_inc, S;
    unsigned Q;
    while (scanf("%llu %llu %u", &M_inc, &S, &Q) == 3) {
        cs::MClasses mc = cs::EVERY_M;
        mc.Q = Q;
        printf("%llu\n", (unsigned long long)cs::few_from(M_inc, S, mc));
    }
    return 0;
}
