// Host build of the large-prime chunks' ends (csrc/cs_classes.h): reads "lo hi"
// lines, prints where the chunk ends.
#include <cstdio>

#include "../../paper_2012_03771_gb300/csrc/cs_classes.h"

int main() {
    unsigned long long lo, hi;
    while (scanf("%llu %llu", &lo, &hi) == 2) printf("%llu\n", (unsigned long long)cs::chunk_end(lo, hi));
    return 0;
}
