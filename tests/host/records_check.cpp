// Host build of the apply groups as the plan asks for them (csrc/cs_buckets.h):
// reads "M_c wpr W l2 walk_ctas n_wheel q_1 .. q_k n lo_1 hi_1 .. lo_n hi_n" lines,
// prints the columns that become records, the number of groups, and 1 when the
// last chunk ends one.
#include <cstdint>
#include <cstdio>
#include <utility>
#include <vector>

#include "../../paper_2012_03771_gb300/csrc/cs_buckets.h"

int main() {
    unsigned long long M_c, wpr, W, l2, ctas, k, n;
    while (scanf("%llu %llu %llu %llu %llu %llu", &M_c, &wpr, &W, &l2, &ctas, &k) == 6) {
        std::vector<uint32_t> wheel(k);
        for (auto &q : wheel)
            if (scanf("%u", &q) != 1) return 1;
        if (scanf("%llu", &n) != 1) return 1;
        std::vector<std::pair<uint64_t, uint64_t>> chunks(n);
        for (auto &c : chunks) {
            unsigned long long lo, hi;
            if (scanf("%llu %llu", &lo, &hi) != 2) return 1;
            c = {lo, hi};
        }
        const cs::BucketLayout b = cs::bucket_layout(2, 0, 0, true, !chunks.empty(), M_c, wpr, l2, ctas);
        const uint64_t cols = cs::record_columns(W, wheel);
        const std::vector<uint8_t> after = cs::apply_groups(chunks, M_c, cols, b);
        unsigned groups = 0;
        for (uint8_t f : after) groups += f;
        printf("%llu %u %d\n", (unsigned long long)cols, groups, !after.empty() && after.back() == 1);
    }
    return 0;
}
