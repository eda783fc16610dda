// Host build of the walk's short-chain step and first-hit routines
// (cs_basis.cuh): reads "p r w v0" lines, prints "ok a da b ub ok t y", the first
// four from near_steps (32-bit below 2^30, else 64-bit), the last two from
// near_first_hit on those steps ("0 ..." where a routine refuses its operands).
#include <cstdint>
#include <cstdio>
#include "../../paper_2012_03771_gb300/csrc/cs_basis.cuh"

int main() {
    unsigned long long p, r, v0;
    unsigned w;
    while (scanf("%llu %llu %u %llu", &p, &r, &w, &v0) == 4) {
        uint32_t a = 0, da = 0, b = 0, ub = 0, t = 0, y = 0, it = 0;
        const bool ok = p < (1u << 30) ? cs::near_steps<uint32_t>((uint32_t)p, (uint32_t)r, w, a, da, b, ub, it)
                                       : cs::near_steps<uint64_t>(p, r, w, a, da, b, ub, it);
        const bool hit = ok && cs::near_first_hit(cs::rcp_rn(cs::u64_to_f(p)), w, a, da, b, ub, v0, t, y);
        printf("%d %u %u %u %u %d %u %u\n", ok, a, da, b, ub, hit, t, y);
    }
    return 0;
}
