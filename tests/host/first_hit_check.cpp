// Host build of the walk's first hit next to its start (near_first_hit in
// cs_basis.cuh) on steps from the general Euclid run, which also gives it windows
// below those of near_steps: reads "p r w v0" lines, prints "ok a b hit t y" three
// times over, the reciprocal of p exact and off by a relative -2^-24 and +2^-24
// ("hit" 0 where the routine refuses its operands).
#include <cstdint>
#include <cstdio>
#include <initializer_list>

#include "../../paper_2012_03771_gb300/csrc/cs_basis.cuh"

int main() {
    unsigned long long p, r, w, v0;
    while (scanf("%llu %llu %llu %llu", &p, &r, &w, &v0) == 4) {
        uint64_t a = 0, da = 0, b = 0, ub = 0;
        uint32_t it = 0;
        const bool ok = cs::tg_steps<uint64_t>(p, r, w, a, da, b, ub, it, 400);
        for (float e : {0.0f, -5.9604645e-08f, 5.9604645e-08f}) {
            uint32_t t = 0, y = 0;
            const bool hit = ok && ((a | b) >> 31) == 0 &&
                             cs::near_first_hit(cs::rcp_rn(cs::u64_to_f(p)) * (1.0f + e), (uint32_t)w, (uint32_t)a, (uint32_t)da,
                                                (uint32_t)b, (uint32_t)ub, v0, t, y);
            printf("%d %llu %llu %d %u %u%c", ok, (unsigned long long)a, (unsigned long long)b, hit, t, y, e > 0 ? '\n' : ' ');
        }
    }
    return 0;
}
