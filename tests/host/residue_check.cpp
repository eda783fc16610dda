// Host build of the 64-bit primes' residues (cs_residue.cuh) and K's limbs
// (cs_words.h): reads "p M s n q_1 .. q_n" lines (K = product of the q), prints
// "r v chain v' f": r = K mod p, v = (r M + s) mod p, 1 when the chain of whole-sum
// products took p (else the stepwise one), v by near_affine, and r 2^32 / p by
// near_frac32.
#include <cstdint>
#include <cstdio>
#include <vector>
#include "../../paper_2012_03771_gb300/csrc/cs_residue.cuh"
#include "../../paper_2012_03771_gb300/csrc/cs_words.h"

template <bool P32>
static void one(uint64_t p, uint64_t M, uint32_t s, const std::vector<uint32_t> &k) {
    const cs::ResMod q = cs::res_mod<P32>(p);
    const uint32_t n = (uint32_t)k.size();
    const bool chain = q.p0 <= cs::RES_P0_MAX;
    uint64_t t = chain ? k[0] : 0;
    for (uint32_t i = 0; i < n; i++)
        t = chain ? cs::res_limb<P32>(t, i + 1 < n ? k[i + 1] : 0, q) : cs::res_step<P32>(t + k[i], q);
    const uint64_t r = cs::res_finish<P32>(t, n, q);
    printf("%llu %llu %d %llu %u\n", (unsigned long long)r, (unsigned long long)cs::res_affine<P32>(r, M, s, q), chain,
           (unsigned long long)cs::near_affine(r, M, s, p), cs::near_frac32(r, p, cs::rcp_rn(cs::u64_to_f(p))));
}

int main() {
    unsigned long long p, M;
    unsigned s, n;
    while (scanf("%llu %llu %u %u", &p, &M, &s, &n) == 4) {
        std::vector<uint32_t> qK(n), w32;
        for (auto &q : qK)
            if (scanf("%u", &q) != 1) return 1;
        std::vector<uint64_t> w64;
        cs::pack_k_words(qK, w32, w64);
        const std::vector<uint32_t> k = cs::k_limbs(w64);
        if (p >> 32) one<false>(p, M, s, k);
        else one<true>(p, M, s, k);
    }
    return 0;
}
