// The m-classes the three-gap walk takes per large-prime chunk (host code).
//
// Rows are the m coprime to d, so a walk can skip every m that shares a factor
// with a divisor Q of d.  Tiers, from the chunks whose primes have the most hits
// per prime to those with the fewest:
//   class items mod 210 (or 30): every class of m mod Q coprime to Q is a work
//     item of its own, 8/35 (4/15) of the hits, when a class still has at least
//     class_item_hits expected hits per prime;
//   m = 1, 5 (mod 6) as two walkers of one item (6 | d), a third of the hits,
//     from class_min_hits expected hits per prime;
//   the odd m (2 | d), one walker, half of the hits;
//   every m (odd d).
// Class residues are offsets of m - M_start mod Q.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <initializer_list>
#include <numeric>
#include <vector>

#include "cs_internal.h"

namespace cs {

// Class items mod Q: one class per residue c of m mod Q with gcd(c, Q) = 1.
inline MClasses class_items(uint32_t Q, uint64_t M_start) {
    MClasses mc = EVERY_M;
    mc.Q = Q;
    mc.n = 0;
    const uint32_t ms = (uint32_t)(M_start % Q);
    for (uint32_t c = 1; c < Q; c++)
        if (std::gcd(c, Q) == 1) mc.item_off[mc.n++] = (uint8_t)((c + Q - ms) % Q);
    mc.items = mc.n;
    mc.off[0] = mc.item_off[0];
    return mc;
}

struct ClassTiers {
    MClasses mcls = EVERY_M;         // classes of the chunks with many hits (mod 6, else mod 2)
    MClasses mcls_light = EVERY_M;   // classes of the other chunks (the odd m when 2 | d)
    std::vector<MClasses> fine;      // class-item candidates, finest first
    uint32_t m_classes = 0;          // cs_tuning.m_classes
    double hits_scale = 0;           // M_inc * S: expected hits of a prime p are hits_scale / p
    double split_min_hits = 48.0;
    double class_item_hits = 64.0;

    // chunks whose low end is lo walk the two classes mod 6 (or the one mod 2)
    bool split(uint64_t lo) const {
        if (mcls.Q == 1) return false;
        if (m_classes == 2) return true;
        return hits_scale / (double)std::max<uint64_t>(lo, 1) >= split_min_hits;
    }
    // the classes a chunk whose primes start above lo walks
    MClasses for_chunk(uint64_t lo) const {
        if (m_classes == 3) return fine.empty() ? EVERY_M : fine[0];
        if (m_classes == 0)
            for (const MClasses &mc : fine)
                if (hits_scale / ((double)std::max<uint64_t>(lo, 1) * mc.Q) >= class_item_hits) return mc;
        return split(lo) ? mcls : mcls_light;
    }
};

// Tiers for a plan: three_gap = the three-gap walk is used and SL > 0 (the
// one-solve-per-hit walk and SL = 0 take every m); t.m_classes <= 3.
inline ClassTiers class_tiers(bool three_gap, uint64_t d, uint64_t M_start, uint64_t M_inc, uint64_t S,
                              const cs_tuning &t) {
    ClassTiers ct;
    ct.m_classes = t.m_classes;
    ct.hits_scale = (double)M_inc * (double)S;
    if (t.class_min_hits) ct.split_min_hits = (double)t.class_min_hits;
    if (t.class_item_hits) ct.class_item_hits = (double)t.class_item_hits;
    if (three_gap && t.m_classes != 1) {
        const uint32_t m6 = (uint32_t)(M_start % 6), m2 = (uint32_t)(M_start % 2);
        if (d % 2 == 0) ct.mcls_light = ct.mcls = MClasses{2, 1, {(1 + 2 - m2) % 2, 0}, 0, {}};
        if (d % 6 == 0) ct.mcls = MClasses{6, 2, {(1 + 6 - m6) % 6, (5 + 6 - m6) % 6}, 0, {}};
        // class items mod 210 and 30 by default; mod 6 and 2 too when forced everywhere
        for (uint32_t Q : {210u, 30u, 6u, 2u})
            if (d % Q == 0 && (Q > 6 || t.m_classes == 3)) ct.fine.push_back(class_items(Q, M_start));
    }
    return ct;
}

// Where a chunk (lo, hi] of large primes ends: below 2^30 or 2^32 when it would cross
// it, so that all its primes take one form (32-bit fields below 2^30; of the 64-bit
// ones, residues with one word per prime below 2^32 and two above, whose float
// quotients are derived for those ranges).
inline uint64_t chunk_end(uint64_t lo, uint64_t hi) {
    for (uint64_t limit : {1ull << 30, 1ull << 32})
        if (lo < limit - 1 && hi >= limit) return limit - 1;
    return hi;
}

// The light chunks' form for few m: from which prime on trying every m of the class
// (k_few_m) costs less than a prepared walker (22 to 27 ps a prime for preparation and
// walk, hardly depending on p).  With n m tried, k_few_m takes 6 + 0.085 n ps and 250 ps
// for every expected hit, n S / p of them (one GB300, n 1 to 256, S 601 to 50,001, p
// 2^17 to 2^31: 128 m of S = 50,001 52 ps at p = 2^25, 25 at 2^27, 20 at 2^29; 44 m of
// 16,001 17, 11 and 10; 256 m of 4001 38, 29 and 27).  That is below 22 ps from p = 25000
// n S / (1600 - 9 n) on.  Where that prime is below 2^24, the primes under it are too few
// to be worth a chunk and its three launches, and every prime with at most one
// expected hit tries every m (22 m of 40,001 to 1e7: 157 us a sieve either way; 128 of
// 601 124 against 123).
inline uint64_t few_from(uint64_t M_inc, uint64_t S, const MClasses &mc) {
    const uint64_t n = (M_inc + mc.Q - 1) / mc.Q;
    if (9 * n >= 1600) return ~0ull;
    const uint64_t from = 25000 * n * S / (1600 - 9 * n);
    return from < (1u << 24) ? n * S : from;
}

}  // namespace cs
