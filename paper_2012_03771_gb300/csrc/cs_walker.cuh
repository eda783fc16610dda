// The walker of one prime for the three-gap walk's one-walker chunks (odd m,
// or every m for odd d; one segment per prime), computed ahead of the walk by
// the preparation kernel k_tg_prep.  (Computed inside the 64-bit residue
// kernel right after K mod p instead, it made that kernel 80 registers wide and
// the two together 22% slower than apart.)
//
// With r' = Q r mod p, the two steps of the walk come from one run of Euclid's
// algorithm on (p, r') (walker_steps), and the class's first hit from the step
// basis in O(1) (walker_first_hit): the same work, in the same order and
// arithmetic, as the walk kernel does for an item it prepares itself, so the
// results and the solver statistics are identical.  The descriptor: d0 = {first
// m - M_start (NO_WALKER when no hit falls in the range), v at that m, d_a, u_b},
// d1 = {steps of m a Q, b Q, clamped to M_inc}.
#pragma once
#include <stdint.h>

#include "cs_arith.cuh"
#include "cs_basis.cuh"
#include "cs_errors.h"

namespace cs {

constexpr uint32_t NO_WALKER = 0xffffffffu;

// v + k r mod p for a small k (v, r < p, 2p fits in UT)
template <class UT>
__device__ __forceinline__ UT add_times(UT v, UT r, uint32_t k, UT p) {
    for (; k; k--) {
        v += r;
        if (v >= p) v -= p;
    }
    return v;
}

// The two steps and the first hit by the general routines of cs_arith.cuh, for
// the operands that the near_* routines refuse (about one prime in a thousand).
// The preparation kernel calls them (CALL), which keeps its registers and code
// small; the walk kernels have them inline, as a call there would move the
// walkers' state out of registers.
struct GeneralSteps {
    uint64_t a, da, b, ub;
    uint32_t it;
    bool ok;
};
template <class UT>
__device__ __forceinline__ GeneralSteps walker_steps_general(UT pp, UT rq, UT w, uint32_t max_iter) {
    GeneralSteps g{0, 0, 0, 0, 0, false};
    if (sizeof(UT) == 8 && w >= 1024) {
        uint32_t da32, ub32;
        g.ok = tg_steps_w(pp, rq, (uint32_t)w, g.a, da32, g.b, ub32, g.it, max_iter);
        g.da = da32;
        g.ub = ub32;
    } else {
        UT a, da, b, ub;
        g.ok = tg_steps<UT>(pp, rq, w, a, da, b, ub, g.it, max_iter);
        if (g.ok) {
            g.a = a; g.da = da; g.b = b; g.ub = ub;
        }
    }
    return g;
}
struct GeneralHit {
    uint64_t t, y;
};
template <class UT>
__device__ __noinline__ GeneralSteps walker_steps_call(UT pp, UT rq, UT w, uint32_t max_iter) {
    return walker_steps_general<UT>(pp, rq, w, max_iter);
}
template <class UT>
__device__ __forceinline__ GeneralHit walker_hit_general(UT pp, UT w, UT a, UT da, UT b, UT ub, UT v0) {
    GeneralHit h;
    if constexpr (sizeof(UT) == 4) {
        uint32_t y;
        h.t = first_hit32(pp, rcp_rn((float)pp), w, a, da, b, ub, v0, y);
        h.y = y;
    } else if (w >= 1024 && ((a | b) >> 31) == 0) {
        uint32_t y;
        h.t = first_hit_w(pp, rcp_rn(u64_to_f(pp)), (uint32_t)w, (uint32_t)a, (uint32_t)da, (uint32_t)b,
                          (uint32_t)ub, v0, y);
        h.y = y;
    } else {
        uint64_t y;
        h.t = first_hit64(pp, w, a, da, b, ub, v0, y);
        h.y = y;
    }
    return h;
}
template <class UT>
__device__ __noinline__ GeneralHit walker_hit_call(UT pp, UT w, UT a, UT da, UT b, UT ub, UT v0) {
    return walker_hit_general<UT>(pp, w, a, da, b, ub, v0);
}

// The two steps of (p, r'): false after max_iter Euclid steps.
template <class UT, bool CALL = false>
__device__ __forceinline__ bool walker_steps(UT pp, UT rq, UT w, UT &a, UT &da, UT &b, UT &ub, uint32_t &it,
                                             uint32_t max_iter) {
    uint32_t a32, da32, b32, ub32;
    if (w >= (sizeof(UT) == 8 ? 1024u : 512u) && near_steps<UT>(pp, rq, (uint32_t)w, a32, da32, b32, ub32, it)) {
        a = a32; da = da32; b = b32; ub = ub32;
        return true;
    }
    const GeneralSteps g = CALL ? walker_steps_call<UT>(pp, rq, w, max_iter)
                                : walker_steps_general<UT>(pp, rq, w, max_iter);
    a = (UT)g.a; da = (UT)g.da; b = (UT)g.b; ub = (UT)g.ub;
    it += g.it;
    return g.ok;
}
// The smallest t >= 0 with (v + r' t) mod p <= w from the two steps, for v > w;
// v becomes that residue.  fp = 1 / p.
template <class UT, bool CALL = false>
__device__ __forceinline__ uint64_t walker_first_hit(UT pp, float fp, UT w, UT a, UT da, UT b, UT ub, UT &v) {
    uint32_t t, y;
    if (((a | b) >> 31) == 0 &&
        near_first_hit(fp, (uint32_t)w, (uint32_t)a, (uint32_t)da, (uint32_t)b, (uint32_t)ub, (uint64_t)v, t, y)) {
        v = (UT)y;
        return t;
    }
    const GeneralHit h = CALL ? walker_hit_call<UT>(pp, w, a, da, b, ub, v)
                              : walker_hit_general<UT>(pp, w, a, da, b, ub, v);
    v = (UT)h.y;
    return h.t;
}
__device__ __forceinline__ float walker_rcp(uint32_t pp) { return rcp_rn((float)pp); }
__device__ __forceinline__ float walker_rcp(uint64_t pp) { return rcp_rn(u64_to_f(pp)); }

// pp: the prime; r = K mod p; vv = (r M_start + SL) mod p; w = 2 SL > 0; M =
// M_inc; Q <= 2 and off0 < Q: the class of m walked.  Adds the solver's work to
// solves / levels and ERR_SOLVER_LIMIT to err when a run exceeds max_iter.
template <class UT>
__device__ __forceinline__ void prep_walker(UT pp, UT r, UT vv, UT w, uint64_t M, uint32_t Q, uint32_t off0,
                                            uint32_t max_iter, unsigned long long &solves,
                                            unsigned long long &levels, unsigned long long &err, uint4 &d0,
                                            uint2 &d1) {
    uint32_t it = 0;
    UT ma_ = 0, da_ = 0, mb_ = 0, ub_ = 0;
    uint64_t first = 0;
    // the class's first m is m = off0 (mod Q): v advances by r per m
    const uint32_t dd = off0;
    UT vk = dd ? add_times(vv, r, 1, pp) : vv;
    const UT rq = Q > 1 ? add_times(r, r, 1, pp) : r;
    const bool ok = walker_steps<UT, true>(pp, rq, w, ma_, da_, mb_, ub_, it, max_iter);
    if (!ok) err |= ERR_SOLVER_LIMIT;
    solves += 2 + (vk > w);
    if (ok && vk > w) first = walker_first_hit<UT, true>(pp, walker_rcp(pp), w, ma_, da_, mb_, ub_, vk) * Q;
    levels += it;
    const uint64_t mf = dd + first;
    const uint64_t sa = (uint64_t)ma_ * Q, sb = (uint64_t)mb_ * Q;
    d0 = make_uint4(ok && mf < M ? (uint32_t)mf : NO_WALKER, (uint32_t)vk, (uint32_t)da_, (uint32_t)ub_);
    d1 = make_uint2((uint32_t)(sa < M ? sa : M), (uint32_t)(sb < M ? sb : M));
}

}  // namespace cs
